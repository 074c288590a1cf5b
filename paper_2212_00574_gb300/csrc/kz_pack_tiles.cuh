// kz_pack_tiles.cuh -- the tile form of the dense packer: a caller's 0/1 bit
// matrix (caller vertex ids, strict upper triangle read) into symmetric
// block-plane rows, 32 caller rows at a time, shared by the dense loader and
// the allocation-free entry point.
//
// The relabelling moves columns, so a CTA takes 32 caller rows i0 .. i0 + 31
// (i0 a multiple of 32) and turns the bit permutation into a word gather.
// (1) Column words: word j holds column j over the 32 rows, kept in shared
// memory.  Columns right of the rows come from the rows themselves (lane r
// reads 32 bytes of row i0 + r, a warp transpose per 32 columns); columns
// left of them are read off the rows above, whose 32-bit word i0 / 32 is the
// column word already; the 32 columns on the diagonal take both halves.  So
// the rows come out symmetric in one pass, and rows above suffice: a loader
// can pack each chunk of rows as it arrives.  (2) Output: for word w = r k +
// c of the relabelled rows, lane b fetches the column word of caller column
// perm[y], y = coff[c] + 32 r + b, and a transpose gives lane r word w of row
// inv[i0 + r]; a lane collects kTileWords words before its 32-byte stores.
//
// What bounds it: the two transposes (10 shuffles a word) and scattered
// 32-byte sectors, not the bytes.  One pass instead of an upper-triangle pass
// and a symmetrizing pass over the whole matrix saves the latter (118 us for
// n = 32768, 7.4 us for n = 4096).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kz_rules.cuh"

namespace kz {

constexpr int kTileThreads = 512;
constexpr int kTileWords = 8;

// (1): column words of the rows i0 .. i0 + rows - 1 (whole block).
__device__ __forceinline__ void tile_columns(uint32_t *colw, const uint64_t *__restrict__ bits, int64_t row_words,
                                             int32_t n, int64_t i0, int rows) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int nq = (n + 31) >> 5, qi = (int)(i0 >> 5);
  const uint32_t *bits32 = reinterpret_cast<const uint32_t *>(bits);  // a 64-bit word's low half first
  const uint32_t in_rows = rows < 32 ? (1u << rows) - 1u : 0xffffffffu;
  const uint64_t *row = bits + (i0 + lane) * row_words;
  for (int q0 = warp * kTileWords; q0 < nq; q0 += nwarps * kTileWords) {
    uint32_t v[kTileWords];
#pragma unroll
    for (int u = 0; u < kTileWords; u += 2) {
      const int q = q0 + u;
      v[u] = v[u + 1] = 0u;
      if (q >= qi) {
        const uint64_t x = (lane < rows && (q >> 1) < row_words) ? row[q >> 1] : 0ull;
        v[u] = (uint32_t)x;
        v[u + 1] = (uint32_t)(x >> 32);
      } else {
        v[u] = bits32[(int64_t)(32 * q + lane) * 2 * row_words + qi] & in_rows;
        if (q + 1 < qi) v[u + 1] = bits32[(int64_t)(32 * q + 32 + lane) * 2 * row_words + qi] & in_rows;
        else if (lane < rows) v[u + 1] = (uint32_t)(row[q >> 1] >> 32);
      }
    }
#pragma unroll
    for (int u = 0; u < kTileWords; u++) {
      const int q = q0 + u;  // uniform in the warp
      if (q >= nq) break;
      if (q > qi) {
        v[u] = transpose32(v[u]);
      } else if (q == qi) {
        v[u] &= ~((2u << lane) - 1u);
        v[u] = (v[u] | transpose32(v[u])) & in_rows;
      }
      colw[32 * q + lane] = v[u];
    }
  }
}

// (2): the relabelled rows, written to A and to the copies B and C unless
// null (whole block; colw complete).  Returns the thread's set bits; *bad is
// set when an edge lies inside one class.
__device__ __forceinline__ unsigned long long tile_rows(const uint32_t *colw, uint32_t *__restrict__ A,
                                                        uint32_t *__restrict__ B, uint32_t *__restrict__ C,
                                                        int32_t ldw, int32_t k, int32_t R, const int32_t *scoff,
                                                        const int32_t *__restrict__ perm, int32_t x, int32_t own,
                                                        bool valid, bool *bad) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, rk = R * k;
  unsigned long long mine = 0;
  for (int w0 = warp * kTileWords; w0 < ldw; w0 += nwarps * kTileWords) {
    uint32_t out[kTileWords];
    int c = w0 % k, r = w0 / k;  // class and round of word w0 + u
#pragma unroll
    for (int u = 0; u < kTileWords; u++) {
      uint32_t col = 0u;
      if (w0 + u < rk) {
        const int32_t y = scoff[c] + 32 * r + lane;
        if (y < scoff[c + 1]) col = colw[perm[y]];
      }
      out[u] = transpose32(col);
      if (out[u] && c == own && w0 + u < rk) {
        *bad = true;
        out[u] = 0u;
      }
      if (++c == k) {
        c = 0;
        ++r;
      }
    }
    if (valid) {
      const uint4 lo = make_uint4(out[0], out[1], out[2], out[3]), hi = make_uint4(out[4], out[5], out[6], out[7]);
      const int64_t at = (int64_t)x * ldw + w0;
      const bool both = w0 + kTileWords <= ldw;
      *reinterpret_cast<uint4 *>(A + at) = lo;
      if (both) *reinterpret_cast<uint4 *>(A + at + 4) = hi;
      if (B) {
        *reinterpret_cast<uint4 *>(B + at) = lo;
        if (both) *reinterpret_cast<uint4 *>(B + at + 4) = hi;
      }
      if (C) {
        *reinterpret_cast<uint4 *>(C + at) = lo;
        if (both) *reinterpret_cast<uint4 *>(C + at + 4) = hi;
      }
      mine += __popc(lo.x) + __popc(lo.y) + __popc(lo.z) + __popc(lo.w);
      if (both) mine += __popc(hi.x) + __popc(hi.y) + __popc(hi.z) + __popc(hi.w);
    }
  }
  return mine;
}

}  // namespace kz
