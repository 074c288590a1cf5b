// kz_pairs.cu -- pair form of a Jacobi pass on the bitset rows, for graphs
// whose live edges are a small share of the vertex pairs (thesis Section 4.2
// rules; the sweep kernels of kz_bitset.cu test 32 x 32 blocks of pairs, live
// or not, and the tensor form counts every pair of the graph in every class).
//
// Every live edge {u, v} and every class c it needs is one test: do the
// class-c words of rows u and v share a bit?  A few words settle most tests,
// so a test looks at the first W words of the class in shared memory and the
// rare miss searches the rest in global memory.
//
// Work split.  The vertices' blocks are cut into tiles of kTileBlocks blocks.
// lists_kernel writes, for every tile and block of v's of higher classes, each
// v's neighbours in the tile.  A job of pair_kernel is one tile of u's, one
// group of G classes and a range of v blocks: the CTA stages the group's
// first words of the tile's rows (32 words a row: G classes x W words), and
// its warps take the v blocks one at a time, one v per lane: the lane walks
// its v's list with the v's own 32 words in registers, and eight 16-byte
// shared loads and 32 logic operations settle the G tests of an edge.
//
// What bounds it: shared-memory bandwidth.  The lanes read different rows, so
// their reads would collide; instead lane l reads a row's eight 16-byte
// chunks in the order q ^ (l & 7) and holds its own words in the same order,
// so the eight lanes of a 128-byte wavefront always hit different banks, for
// any rows: a test costs W / 32 wavefronts, divided by how full the lanes are
// (a block's longest list against the mean, about 0.8).  Two CTAs of eight
// warps an SM, so that one stages while the other tests, and two edges a step
// for sixteen loads in flight.
//
// A test that misses in the staged words joins a small per-lane queue; when a
// lane's queue fills, and at the end of a list, the warp searches the queued
// tests' later words in global memory (two 16-byte loads a row and step).
//
// Measured, one pass on GB300, against the tensor form and the bitset sweep:
//   n = 32768, k = 24, p = 0.07 (36M edges)   4.7 ms   14.3 ms    100 ms
//   n = 32768, k = 24, p = 0.12 (62M edges)   3.3 ms   14.3 ms     44 ms
//   n = 16384, k = 24, p = 0.1                0.95 ms   2.2 ms   14.6 ms
//   n =  9001, k = 17, p = 0.112              0.30 ms   0.50 ms   2.5 ms
//   n =  4500, k = 12, p = 0.12               0.13 ms   0.16 ms   0.30 ms
// (ncu, n = 16384, p = 0.1: logic pipe 57% busy, issue slots 46%).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <new>
#include <vector>

#include "kz_internal.cuh"
#include "kz_rules.cuh"
#include "kz_sweep.cuh"

namespace kz {
namespace pairs {

constexpr int kTileBlocks = 24;              // blocks of u's per tile
constexpr int kTileRows = 32 * kTileBlocks;  // 768
constexpr int kRowWords = 32;                // staged words of a row
constexpr int kWarps = 8;                    // two CTAs an SM
constexpr int kThreads = 32 * kWarps;
constexpr int kQueue = 12;                 // queued misses per lane
// the rows of a tile and one row of ones, which pads the lists
constexpr size_t kRowBytes = (size_t)(kTileRows + 1) * kRowWords * 4;
constexpr size_t kSmemBytes = kRowBytes + (size_t)kQueue * kThreads * 4;
constexpr uint32_t kPad = kTileRows;

// The list of one block of v's in one tile: `rows` rows of 32 pairs of
// entries (one pair a lane) from row `first` on.
struct ListRef {
  uint32_t first, rows;
};

struct PairArgs {
  const uint32_t *cm;       // current rows by class: class c of row x at (c n + x) Rp
  uint32_t *Edel;           // deletion bitmap, rows x ldw (zeroed)
  const BlockDesc *blocks;
  const ListRef *refs;      // tile-major: refs[tile * nb + block]
  const uint32_t *lists;
  const int2 *jobs;         // (tile, first block of v's)
  int32_t n_jobs, n_groups, span;  // a job covers `span` blocks of v's; it runs once per class group
  int32_t nb, k, ldw, Rp;
  int64_t cls;              // words of a class, n Rp
  unsigned long long *counts;  // [0] failing edges [1] live edges tested [2] failing vertices
  unsigned int *queue;         // next job
};

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}

__device__ __forceinline__ uint32_t mad(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

__device__ __forceinline__ uint32_t and_any(const uint4 &a, const uint4 &b) {
  return ((a.x & b.x) | (a.y & b.y)) | ((a.z & b.z) | (a.w & b.w));
}

// The queued misses of the warp's lanes, searched in the words from W on.  A
// class without a common neighbour anywhere marks the edge.
template <int W>
__device__ __noinline__ void search_tail(const PairArgs &p, const uint32_t *queue, int cnt, const BlockDesc *tile,
                                         int c0, int v, const BlockDesc Y, unsigned int &fails) {
  const int most = __reduce_max_sync(0xffffffffu, cnt);
  const int quads = p.Rp >> 2;
  for (int i = 0; i < most; i++) {
    if (i >= cnt) continue;
    const uint32_t w = queue[i * kThreads + threadIdx.x];
    const int idx = w & 0xffffu;
    if (idx >= kTileRows) continue;  // padding
    const BlockDesc B = tile[idx >> 5];
    const int u = B.base + (idx & 31);
    bool fail = false;
    for (uint32_t mask = w >> 16; mask && !fail; mask &= mask - 1) {
      const int c = c0 + __ffs(mask) - 1;
      if (c >= p.k || c == Y.c || c == B.c) continue;
      const uint4 *pu = reinterpret_cast<const uint4 *>(p.cm + c * p.cls + (int64_t)u * p.Rp);
      const uint4 *pv = reinterpret_cast<const uint4 *>(p.cm + c * p.cls + (int64_t)v * p.Rp);
      uint32_t any = 0;
      for (int q = W / 4; q < quads && !any; q += 2) {
        const uint4 a0 = pu[q], b0 = pv[q];
        any = and_any(a0, b0);
        if (q + 1 < quads) {
          const uint4 a1 = pu[q + 1], b1 = pv[q + 1];
          any |= and_any(a1, b1);
        }
      }
      fail = !any;
    }
    if (fail) {
      const uint32_t bu = 1u << (idx & 31);
      const uint32_t old = atomicOr(&p.Edel[(int64_t)v * p.ldw + B.r * p.k + B.c], bu);
      atomicOr(&p.Edel[(int64_t)u * p.ldw + Y.r * p.k + Y.c], 1u << (threadIdx.x & 31));
      fails += (old & bu) ? 0u : 1u;
    }
  }
}

// W: words of a class staged per row (4, 8, 16 or 32); G = 32 / W classes.
template <int W>
__global__ void __launch_bounds__(kThreads, 2) pair_kernel(const __grid_constant__ PairArgs p) {
  constexpr int G = kRowWords / W;  // classes of a group
  constexpr int Q = W / 4;          // 16-byte chunks of a class
  extern __shared__ __align__(128) unsigned char smem[];
  uint32_t *rows = reinterpret_cast<uint32_t *>(smem);
  uint32_t *queue = reinterpret_cast<uint32_t *>(smem + kRowBytes);
  __shared__ BlockDesc s_tile[kTileBlocks];
  __shared__ unsigned int s_job, s_next;
  const int t = threadIdx.x, lane = t & 31;
  const int rot = lane & 7;
  const int k = p.k, Rp = p.Rp;
  uint32_t off[8];  // address of chunk q ^ rot in the first row
#pragma unroll
  for (int q = 0; q < 8; q++) off[q] = smem_addr(rows) + ((uint32_t)(q ^ rot) << 4);
  unsigned int fails = 0;
  if (t < kRowWords) rows[kTileRows * kRowWords + t] = ~0u;
  for (;;) {
    __syncthreads();  // the previous job's rows are no longer read
    if (t == 0) {
      s_job = atomicAdd(p.queue, 1u);
      s_next = 0;
    }
    __syncthreads();
    const unsigned int j = s_job;
    if (j >= (unsigned int)p.n_jobs * (unsigned int)p.n_groups) break;
    const int2 job = p.jobs[j % (unsigned int)p.n_jobs];
    const int c0 = (int)(j / (unsigned int)p.n_jobs) * G;
    const int b0 = job.x * kTileBlocks;
    if (t < kTileBlocks) {
      BlockDesc b = {0, 0, 0, 0};
      if (b0 + t < p.nb) b = p.blocks[b0 + t];
      s_tile[t] = b;
    }
    __syncthreads();
    for (int i = t; i < kTileRows * 8; i += kThreads) {
      const int row = i >> 3, q = i & 7;
      const BlockDesc B = s_tile[row >> 5];
      const int c = c0 + q / Q, w = 4 * (q % Q);
      if ((row & 31) < B.size) {
        uint32_t *dst = rows + i * 4;
        if (c >= k || c == B.c)  // not a class the pair needs
          *reinterpret_cast<uint4 *>(dst) = make_uint4(~0u, ~0u, ~0u, ~0u);
        else if (w < Rp)
          cp_async16(dst, p.cm + c * p.cls + (int64_t)(B.base + (row & 31)) * Rp + w);
        else
          *reinterpret_cast<uint4 *>(dst) = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    // the warps take the job's blocks of v's one at a time
    const int y_end = min(job.y + p.span, p.nb);
    for (;;) {
      const int yb = job.y + (int)__shfl_sync(0xffffffffu, lane == 0 ? atomicAdd(&s_next, 1u) : 0u, 0);
      if (yb >= y_end) break;
      const ListRef ref = p.refs[(int64_t)job.x * p.nb + yb];
      if (ref.rows == 0) continue;
      const uint32_t *lp = p.lists + (int64_t)ref.first * 32 + lane;
      const int n2 = (int)ref.rows;
      constexpr uint32_t kPads = kPad | kPad << 16;
      uint32_t next0 = lp[0], next1 = n2 > 1 ? lp[32] : kPads;
      const BlockDesc Y = p.blocks[yb];
      const int v = Y.base + min(lane, Y.size - 1);
      const uint32_t *cmv = p.cm + (int64_t)v * Rp;
      uint4 x[8];  // this lane's words, chunk q ^ rot in slot q
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int pos = q ^ rot;
        const int c = c0 + pos / Q, w = 4 * (pos % Q);
        x[q] = make_uint4(0u, 0u, 0u, 0u);
        if (c >= k || c == Y.c) x[q] = make_uint4(~0u, ~0u, ~0u, ~0u);
        else if (w < Rp) x[q] = *reinterpret_cast<const uint4 *>(cmv + c * p.cls + w);
      }
      int cnt = 0;
      for (int i = 0; i < n2; i++) {
        const uint32_t two = next0;
        next0 = next1;
        next1 = i + 2 < n2 ? lp[(i + 2) * 32] : kPads;
        const uint32_t i0 = two & 0xffffu, i1 = two >> 16;
        uint32_t h0[G], h1[G];
#pragma unroll
        for (int q = 0; q < 8; q++) {
          const uint32_t a0 = and_any(lds128(mad(i0, kRowWords * 4, off[q])), x[q]);
          const uint32_t a1 = and_any(lds128(mad(i1, kRowWords * 4, off[q])), x[q]);
          h0[q / Q] = q % Q == 0 ? a0 : h0[q / Q] | a0;
          h1[q / Q] = q % Q == 0 ? a1 : h1[q / Q] | a1;
        }
        uint32_t least0 = h0[0], least1 = h1[0];
#pragma unroll
        for (int j2 = 1; j2 < G; j2++) {
          least0 = min(least0, h0[j2]);
          least1 = min(least1, h1[j2]);
        }
        if (__any_sync(0xffffffffu, min(least0, least1) == 0u)) {
          uint32_t m0 = 0, m1 = 0;
#pragma unroll
          for (int j2 = 0; j2 < G; j2++) {
            if (h0[j2] == 0u) m0 |= 1u << (j2 ^ (rot / Q));
            if (h1[j2] == 0u) m1 |= 1u << (j2 ^ (rot / Q));
          }
          if (m0) queue[cnt++ * kThreads + t] = (two & 0xffffu) | m0 << 16;
          if (m1) queue[cnt++ * kThreads + t] = (two >> 16) | m1 << 16;
          if (__any_sync(0xffffffffu, cnt >= kQueue - 1)) {
            search_tail<W>(p, queue, cnt, s_tile, c0, v, Y, fails);
            cnt = 0;
          }
        }
      }
      if (__any_sync(0xffffffffu, cnt > 0)) search_tail<W>(p, queue, cnt, s_tile, c0, v, Y, fails);
    }
  }
  fails = __reduce_add_sync(0xffffffffu, fails);
  if (lane == 0 && fails) atomicAdd(&p.counts[0], (unsigned long long)fails);
}

// The lists: one warp per block of v's walks the tiles of lower classes; a
// lane's entries are its v's neighbours in the tile (vertex i of the tile's
// block b as 32 b + i), two to a word, padded to the longest list of the block
// with the index past the tile's rows.  pos[b] is block b's word in a row (rows of `stride` words).
// FILL = false only adds up the rows the lists take.
template <bool FILL>
__global__ void __launch_bounds__(256) lists_kernel(const uint32_t *__restrict__ rows, int64_t stride,
                                                    const int64_t *__restrict__ pos,
                                                    const BlockDesc *__restrict__ blocks,
                                                    const int32_t *__restrict__ boff, int32_t nb, int32_t n_tiles,
                                                    int32_t tile_blocks, ListRef *__restrict__ refs, uint32_t *__restrict__ lists,
                                                    unsigned long long *cursor, unsigned long long *n_tests) {
  const int lane = threadIdx.x & 31;
  const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t pad = 32u * (uint32_t)tile_blocks;
  unsigned long long tests = 0;
  for (int64_t job = warp0; job < (int64_t)nb * n_tiles; job += warps) {
    const int tile = (int)(job / nb), y = (int)(job - (int64_t)tile * nb);
    const BlockDesc Y = blocks[y];
    const int b0 = tile * tile_blocks, b1 = min(b0 + tile_blocks, boff[Y.c]);
    const uint32_t *row = rows + (int64_t)(Y.base + min(lane, Y.size - 1)) * stride;
    int deg = 0;
    if (lane < Y.size)
      for (int b = b0; b < b1; b++) deg += __popc(row[pos[b]]);
    const uint32_t n2 = (uint32_t)(__reduce_max_sync(0xffffffffu, deg) + 1) / 2;
    unsigned long long first = 0;
    if (lane == 0 && n2) first = atomicAdd(cursor, (unsigned long long)n2);
    if constexpr (FILL) {
      first = __shfl_sync(0xffffffffu, first, 0);
      if (lane == 0) refs[job] = {(uint32_t)first, n2};
      tests += deg;
      uint32_t *out = lists + first * 32 + lane;
      uint32_t held = 0, e = 0;
      if (lane < Y.size)
        for (int b = b0; b < b1; b++)
          for (uint32_t w = row[pos[b]]; w; w &= w - 1) {
            const uint32_t ent = (uint32_t)(32 * (b - b0) + __ffs(w) - 1);
            if (e & 1) out[(e >> 1) * 32] = held | ent << 16;
            else held = ent;
            e++;
          }
      if (e & 1) {
        out[(e >> 1) * 32] = held | pad << 16;
        e++;
      }
      for (uint32_t i = e >> 1; i < n2; i++) out[i * 32] = pad | pad << 16;
    }
  }
  if constexpr (FILL) {
    for (int o = 16; o > 0; o >>= 1) tests += __shfl_down_sync(0xffffffffu, tests, o);
    if (lane == 0 && tests) atomicAdd(n_tests, tests);
  }
}

// ---------------------------------------------------------------------------
// Passes from the third of a run on: every test remembers a witness.
//
// hint[class][list row][lane] names, for both entries, the word of the class
// in which the pair last shared a bit.  A pass looks at that one word of both
// rows and searches the class only when its bits are gone, so a test costs one
// random and one conflict-free 4-byte shared load (about 4.5 wavefronts for 32
// tests) whatever the class length, where pair_kernel reads W words.  Witnesses
// live as long as a run's lists do: a deleted edge's entry becomes padding, and
// once three tenths of the listed edges are gone the lists are built anew, and
// the hints with them.
//
// A job is one class, one tile of u's (all its words of the class staged) and
// a range of v blocks; a warp holds its block's words transposed, [word][lane].
// Bound by latency: of 16 warps an SM 3.4 an issue wait at the staging's barriers
// and 1.9 for lists and hints; issue slots are 40% busy, the rate of shared-memory
// wavefronts 30% (8 per 32 tests, the staging with them; n = 9001, k = 17, p =
// 0.112, the third pass with hints).  The
// first pass with hints, which finds them, takes 0.58 ms there (0.99 when every
// test went to the search), the next 0.19 and the later ones 0.13, where
// pair_kernel takes 0.22; at n = 32768, k = 24, p = 0.07 12.6, 2.9 and 2.1 ms
// against 4.6.  Whole runs, k-partite graphs of four seeds each: n = 32768 23 to
// 31 passes in 73 to 91 ms (on the tensor form 329 ms for 23), n = 9001 12 to 14
// passes in 3.1 to 3.5 ms (7.1 for 14).  Runs of two passes, the common kind, keep
// pair_kernel.  Padding tested as a row of ones instead of masked: 8% slower; list
// rows of four entries: 8%.
// ---------------------------------------------------------------------------

constexpr int kHintQueue = 12;
constexpr int kHintAhead = 4;
constexpr size_t kHintSmem = 225 * 1024;
constexpr double kHintRebuild = 0.7;  // share of the listed edges still alive below which lists are rebuilt

struct HintArgs {
  const uint32_t *cm;
  uint32_t *Edel;
  const BlockDesc *blocks;
  const ListRef *refs;
  uint32_t *lists;
  uint16_t *hints;          // [class][list row][lane], one byte an entry
  int64_t hint_rows;        // list rows of a class
  const int2 *jobs;
  int32_t n_jobs, span, tile_blocks;
  int32_t nb, k, ldw, Rp;
  int64_t cls;
  unsigned long long *counts;
  unsigned int *queue;
};

__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}

// The queued tests of the warp's lanes, searched over the class from its
// 16-byte chunk `from` on: a new hint, or a failing edge.
static __device__ __noinline__ void search_class(const HintArgs &p, const uint32_t *queue, int stride, int cnt,
                                                 const BlockDesc *tile, uint32_t rows_addr, uint32_t vt_addr, int c,
                                                 uint32_t first, int from, int v, const BlockDesc Y,
                                                 unsigned int &fails) {
  const int lane = threadIdx.x & 31;
  const int quads = p.Rp >> 2;
  // every lane walks its own queue, one 16-byte chunk a step, so lanes with
  // short searches move on to their next test
  uint32_t e = 0, row = 0;
  bool next = true;
  for (int i = -1, q = from;;) {
    if (next) {
      if (++i >= cnt) break;
      e = queue[i * stride];
      row = rows_addr + (e & 0xffffu) * (uint32_t)p.Rp * 4u;
      q = from;
      next = false;
    }
    const uint4 a = lds128(row + 16 * q);
    const uint32_t vw = vt_addr + 512 * q;
    const uint32_t m0 = a.x & lds32(vw), m1 = a.y & lds32(vw + 128), m2 = a.z & lds32(vw + 256),
                   m3 = a.w & lds32(vw + 384);
    const bool hit = (m0 | m1 | m2 | m3) != 0u;
    if (!hit && ++q < quads) continue;
    const uint32_t idx = e & 0xffffu, place = e >> 16;
    const int64_t slot = (((int64_t)first + (place >> 1)) * 32 + lane) * 2 + (place & 1);
    if (hit) {
      reinterpret_cast<uint8_t *>(p.hints + c * p.hint_rows * 32)[slot] = (uint8_t)(4 * q + (m0 ? 0 : m1 ? 1 : m2 ? 2 : 3));
    } else {
      // (other classes' CTAs may read the entry meanwhile: the edge fails either way)
      reinterpret_cast<uint16_t *>(p.lists)[slot] = (uint16_t)(32 * p.tile_blocks);
      const BlockDesc B = tile[idx >> 5];
      const int u = B.base + (int)(idx & 31);
      const uint32_t bu = 1u << (idx & 31);
      const uint32_t old = atomicOr(&p.Edel[(int64_t)v * p.ldw + B.r * p.k + B.c], bu);
      atomicOr(&p.Edel[(int64_t)u * p.ldw + Y.r * p.k + Y.c], 1u << lane);
      fails += (old & bu) ? 0u : 1u;
    }
    next = true;
  }
  __syncwarp();
}

// FRESH: the lists are new and have no hints.  A test then looks at the first
// four words (one 16-byte load of u's row, v's words in registers), which find
// most of the witnesses, and the hints are written as the list is walked.
template <int WARPS, bool FRESH>
__global__ void __launch_bounds__(32 * WARPS, 1) hint_kernel(const __grid_constant__ HintArgs p) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ BlockDesc s_tile[kTileBlocks];
  __shared__ unsigned int s_job, s_next;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int Rp = p.Rp, quads = Rp >> 2, tile_rows = 32 * p.tile_blocks;
  uint32_t *rows = reinterpret_cast<uint32_t *>(smem);
  uint32_t *vt = rows + (size_t)tile_rows * Rp + (size_t)warp * Rp * 32 + lane;
  uint32_t *queue = rows + (size_t)tile_rows * Rp + (size_t)WARPS * Rp * 32 + t;
  const uint32_t rows_addr = smem_addr(rows), vt_addr = smem_addr(vt);
  const uint32_t row_bytes = (uint32_t)Rp * 4u, last_row = (uint32_t)tile_rows - 1u;
  unsigned int fails = 0;
  for (;;) {
    __syncthreads();  // the previous job's rows are no longer read
    if (t == 0) {
      s_job = atomicAdd(p.queue, 1u);
      s_next = 0;
    }
    __syncthreads();
    const unsigned int j = s_job;
    if (j >= (unsigned int)p.n_jobs * (unsigned int)p.k) break;
    const int2 job = p.jobs[j % (unsigned int)p.n_jobs];
    const int c = (int)(j / (unsigned int)p.n_jobs);
    if (t < p.tile_blocks) {
      BlockDesc b = {0, 0, 0, 0};
      if (job.x * p.tile_blocks + t < p.nb) b = p.blocks[job.x * p.tile_blocks + t];
      s_tile[t] = b;
    }
    __syncthreads();
    const uint32_t *cmc = p.cm + c * p.cls;
    for (int i = t; i < tile_rows * quads; i += 32 * WARPS) {
      const int row = i / quads, q = i - row * quads;
      const BlockDesc B = s_tile[row >> 5];
      if ((row & 31) >= B.size) continue;
      uint32_t *dst = rows + (size_t)row * Rp + 4 * q;
      if (B.c == c)  // not a class the pair needs: v itself has u in it
        *reinterpret_cast<uint4 *>(dst) = make_uint4(~0u, ~0u, ~0u, ~0u);
      else
        cp_async16(dst, cmc + (int64_t)(B.base + (row & 31)) * Rp + 4 * q);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    const int y_end = min(job.y + p.span, p.nb);
    auto take = [&]() { return job.y + (int)__shfl_sync(0xffffffffu, lane == 0 ? atomicAdd(&s_next, 1u) : 0u, 0); };
    int yb = take();
    ListRef ref = {0, 0};
    BlockDesc Y = {0, 0, 0, 0};
    if (yb < y_end) {
      ref = p.refs[(int64_t)job.x * p.nb + yb];
      Y = p.blocks[yb];
    }
    while (yb < y_end) {
      const uint32_t first = ref.first;
      const int n2 = Y.c == c ? 0 : (int)ref.rows;
      const BlockDesc Yc = Y;
      // the next block's list and place are on their way meanwhile
      yb = take();
      if (yb < y_end) {
        ref = p.refs[(int64_t)job.x * p.nb + yb];
        Y = p.blocks[yb];
      }
      if (n2 == 0) continue;
      const uint32_t *lp = p.lists + (int64_t)first * 32 + lane;
      uint16_t *hp = p.hints + (c * p.hint_rows + (int64_t)first) * 32 + lane;
      const uint32_t pads = (uint32_t)tile_rows * 0x10001u;
      // list rows and hints kHintAhead steps (of two rows) ahead
      uint32_t le[kHintAhead][2], lh[kHintAhead][2];
#pragma unroll
      for (int d = 0; d < kHintAhead; d++)
#pragma unroll
        for (int r = 0; r < 2; r++) {
          const int i = 2 * d + r;
          le[d][r] = i < n2 ? lp[i * 32] : pads;
          if constexpr (!FRESH) lh[d][r] = i < n2 ? hp[i * 32] : 0u;
        }
      const int v = Yc.base + min(lane, Yc.size - 1);
      const uint4 *vrow = reinterpret_cast<const uint4 *>(cmc + (int64_t)v * Rp);
      __syncwarp();  // the previous block's words are no longer read
#pragma unroll 4
      for (int q = 0; q < quads; q++) {
        const uint4 x = vrow[q];
        vt[128 * q] = x.x;
        vt[128 * q + 32] = x.y;
        vt[128 * q + 64] = x.z;
        vt[128 * q + 96] = x.w;
      }
      __syncwarp();
      uint4 v4 = make_uint4(0u, 0u, 0u, 0u);
      if constexpr (FRESH) v4 = make_uint4(vt[0], vt[32], vt[64], vt[96]);
      int cnt = 0;
      for (int i0 = 0; i0 < n2; i0 += 2 * kHintAhead) {
#pragma unroll
        for (int d = 0; d < kHintAhead; d++) {
          const int i = i0 + 2 * d;
          const uint32_t e[4] = {le[d][0] & 0xffffu, le[d][0] >> 16, le[d][1] & 0xffffu, le[d][1] >> 16};
          uint32_t h[4] = {0u, 0u, 0u, 0u};
          if constexpr (!FRESH) {
            h[0] = lh[d][0] & 0xffu;
            h[1] = lh[d][0] >> 8;
            h[2] = lh[d][1] & 0xffu;
            h[3] = lh[d][1] >> 8;
          }
#pragma unroll
          for (int r = 0; r < 2; r++) {
            const int in = i + 2 * kHintAhead + r;
            le[d][r] = in < n2 ? lp[in * 32] : pads;
            if constexpr (!FRESH) lh[d][r] = in < n2 ? hp[in * 32] : 0u;
          }
          bool miss[4];
          bool any = false;
#pragma unroll
          for (int x = 0; x < 4; x++) {
            if constexpr (FRESH) {
              const uint4 a = lds128(mad(min(e[x], last_row), row_bytes, rows_addr));
              const uint32_t m0 = a.x & v4.x, m1 = a.y & v4.y, m2 = a.z & v4.z;
              miss[x] = (m0 | m1 | m2 | (a.w & v4.w)) == 0u && e[x] <= last_row;
              h[x] = m0 ? 0u : m1 ? 1u : m2 ? 2u : 3u;
            } else {
              const uint32_t wu = lds32(rows_addr + mad(min(e[x], last_row), row_bytes, h[x] * 4u));
              const uint32_t wv = lds32(vt_addr + h[x] * 128u);
              miss[x] = (wu & wv) == 0u && e[x] <= last_row;
            }
            any |= miss[x];
          }
          if constexpr (FRESH) {
            // (a queued test's hint is replaced when its search ends)
            if (i < n2) hp[i * 32] = (uint16_t)(h[0] | h[1] << 8);
            if (i + 1 < n2) hp[(i + 1) * 32] = (uint16_t)(h[2] | h[3] << 8);
          }
          if (__any_sync(0xffffffffu, any)) {
#pragma unroll
            for (int x = 0; x < 4; x++)
              if (miss[x]) queue[cnt++ * (32 * WARPS)] = e[x] | (uint32_t)(2 * i + x) << 16;
            if (__any_sync(0xffffffffu, cnt > kHintQueue - 4)) {
              search_class(p, queue, 32 * WARPS, cnt, s_tile, rows_addr, vt_addr, c, first, FRESH ? 1 : 0, v, Yc,
                           fails);
              cnt = 0;
            }
          }
        }
      }
      if (__any_sync(0xffffffffu, cnt > 0))
        search_class(p, queue, 32 * WARPS, cnt, s_tile, rows_addr, vt_addr, c, first, FRESH ? 1 : 0, v, Yc, fails);
    }
  }
  fails = __reduce_add_sync(0xffffffffu, fails);
  if (lane == 0 && fails) atomicAdd(&p.counts[0], (unsigned long long)fails);
}

// Class-major copy of the current rows and the vertex rule, one CTA per row:
// the row passes through shared memory once, and a class is covered when any
// of its words is set.  Vn starts as a copy of V.
constexpr int kRowThreads = 128;
constexpr size_t kRowSmemMax = 200 * 1024;

__global__ void __launch_bounds__(kRowThreads) rows_kernel(const uint32_t *__restrict__ A, uint32_t *__restrict__ cm,
                                                           const uint32_t *__restrict__ V, uint32_t *__restrict__ Vn,
                                                           const BlockDesc *__restrict__ blocks,
                                                           const int32_t *__restrict__ block_of, int32_t n, int32_t k,
                                                           int32_t R, int32_t ldw, int32_t Rp, int32_t q,
                                                           int32_t *__restrict__ v_sweep, const DevState *st,
                                                           unsigned long long *counts, unsigned int *queue,
                                                           unsigned long long *cursor) {
  extern __shared__ uint32_t srow[];  // plane r at r * ks
  const int ks = k | 1;               // an odd stride: a class's words lie in different banks
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *queue = 0;
    *cursor = 0;
  }
  for (int64_t x = blockIdx.x; x < n; x += gridDim.x) {
    const uint32_t *row = A + x * ldw;
    for (int i = threadIdx.x; i < R * k; i += kRowThreads) srow[i / k * ks + i % k] = row[i];
    __syncthreads();
    for (int i = threadIdx.x; i < k * Rp; i += kRowThreads) {
      const int c = i / Rp, r = i - c * Rp;
      cm[((int64_t)c * n + x) * Rp + r] = r < R ? srow[r * ks + c] : 0u;
    }
    if (threadIdx.x < 32) {
      const BlockDesc b = blocks[block_of[x]];
      const int wv = b.r * k + b.c, bit = (int)x - b.base;
      int cover = 0;
      for (int c = threadIdx.x; c < k; c += 32) {
        uint32_t any = 0;
        if (c != b.c)
          for (int r = 0; r < R; r++) any |= srow[r * ks + c];
        cover += any != 0u;
      }
      cover = __reduce_add_sync(0xffffffffu, cover);
      if (threadIdx.x == 0 && ((V[wv] >> bit) & 1u) && cover < q - 1) {
        atomicAnd(&Vn[wv], ~(1u << bit));
        atomicAdd(&counts[2], 1ull);
        if (v_sweep) v_sweep[x] = (int32_t)(st->sweeps + 1);
      }
    }
    __syncthreads();
  }
}

// Next rows = current rows minus the deletion bitmap (which empties).
__global__ void commit_kernel(const uint4 *__restrict__ A, uint4 *__restrict__ An, uint4 *__restrict__ Edel,
                              int64_t quads) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < quads; i += (int64_t)gridDim.x * blockDim.x) {
    uint4 a = A[i];
    const uint4 d = Edel[i];
    if (d.x | d.y | d.z | d.w) {
      a = make_uint4(a.x & ~d.x, a.y & ~d.y, a.z & ~d.z, a.w & ~d.w);
      Edel[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    An[i] = a;
  }
}

// Closes the pass; report[0] = 1 when the run goes on, report[1] = live edges
// left.  known: the live edges, where no list was counted (else negative).
__global__ void finish_kernel(DevState *st, unsigned long long *counts, long long *report, long long known) {
  if (known >= 0) counts[1] = (unsigned long long)known;
  const int cont = finish_pass(st, counts[2], counts[0], counts[1]);
  report[0] = cont;
  report[1] = (long long)(counts[1] - (cont ? counts[0] : 0ull));
  counts[0] = counts[1] = counts[2] = 0;
}

}  // namespace pairs

using namespace pairs;

namespace {

int sms_p() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return std::max(sms, 1);
}

typedef void (*PairFn)(PairArgs);

PairFn pair_fn(int W) {
  return W == 4 ? pair_kernel<4> : W == 8 ? pair_kernel<8> : W == 16 ? pair_kernel<16> : pair_kernel<32>;
}

}  // namespace

// Per-graph buffers of the pair form (allocated on first use).
struct PairBufs {
  uint32_t *cm = nullptr, *Edel = nullptr, *lists = nullptr;
  ListRef *refs = nullptr;
  int2 *jobs = nullptr;
  int32_t n_jobs = 0, span = 0, n_tiles = 0, Rp = 0;
  int32_t *block_of = nullptr;                  // block of a vertex
  int64_t *pos = nullptr;                       // word of a block in cm, then in a row
  unsigned long long *counts = nullptr;         // counts [3], list rows used
  long long *report = nullptr;                  // of the last pass
  unsigned int *queue = nullptr;
  double live = 0;                              // live edges, as far as the host knows
  // passes with hints
  int32_t hint_tile = 0, hint_tiles = 0, hint_warps = 0, hint_span = 0, n_hint_jobs = 0;
  std::vector<int2> hint_jobs_host;
  uint8_t *hint_mem = nullptr;  // of the run in progress; the four below lie in it
  size_t hint_bytes = 0;
  int2 *hint_jobs = nullptr;
  ListRef *hint_refs = nullptr;
  uint32_t *hint_lists = nullptr;
  uint16_t *hints = nullptr;
  int64_t hint_rows = 0;
  bool hint_off = false;   // not for this run
  double hint_listed = 0;  // live edges when the lists in use were built (0: none)
};

// Jobs (tile, first block of v's) of `span` blocks of v's each: a tile's words
// are staged once per job and class group, so long jobs stage less, but there
// should be about `want` jobs times classes, and a block for every warp.
static void plan_jobs(kz_graph g, int tile_blocks, int warps, int want, int32_t *span,
                      std::vector<int2> &jobs) {
  const int nb = (int)g->blocks.size(), tiles = (nb + tile_blocks - 1) / tile_blocks;
  std::vector<int> begin((size_t)tiles, 0);
  int64_t pairs = 0;
  for (int t = 0; t < tiles; t++) {
    int y = 0;
    while (y < nb && g->boff[g->blocks[y].c] <= t * tile_blocks) y++;
    begin[t] = y;
    pairs += nb - y;
  }
  *span = (int)std::max<int64_t>(warps, std::min<int64_t>(8 * warps, pairs * g->k / want));
  jobs.clear();
  for (int t = 0; t < tiles; t++)
    for (int y = begin[t]; y < nb; y += *span) jobs.push_back(make_int2(t, y));
}

static kz_status pairs_prepare(kz_graph g, PairBufs &b, cudaStream_t s) {
  const int nb = (int)g->blocks.size(), sms = sms_p();
  b.Rp = (g->R + 3) / 4 * 4;
  b.n_tiles = (nb + kTileBlocks - 1) / kTileBlocks;
  std::vector<int2> jobs;
  plan_jobs(g, kTileBlocks, kWarps, 32 * sms, &b.span, jobs);  // a class group is four classes or more
  b.n_jobs = (int32_t)jobs.size();
  std::vector<int32_t> block_of((size_t)std::max(g->n, 1));
  std::vector<int64_t> pos((size_t)2 * std::max(nb, 1));
  for (int i = 0; i < nb; i++) {
    for (int j = 0; j < g->blocks[i].size; j++) block_of[(size_t)g->blocks[i].base + j] = i;
    pos[i] = (int64_t)g->blocks[i].c * g->n * b.Rp + g->blocks[i].r;
    pos[(size_t)nb + i] = g->blocks[i].r * g->k + g->blocks[i].c;
  }
  KZ_TRY(graph_alloc(g, &b.cm, (size_t)std::max(g->n, 1) * g->k * b.Rp, s));
  KZ_TRY(graph_alloc(g, &b.Edel, (size_t)std::max(g->n, 1) * g->ldw, s));
  KZ_TRY(graph_alloc(g, &b.jobs, std::max<size_t>(jobs.size(), 1), s));
  KZ_TRY(graph_alloc(g, &b.block_of, block_of.size(), s));
  KZ_TRY(graph_alloc(g, &b.pos, pos.size(), s));
  KZ_TRY(graph_alloc(g, &b.refs, std::max<size_t>((size_t)b.n_tiles * nb, 1), s));
  KZ_TRY(graph_alloc(g, &b.counts, 4, s));
  KZ_TRY(graph_alloc(g, &b.report, 2, s));
  KZ_TRY(graph_alloc(g, &b.queue, 4, s));
  KZ_CUDA_TRY(cudaMemsetAsync(b.Edel, 0, (size_t)std::max(g->n, 1) * g->ldw * 4, s));
  KZ_CUDA_TRY(cudaMemsetAsync(b.counts, 0, 32, s));
  if (!jobs.empty())
    KZ_CUDA_TRY(cudaMemcpyAsync(b.jobs, jobs.data(), sizeof(int2) * jobs.size(), cudaMemcpyHostToDevice, s));
  KZ_CUDA_TRY(cudaMemcpyAsync(b.block_of, block_of.data(), 4 * block_of.size(), cudaMemcpyHostToDevice, s));
  KZ_CUDA_TRY(cudaMemcpyAsync(b.pos, pos.data(), 8 * pos.size(), cudaMemcpyHostToDevice, s));
  for (int W : {4, 8, 16, 32})
    KZ_CUDA_TRY(cudaFuncSetAttribute((const void *)pair_fn(W), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSmemBytes));
  // (a row within the bitset budget takes at most 154 KB: n n k / 32 words
  // of rows fit the budget up to k = 64 at n = 18,900)
  KZ_CUDA_TRY(cudaFuncSetAttribute((const void *)rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kRowSmemMax));
  if ((size_t)g->R * (g->k | 1) * 4 > kRowSmemMax) return KZ_ERR_UNSUPPORTED;
  // the lists of the graph as loaded: every later state's are no longer
  unsigned long long list_rows = 0;
  if (nb > 0) {
    lists_kernel<false><<<16 * sms, 256, 0, s>>>(g->A0, g->ldw, b.pos + nb, g->d_blocks, g->d_boff, nb, b.n_tiles,
                                                 kTileBlocks, nullptr, nullptr, b.counts + 3, nullptr);
    KZ_CUDA_TRY(cudaGetLastError());
  }
  KZ_CUDA_TRY(cudaMemcpyAsync(&list_rows, b.counts + 3, 8, cudaMemcpyDeviceToHost, s));
  KZ_CUDA_TRY(cudaStreamSynchronize(s));  // (the host vectors die here)
  if (list_rows > UINT32_MAX) return KZ_ERR_UNSUPPORTED;
  KZ_TRY(graph_alloc(g, &b.lists, std::max<size_t>((size_t)list_rows * 32, 32), s));
  return KZ_OK;
}

// Words of a class staged per row: the W of least expected cost per test.
// Every test reads W words (1 / 25 wavefront each, the lanes being about 0.8
// full); a miss, of chance exp(-32 W d^2) at edge density d, costs about ten
// wavefronts' worth of time (both fitted to the times above); the staged
// words of a class need not exceed what it has.
static int pick_words(double density, int Rp) {
  int best = 4;
  double cost = 1e300;
  for (int W : {4, 8, 16, 32}) {
    const double c = W / 25.0 + (W >= Rp ? 0.0 : 10.0 * std::exp(-32.0 * W * density * density));
    if (c < cost) {
      cost = c;
      best = W;
    }
  }
  return best;
}

kz_status pairs_buffers(kz_graph g, cudaStream_t s) {
  if (g->pairs_bufs) return KZ_OK;
  PairBufs *b = new (std::nothrow) PairBufs();
  if (!b) return KZ_ERR_OOM;
  const kz_status st = all_or_none(g, s, [&] { return pairs_prepare(g, *b, s); });
  if (st != KZ_OK) {
    delete b;
    return st;
  }
  b->live = (double)g->m;
  g->pairs_bufs = b;
  return KZ_OK;
}

// The hint pass's tile, lists and hints, for the rest of a run: they are given
// back when it ends.  A graph whose classes are too short to gain, too long for
// a byte, or whose hints do not fit stays with pair_kernel (hint_off).
constexpr int kHintMinWords = 12, kHintMaxWords = 255;
constexpr size_t kHintBudgetBytes = size_t(8) << 30;

typedef void (*HintFn)(const HintArgs);
static HintFn hint_fn(int warps, bool fresh) {
  if (warps == 16) return fresh ? hint_kernel<16, true> : hint_kernel<16, false>;
  return fresh ? hint_kernel<8, true> : hint_kernel<8, false>;
}

static kz_status hint_buffers(kz_graph g, PairBufs &b, cudaStream_t s) {
  if (b.hint_mem || b.hint_off) return KZ_OK;
  b.hint_off = true;
  if (g->R < kHintMinWords || b.Rp > kHintMaxWords) return KZ_OK;
  const int nb = (int)g->blocks.size(), sms = sms_p();
  b.hint_warps = b.Rp <= 48 ? 16 : 8;
  const size_t fixed = (size_t)b.hint_warps * (b.Rp * 128 + kHintQueue * 128);
  if (fixed + (size_t)b.Rp * 128 > kHintSmem) return KZ_OK;
  b.hint_tile = (int)std::min<size_t>(kTileBlocks, (kHintSmem - fixed) / ((size_t)b.Rp * 128));
  if (b.hint_tile < 4) return KZ_OK;  // lists of a few entries
  b.hint_tiles = (nb + b.hint_tile - 1) / b.hint_tile;
  if (b.hint_jobs_host.empty()) plan_jobs(g, b.hint_tile, b.hint_warps, 8 * sms, &b.hint_span, b.hint_jobs_host);
  b.n_hint_jobs = (int32_t)b.hint_jobs_host.size();
  if (b.n_hint_jobs == 0) return KZ_OK;
  // the lists of this state: a later one of the run, with fewer edges, takes no
  // more rows
  unsigned long long rows = 0;
  KZ_CUDA_TRY(cudaMemsetAsync(b.counts + 3, 0, 8, s));
  lists_kernel<false><<<16 * sms, 256, 0, s>>>(b.cm, b.Rp, b.pos, g->d_blocks, g->d_boff, nb, b.hint_tiles,
                                               b.hint_tile, nullptr, nullptr, b.counts + 3, nullptr);
  KZ_CUDA_TRY(cudaGetLastError());
  KZ_CUDA_TRY(cudaMemcpyAsync(&rows, b.counts + 3, 8, cudaMemcpyDeviceToHost, s));
  // the cursor goes back to zero: a pass left without hints fills pair_kernel's
  // lists from there, which have no room for as many rows again
  KZ_CUDA_TRY(cudaMemsetAsync(b.counts + 3, 0, 8, s));
  KZ_CUDA_TRY(cudaStreamSynchronize(s));
  const auto part = [](size_t bytes) { return (bytes + 255) & ~(size_t)255; };
  const size_t jobs = part(sizeof(int2) * b.n_hint_jobs), refs = part(sizeof(ListRef) * b.hint_tiles * nb);
  const size_t lists = part((size_t)rows * 128), hints = part((size_t)rows * 64 * g->k);
  if (rows == 0 || rows > UINT32_MAX || lists + hints > kHintBudgetBytes) return KZ_OK;
  b.hint_bytes = jobs + refs + lists + hints;
  b.hint_mem = static_cast<uint8_t *>(dev_alloc(b.hint_bytes, s));
  if (!b.hint_mem) return KZ_OK;  // the passes stay with pair_kernel
  b.hint_jobs = reinterpret_cast<int2 *>(b.hint_mem);
  b.hint_refs = reinterpret_cast<ListRef *>(b.hint_mem + jobs);
  b.hint_lists = reinterpret_cast<uint32_t *>(b.hint_mem + jobs + refs);
  b.hints = reinterpret_cast<uint16_t *>(b.hint_mem + jobs + refs + lists);
  b.hint_rows = (int64_t)rows;
  KZ_CUDA_TRY(cudaMemcpyAsync(b.hint_jobs, b.hint_jobs_host.data(), sizeof(int2) * b.n_hint_jobs,
                              cudaMemcpyHostToDevice, s));
  for (int w : {8, 16})
    for (bool fresh : {false, true})
      KZ_CUDA_TRY(cudaFuncSetAttribute((const void *)hint_fn(w, fresh), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kHintSmem));
  b.hint_off = false;
  return KZ_OK;
}

static void hint_release(PairBufs &b, cudaStream_t s) {
  if (b.hint_mem) dev_free(b.hint_mem, b.hint_bytes, s);
  b.hint_mem = nullptr;
  b.hint_off = false;
  b.hint_listed = 0;
}

// One pass from row buffer `cur` into the other; *cont = 1 when it deleted
// something and the run goes on.  hints: a later pass of a run, whose tests
// keep their witnesses.
static kz_status pairs_pass(kz_graph g, int cur, bool hints, cudaStream_t s, int *cont) {
  PairBufs &b = *static_cast<PairBufs *>(g->pairs_bufs);
  const int sms = sms_p(), nb = (int)g->blocks.size();
  const double density = g->m > 0 ? g->density * b.live / (double)g->m : 0.0;
  const int W = pick_words(density, b.Rp);
  PairArgs a;
  a.cm = b.cm;
  a.Edel = b.Edel;
  a.blocks = g->d_blocks;
  a.refs = b.refs;
  a.lists = b.lists;
  a.jobs = b.jobs;
  a.n_jobs = b.n_jobs;
  a.n_groups = (g->k + kRowWords / W - 1) / (kRowWords / W);
  a.span = b.span;
  a.nb = nb;
  a.k = g->k;
  a.ldw = g->ldw;
  a.Rp = b.Rp;
  a.cls = (int64_t)g->n * b.Rp;
  a.counts = b.counts;
  a.queue = b.queue;
  KZ_CUDA_TRY(cudaMemcpyAsync(g->V[cur ^ 1], g->V[cur], (size_t)g->ldw * 4, cudaMemcpyDeviceToDevice, s));
  const size_t srow = (size_t)g->R * (g->k | 1) * 4;
  rows_kernel<<<std::min(g->n, 16 * sms), kRowThreads, srow, s>>>(
      g->A[cur], b.cm, g->V[cur], g->V[cur ^ 1], g->d_blocks, b.block_of, g->n, g->k, g->R, g->ldw, b.Rp, g->k,
      g->v_sweep, g->st, b.counts, b.queue, b.counts + 3);
  bool hinted = hints && b.n_jobs > 0;
  if (hinted) {
    KZ_TRY(hint_buffers(g, b, s));
    hinted = !b.hint_off;
  }
  long long known = -1;
  bool fresh = false;
  if (hinted) {
    if (b.hint_listed > 0 && b.live >= kHintRebuild * b.hint_listed) {
      known = (long long)b.live;
    } else {
      KZ_CUDA_TRY(cudaMemsetAsync(b.counts + 3, 0, 8, s));
      lists_kernel<true><<<16 * sms, 256, 0, s>>>(b.cm, b.Rp, b.pos, g->d_blocks, g->d_boff, nb, b.hint_tiles,
                                                  b.hint_tile, b.hint_refs, b.hint_lists, b.counts + 3, b.counts + 1);
      fresh = true;
      b.hint_listed = b.live;
    }
    HintArgs h;
    h.cm = b.cm;
    h.Edel = b.Edel;
    h.blocks = g->d_blocks;
    h.refs = b.hint_refs;
    h.lists = b.hint_lists;
    h.hints = b.hints;
    h.hint_rows = b.hint_rows;
    h.jobs = b.hint_jobs;
    h.n_jobs = b.n_hint_jobs;
    h.span = b.hint_span;
    h.tile_blocks = b.hint_tile;
    h.nb = nb;
    h.k = g->k;
    h.ldw = g->ldw;
    h.Rp = b.Rp;
    h.cls = a.cls;
    h.counts = b.counts;
    h.queue = b.queue;
    const size_t smem = (size_t)b.hint_tile * b.Rp * 128 + (size_t)b.hint_warps * (b.Rp * 128 + kHintQueue * 128);
    const int grid = (int)std::min<int64_t>((int64_t)b.n_hint_jobs * g->k, sms);
    hint_fn(b.hint_warps, fresh)<<<grid, 32 * b.hint_warps, smem, s>>>(h);
  } else if (b.n_jobs > 0) {
    lists_kernel<true><<<16 * sms, 256, 0, s>>>(b.cm, b.Rp, b.pos, g->d_blocks, g->d_boff, nb, b.n_tiles,
                                                kTileBlocks, b.refs, b.lists, b.counts + 3, b.counts + 1);
    const int64_t work = (int64_t)a.n_jobs * a.n_groups;
    pair_fn(W)<<<(int)std::min<int64_t>(work, 2 * sms), kThreads, kSmemBytes, s>>>(a);
  }
  const int64_t quads = (int64_t)g->n * g->ldw / 4;
  commit_kernel<<<(int)std::min<int64_t>((quads + 255) / 256, 16 * sms), 256, 0, s>>>(
      reinterpret_cast<const uint4 *>(g->A[cur]), reinterpret_cast<uint4 *>(g->A[cur ^ 1]),
      reinterpret_cast<uint4 *>(b.Edel), quads);
  finish_kernel<<<1, 1, 0, s>>>(g->st, b.counts, b.report, known);
  KZ_CUDA_TRY(cudaGetLastError());
  long long report[2] = {0, 0};
  KZ_CUDA_TRY(cudaMemcpyAsync(report, b.report, sizeof(report), cudaMemcpyDeviceToHost, s));
  KZ_CUDA_TRY(cudaStreamSynchronize(s));
  *cont = (int)report[0];
  b.live = (double)report[1];
  return KZ_OK;
}

static kz_status current_buffer(kz_graph g, cudaStream_t s, int *cur) {
  int32_t c = 0;
  KZ_CUDA_TRY(cudaMemcpyAsync(&c, &g->st->cur, 4, cudaMemcpyDeviceToHost, s));
  KZ_CUDA_TRY(cudaStreamSynchronize(s));
  *cur = c & 1;
  return KZ_OK;
}

kz_status pairs_one_pass(kz_graph g, cudaStream_t s, int *cont) {
  *cont = 0;
  if (g->n == 0) return KZ_OK;
  KZ_TRY(pairs_buffers(g, s));
  int cur = 0;
  KZ_TRY(current_buffer(g, s, &cur));
  return pairs_pass(g, cur, false, s, cont);
}

kz_status pairs_kernelize(kz_graph g, const kz_options &opt, cudaStream_t s) {
  const int64_t max_sweeps = opt.max_sweeps > 0 ? opt.max_sweeps : (int64_t)g->n + g->m + 1;
  KZ_TRY(pairs_buffers(g, s));
  KZ_TRY(bitset_begin_run(g, max_sweeps, s));
  if (g->n == 0) return KZ_OK;
  PairBufs &b = *static_cast<PairBufs *>(g->pairs_bufs);
  b.live = (double)g->m;  // the state may have been reset
  int cur = 0;
  KZ_TRY(current_buffer(g, s, &cur));
  // a run that reaches a third pass is a cascade of many, as a rule
  int pass = 0;
  kz_status rc = KZ_OK;
  for (int cont = 1; cont && rc == KZ_OK; cur ^= 1) rc = pairs_pass(g, cur, pass++ >= 2, s, &cont);
  hint_release(b, s);
  return rc;
}

void pairs_release(kz_graph g) {
  delete static_cast<PairBufs *>(g->pairs_bufs);  // the device buffers are in g->allocs
  g->pairs_bufs = nullptr;
}

}  // namespace kz
