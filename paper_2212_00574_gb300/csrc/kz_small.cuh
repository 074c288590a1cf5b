// kz_small.cuh -- the device-resident state of one graph of at most 4096
// vertices and 32 colours whose layout is found on the device: what the
// allocation-free entry point keeps in its static array, and what the CSR path
// allocates for the remnant of a large graph (kz_sparse.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kz_internal.cuh"

namespace kz {
namespace noalloc {

constexpr int kMaxN = KZ_NOALLOC_MAX_N;          // vertices
constexpr int kMaxWords = KZ_NOALLOC_MAX_WORDS;  // words per adjacency buffer
constexpr int kMaxLdw = 4096;                    // words per row
constexpr int kMaxBlocks = 256;

struct Header {
  CtaGraph desc;
  int32_t status;   // found by the set-up
  int32_t illegal;  // KZ_ERR_ILLEGAL_COLOURING, found by the packer
  int32_t R, pad;
  int64_t cross;            // pairs of vertices in different classes
  unsigned long long bits;  // set bits of the packed rows: twice the edges
  int32_t coff[65];
  int32_t boff[65];
  int32_t rounds[64];
  int32_t pair_off[kMaxBlocks + 1];
  int32_t unit_off[kMaxBlocks + 1];  // prefix of the grid kernel's units: block pairs, one for a block without any
  BlockDesc blocks[kMaxBlocks];
};

struct Scratch {
  alignas(256) Header h;
  alignas(256) DevState st;
  alignas(256) uint32_t A0[kMaxWords];
  alignas(256) uint32_t A1[kMaxWords];
  alignas(256) uint32_t V0[kMaxLdw];
  alignas(256) uint32_t V1[kMaxLdw];
  alignas(256) int32_t perm[kMaxN];
  alignas(256) int32_t inv[kMaxN];
  alignas(256) int32_t pos[kMaxN];  // caller vertex -> (word << 5) | bit of its relabelled vertex inside any row
  alignas(256) int32_t v_sweep[kMaxN];
};

}  // namespace noalloc
}  // namespace kz

namespace kz {

// Set-up (colour classes, blocks, relabelling, live words) of a graph whose n
// colours are in device memory; a layout beyond the scratch leaves a non-zero
// status in h.status and the later kernels idle.
void small_setup(noalloc::Scratch *s, int32_t n, int32_t k, const int32_t *colour, cudaStream_t stream);

}  // namespace kz
