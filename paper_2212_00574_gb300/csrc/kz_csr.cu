// kz_csr.cu -- the CSR of an edge-list graph, built on the device.
//
// The sparse path (kz_sparse.cu) needs, for the caller's edges:
//   * the canonical edge list (u < v) sorted by (u, v), duplicates merged or
//     rejected; an edge's id is its index in that order (eu, ev);
//   * the CSR: row u holds u's lower neighbours in ascending order, then its
//     higher ones in ascending order, each with its edge id (row0, adj0, eid0);
//   * the orientation rank: vertices ordered by degree, ties by id.
// Two stable LSD radix sorts do the work: the keys (u, v) on all their bits,
// which gives the edge order and the upper halves of the rows, and then the
// edge ids, in that order, by v alone: equal v's keep ascending u's, which
// gives the lower halves.  A third, of the vertices in id order by degree,
// gives the rank.  Where a vertex begins in either order is found by bisection
// (up_off, low_off), and every position in the rows follows from the two:
// row0 = up_off + low_off, edge e is entry e + low_off[u + 1] of row u, and the
// j-th edge by v is entry j + up_off[v] of row v.
//
// Measured on a Chung-Lu graph of 200,000 vertices and 5.9 million edges:
// device work of the build 1.72 ms before (atomic per-vertex counts, five
// scans, the second sort on (v, u) with values), 0.9 ms now; the load 3.95 to
// 3.15 ms, once the caller's list is checked by several threads.  The floor is the sorts' traffic, 8 passes of 24 bytes a key: 0.17 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "kz_internal.cuh"

namespace kz {

namespace {

constexpr int kRadixThreads = 256;  // one bin per thread
constexpr int kRadixItems = 16;     // keys per thread per tile
constexpr int kRadixTile = kRadixThreads * kRadixItems;
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kWarpKeys = kRadixTile / kRadixWarps;  // a warp's consecutive keys

int sms_csr() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return std::max(sms, 1);
}

int bits_for(uint64_t x) {  // bits needed to hold every value up to x
  int b = 1;
  while (b < 63 && (x >> b) != 0) b++;
  return b;
}

// ---------------------------------------------------------------------------
// stable LSD radix sort of 64-bit keys, 8 bits a pass.  A tile is kRadixTile
// consecutive keys; a warp ranks its kWarpKeys of them, 32 at a time in order,
// with counts of its own (no block barrier in between), so each pass is stable.
// The tile is then brought into digit order in shared memory and leaves it in
// runs of one digit, 128 bytes on average.  Bound by memory: 16 bytes a key and
// pass in the scatter, 8 in the histogram.  Over 5.9 million keys a pass
// of the scatter takes 37 us; with tiles of 2048 keys, ranked with four block
// barriers per 256 and written key by key, it took 65.
// ---------------------------------------------------------------------------

__global__ void radix_hist_kernel(const uint64_t *__restrict__ keys, int64_t m, int shift,
                                  int32_t *__restrict__ hist, int64_t tiles) {
  __shared__ int32_t h[256];
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = t * kRadixTile;
#pragma unroll
    for (int r = 0; r < kRadixItems; r++) {
      const int64_t i = base + (int64_t)r * kRadixThreads + threadIdx.x;
      if (i < m) atomicAdd(&h[(keys[i] >> shift) & 255u], 1);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * tiles + t] = h[threadIdx.x];  // bin-major
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kRadixThreads) radix_scatter_kernel(const uint64_t *__restrict__ keys, int64_t m,
                                                                      int shift, const int64_t *__restrict__ off,
                                                                      int64_t tiles, uint64_t *__restrict__ okeys) {
  __shared__ uint64_t sorted[kRadixTile];
  __shared__ int32_t wcnt[kRadixWarps][256];  // per-warp counts, then positions in the tile
  __shared__ int64_t place[256];              // a digit's keys go to place + position in the tile
  __shared__ int32_t wsum[kRadixWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int64_t base = t * kRadixTile;
    const int64_t mine = base + warp * kWarpKeys + lane;
    uint64_t key[kRadixItems];
    int32_t rank[kRadixItems];
#pragma unroll
    for (int r = 0; r < kRadixItems; r++) key[r] = mine + 32 * r < m ? keys[mine + 32 * r] : 0ull;
    for (int b = lane; b < 256; b += 32) wcnt[warp][b] = 0;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < kRadixItems; r++) {
      const bool valid = mine + 32 * r < m;
      const unsigned d = (unsigned)(key[r] >> shift) & 255u;
      // lanes with this digit, a ballot a bit (a match instruction takes a
      // turn for every digit present: 50 us a pass)
      unsigned same = __ballot_sync(0xffffffffu, valid);
#pragma unroll
      for (int b = 0; b < 8; b++) {
        const unsigned ones = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        same &= (d >> b) & 1u ? ones : ~ones;
      }
      const int before = valid ? wcnt[warp][d] : 0;
      rank[r] = before + __popc(same & lt);
      __syncwarp();
      if (valid && (same & lt) == 0u) wcnt[warp][d] = before + __popc(same);
      __syncwarp();
    }
    __syncthreads();
    // thread b: the tile's keys of digit b, and where they begin in its order
    int total = 0;
#pragma unroll
    for (int w = 0; w < kRadixWarps; w++) total += wcnt[w][threadIdx.x];
    int upto = total;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, upto, d);
      if (lane >= d) upto += y;
    }
    if (lane == 31) wsum[warp] = upto;
    __syncthreads();
    int begin = upto - total;
    for (int w = 0; w < warp; w++) begin += wsum[w];
    place[threadIdx.x] = off[(int64_t)threadIdx.x * tiles + t] - begin;
#pragma unroll
    for (int w = 0; w < kRadixWarps; w++) {
      const int c = wcnt[w][threadIdx.x];
      wcnt[w][threadIdx.x] = begin;
      begin += c;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRadixItems; r++)
      if (mine + 32 * r < m) sorted[wcnt[warp][(key[r] >> shift) & 255u] + rank[r]] = key[r];
    __syncthreads();
    const int count = (int)(m - base < kRadixTile ? m - base : kRadixTile);
    for (int j = threadIdx.x; j < count; j += kRadixThreads) {
      const uint64_t x = sorted[j];
      okeys[place[(x >> shift) & 255u] + j] = x;
    }
    __syncthreads();  // the next tile reuses the shared arrays
  }
}

// Sorts keys[0..m) on their bits [lo, hi); the result is where `keys` points
// afterwards (the two buffers change places with every pass).
kz_status radix_sort(uint64_t *&keys, uint64_t *&tmp, int64_t m, int lo, int hi, int32_t *hist, int64_t *off,
                     int64_t *sums, int64_t *total, cudaStream_t s) {
  if (m <= 1) return KZ_OK;
  const int64_t tiles = (m + kRadixTile - 1) / kRadixTile;
  const int grid = (int)std::min<int64_t>(tiles, 8 * sms_csr());
  for (int shift = lo; shift < hi; shift += 8) {
    radix_hist_kernel<<<grid, kRadixThreads, 0, s>>>(keys, m, shift, hist, tiles);
    KZ_TRY(scan_counts(hist, 256 * tiles, off, sums, total, s));
    radix_scatter_kernel<<<grid, kRadixThreads, 0, s>>>(keys, m, shift, off, tiles, tmp);
    KZ_CUDA_TRY(cudaGetLastError());
    std::swap(keys, tmp);
  }
  return KZ_OK;
}

// ---------------------------------------------------------------------------
// the CSR steps
// ---------------------------------------------------------------------------

__global__ void canon_kernel(const int32_t *__restrict__ edges, int64_t m, int B, uint64_t *__restrict__ keys) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    uint32_t u = (uint32_t)edges[2 * e], v = (uint32_t)edges[2 * e + 1];
    if (u > v) {
      const uint32_t t = u;
      u = v;
      v = t;
    }
    keys[e] = ((uint64_t)u << B) | v;
  }
}

// *dup = 1 when a sorted key repeats
__global__ void repeats_kernel(const uint64_t *__restrict__ keys, int64_t m, int32_t *dup) {
  bool any = false;
  for (int64_t i = 1 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
    any |= keys[i] == keys[i - 1];
  if (any) *dup = 1;
}

// keep[i] = 1 for the first of equal sorted keys
__global__ void first_of_kernel(const uint64_t *__restrict__ keys, int64_t m, int32_t *__restrict__ keep) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
    keep[i] = i == 0 || keys[i] != keys[i - 1] ? 1 : 0;
}

__global__ void compact_kernel(const uint64_t *__restrict__ keys, const int32_t *__restrict__ keep,
                               const int64_t *__restrict__ pos, int64_t m, uint64_t *__restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
    if (keep[i]) out[pos[i]] = keys[i];
}

// endpoints, and the keys (v, edge id) of the second order
__global__ void split_kernel(const uint64_t *__restrict__ keys, int64_t m, int B, int32_t *__restrict__ eu,
                             int32_t *__restrict__ ev, uint64_t *__restrict__ keys2) {
  const uint64_t mask = (1ull << B) - 1ull;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t key = keys[e];
    eu[e] = (int32_t)(key >> B);
    ev[e] = (int32_t)(key & mask);
    keys2[e] = ((key & mask) << 32) | (uint64_t)e;
  }
}

// off[x] = keys before vertex x's, x = 0..n, in keys sorted by (key >> shift)
__device__ __forceinline__ int64_t keys_before(const uint64_t *__restrict__ keys, int64_t m, int shift, uint64_t x) {
  int64_t lo = 0, hi = m;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((keys[mid] >> shift) < x) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

__global__ void offsets_kernel(const uint64_t *__restrict__ by_u, int shift_u, const uint64_t *__restrict__ by_v,
                               int64_t m, int32_t n, int64_t *__restrict__ up_off, int64_t *__restrict__ low_off,
                               int64_t *__restrict__ row) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x <= n; x += (int64_t)gridDim.x * blockDim.x) {
    const int64_t up = keys_before(by_u, m, shift_u, (uint64_t)x), low = keys_before(by_v, m, 32, (uint64_t)x);
    up_off[x] = up;
    low_off[x] = low;
    row[x] = up + low;
  }
}

// both entries of every edge
__global__ void fill_kernel(const int32_t *__restrict__ eu, const int32_t *__restrict__ ev,
                            const uint64_t *__restrict__ by_v, int64_t m, const int64_t *__restrict__ up_off,
                            const int64_t *__restrict__ low_off, int32_t *__restrict__ adj,
                            int32_t *__restrict__ eid) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = i + low_off[eu[i] + 1];
    adj[p] = ev[i];
    eid[p] = (int32_t)i;
    const uint64_t key = by_v[i];
    const int32_t e = (int32_t)(key & 0xffffffffu);
    const int64_t q = i + up_off[key >> 32];
    adj[q] = eu[e];
    eid[q] = e;
  }
}

__global__ void degree_keys_kernel(const int64_t *__restrict__ row, int32_t n, uint64_t *__restrict__ keys) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x)
    keys[x] = ((uint64_t)(row[x + 1] - row[x]) << 32) | (uint64_t)x;
}

__global__ void rank_kernel(const uint64_t *__restrict__ keys, int32_t n, int32_t *__restrict__ rank) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    rank[keys[i] & 0xffffffffu] = (int32_t)i;
}

// Device scratch of one build, released when it goes out of scope.
struct Scratch {
  cudaStream_t s;
  std::vector<std::pair<void *, size_t>> held;
  bool refused = false;
  explicit Scratch(cudaStream_t st) : s(st) {}
  ~Scratch() {
    for (auto &h : held) dev_free(h.first, h.second, s);
  }
  template <class T>
  T *get(size_t count) {
    const size_t bytes = std::max<size_t>(count, 1) * sizeof(T);
    void *p = refused ? nullptr : dev_alloc(bytes, s);
    if (p) held.emplace_back(p, bytes);
    refused = !p;  // nothing more is asked for then
    return static_cast<T *>(p);
  }
};

}  // namespace

kz_status sparse_build_csr(kz_graph g, const int32_t *d_edges, int64_t m_in, bool dedup, cudaStream_t s) {
  const int32_t n = g->n;
  const int B = bits_for((uint64_t)std::max(n - 1, 1));
  const int grid = 8 * sms_csr(), threads = 256;
  const int64_t mm_in = std::max<int64_t>(m_in, 1);
  const int64_t keys_len = std::max<int64_t>(mm_in, n);  // the edge keys, then the vertex keys
  const int64_t tiles = (keys_len + kRadixTile - 1) / kRadixTile;
  Scratch sc(s);
  uint64_t *k0 = sc.get<uint64_t>(keys_len), *k1 = sc.get<uint64_t>(keys_len), *k2 = sc.get<uint64_t>(keys_len);
  int32_t *hist = sc.get<int32_t>(256 * tiles);
  int64_t *off = sc.get<int64_t>(256 * tiles + 1);
  int64_t *sums = sc.get<int64_t>(std::max(256 * tiles, mm_in) / 1024 + 2), *total = sc.get<int64_t>(2);
  int32_t *dup = sc.get<int32_t>(1);
  if (!k0 || !k1 || !k2 || !hist || !off || !sums || !total || !dup) return KZ_ERR_OOM;

  // (u, v) keys, sorted; duplicates merged or rejected
  int64_t m = m_in;
  if (m_in > 0) {
    canon_kernel<<<grid, threads, 0, s>>>(d_edges, m_in, B, k0);
    KZ_TRY(radix_sort(k0, k1, m_in, 0, 2 * B, hist, off, sums, total, s));
    KZ_CUDA_TRY(cudaMemsetAsync(dup, 0, sizeof(int32_t), s));
    repeats_kernel<<<grid, threads, 0, s>>>(k0, m_in, dup);
    KZ_CUDA_TRY(cudaGetLastError());
    int32_t h_dup = 0;
    KZ_CUDA_TRY(cudaMemcpyAsync(&h_dup, dup, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    KZ_CUDA_TRY(cudaStreamSynchronize(s));
    if (h_dup && !dedup) return KZ_ERR_DUPLICATE_EDGE;
    if (h_dup) {
      int32_t *first = sc.get<int32_t>(m_in);
      int64_t *pos = sc.get<int64_t>(m_in + 1);
      if (!first || !pos) return KZ_ERR_OOM;
      first_of_kernel<<<grid, threads, 0, s>>>(k0, m_in, first);
      KZ_TRY(scan_counts(first, m_in, pos, sums, total, s));
      compact_kernel<<<grid, threads, 0, s>>>(k0, first, pos, m_in, k1);
      KZ_CUDA_TRY(cudaGetLastError());
      KZ_CUDA_TRY(cudaMemcpyAsync(&m, total, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
      KZ_CUDA_TRY(cudaStreamSynchronize(s));
      std::swap(k0, k1);
    }
  }
  g->m = m;
  const size_t nn = (size_t)std::max(n, 1), mm = (size_t)std::max<int64_t>(m, 1);
  KZ_TRY(graph_alloc(g, &g->sp_row0, nn + 1, s));
  KZ_TRY(graph_alloc(g, &g->sp_adj0, 2 * mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_eid0, 2 * mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_eu, mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_ev, mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_rank, nn, s));
  int64_t *up_off = sc.get<int64_t>(nn + 1), *low_off = sc.get<int64_t>(nn + 1);
  if (!up_off || !low_off) return KZ_ERR_OOM;
  // the edge ids by v; k0 keeps the (u, v) keys
  if (m > 0) {
    split_kernel<<<grid, threads, 0, s>>>(k0, m, B, g->sp_eu, g->sp_ev, k2);
    KZ_TRY(radix_sort(k2, k1, m, 32, 32 + B, hist, off, sums, total, s));
  }
  offsets_kernel<<<grid, threads, 0, s>>>(k0, B, k2, m, n, up_off, low_off, g->sp_row0);
  if (m > 0)
    fill_kernel<<<grid, threads, 0, s>>>(g->sp_eu, g->sp_ev, k2, m, up_off, low_off, g->sp_adj0, g->sp_eid0);
  KZ_CUDA_TRY(cudaGetLastError());
  // orientation rank: degree order, ties by id (degrees are below n)
  if (n > 0) {
    degree_keys_kernel<<<grid, threads, 0, s>>>(g->sp_row0, n, k0);
    KZ_TRY(radix_sort(k0, k1, n, 32, 32 + B, hist, off, sums, total, s));
    rank_kernel<<<grid, threads, 0, s>>>(k0, n, g->sp_rank);
    KZ_CUDA_TRY(cudaGetLastError());
  }
  // the scratch is released on the stream after this work
  return KZ_OK;
}

}  // namespace kz
