// kz_sparse.cu -- CSR path of the colour-index kernelization, for graphs too
// large or too sparse for bitset rows (thesis Section 4.2 rules).
//
// Vertices keep the caller's ids.  Row u of the live graph starts at the input
// row's place (row0[u]) and holds len[u] entries in ascending order; the rows
// shrink in place, so no pass needs a scan.  Each Jacobi pass:
//   1. vertex_kernel: the vertex rule from the colours of a row's live entries;
//   2. orient_kernel: every live edge of a failing vertex fails the edge rule
//      too (see kz_bitset.cu), whatever its triangles, so it goes at once; the
//      rows keep only edges of two passing vertices for the next pass, and the
//      oriented rows hold every live edge with a passing end once, from its
//      lower to its higher end in degree order;
//   3. triangle_kernel: every live triangle with two passing vertices, found
//      once (u -> v -> w in rank order), ORs the third vertex's colour into the
//      masks of its edges between passing vertices.  A warp holds u's oriented
//      row in a hash table in shared memory and probes it with the oriented
//      rows of u's neighbours v, lanes over the entries;
//   4. verdict_kernel: an edge whose mask has fewer than q-2 bits fails.
// Passes work on the list of vertices still live.  When that list fits (4096
// vertices, 32 colours), the remnant moves to bitset rows and one cooperative
// launch runs it to the fixpoint (kz_small.cuh): its passes need no launches
// and no host.
//
// Measured on n = 200,000, k = 12, 5.9M edges (35 passes, 97% of the edges
// gone after the first): 2.3 ms for the first pass (vertices 0.16, rows 0.33,
// triangles 1.77), 0.45 for the second, 0.65 for the other 33 on bitset rows;
// 3.8, 0.6 and 5.2 ms with a binary search per probe, no vertex filter and
// rows, flags and masks of the whole graph walked every pass.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstddef>
#include <type_traits>
#include <vector>

#include "kz_internal.cuh"
#include "kz_rules.cuh"
#include "kz_small.cuh"

namespace kz {

// ---------------------------------------------------------------------------
// exclusive scan of int32 counts into int64 offsets (3 kernels)
// ---------------------------------------------------------------------------

constexpr int kScanBlock = 1024;

__global__ void scan_block_sums(const int32_t *__restrict__ in, int64_t n, int64_t *__restrict__ sums) {
  __shared__ int64_t s[32];
  const int64_t i = blockIdx.x * (int64_t)kScanBlock + threadIdx.x;
  int64_t v = i < n ? in[i] : 0;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    int64_t w = s[threadIdx.x];
    for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xffffffffu, w, o);
    if (threadIdx.x == 0) sums[blockIdx.x] = w;
  }
}

// Exclusive scan of the block sums in place (one CTA, any count).
__global__ void scan_sums_serial(int64_t *sums, int64_t nblocks, int64_t *total) {
  __shared__ int64_t carry;
  __shared__ int64_t warp_tot[32];
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t base = 0; base < nblocks; base += blockDim.x) {
    const int64_t i = base + threadIdx.x;
    const int64_t v = i < nblocks ? sums[i] : 0;
    // inclusive warp scan
    int64_t x = v;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[w] = x;
    __syncthreads();
    if (w == 0) {
      int64_t t = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0;
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += y;
      }
      warp_tot[lane] = t;  // inclusive over warps
    }
    __syncthreads();
    const int64_t before = carry + (w > 0 ? warp_tot[w - 1] : 0) + x - v;
    if (i < nblocks) sums[i] = before;
    __syncthreads();
    if (threadIdx.x == 0) carry += warp_tot[(blockDim.x >> 5) - 1];
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = carry;
}

__global__ void scan_apply(const int32_t *__restrict__ in, int64_t n, const int64_t *__restrict__ sums,
                           int64_t *__restrict__ out, const int64_t *__restrict__ total) {
  __shared__ int64_t warp_tot[32];
  const int64_t i = blockIdx.x * (int64_t)kScanBlock + threadIdx.x;
  const int64_t v = i < n ? in[i] : 0;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int64_t x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[w] = x;
  __syncthreads();
  if (w == 0) {
    int64_t t = warp_tot[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    warp_tot[lane] = t;
  }
  __syncthreads();
  if (i < n) out[i] = sums[blockIdx.x] + (w > 0 ? warp_tot[w - 1] : 0) + x - v;
  if (i == n - 1) out[n] = *total;
}

// out[0..n] = exclusive prefix of in[0..n-1] (out[n] = total); sums holds
// n / kScanBlock + 1 partial sums.
kz_status scan_counts(const int32_t *in, int64_t n, int64_t *out, int64_t *sums, int64_t *total, cudaStream_t s) {
  if (n <= 0) return cuda_status(cudaMemsetAsync(out, 0, sizeof(int64_t), s));
  const int64_t nb = (n + kScanBlock - 1) / kScanBlock;
  scan_block_sums<<<(unsigned)nb, kScanBlock, 0, s>>>(in, n, sums);
  scan_sums_serial<<<1, kScanBlock, 0, s>>>(sums, nb, total);
  scan_apply<<<(unsigned)nb, kScanBlock, 0, s>>>(in, n, sums, out, total);
  return cuda_status(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// pass kernels
// ---------------------------------------------------------------------------

constexpr int kTableKeys = 256;   // longest oriented row (or run of it) held in a hash table
constexpr int kTableSlots = 512;
constexpr int kItemEdges = 64;    // oriented edges of one u per work item
constexpr int kBloomWords = 256;  // hash bitmap of a table: 8192 bits
constexpr int kTriWarps = 6;

struct SparseArgs {
  int32_t n, k, q;        // q: clique size sought (k for the thesis's rules)
  int32_t from_input;     // the rows are the input's (adj0, eid0), not yet the working ones
  int32_t all_live;       // every edge is live: no flag needs reading
  int32_t apply;          // the pass may be applied (false once the sweep limit is reached)
  const int32_t *col, *rank;
  int2 *vinfo;            // rank, colour and (bit kFailsShift) whether the vertex fails in this pass
  const int64_t *row0;
  const int32_t *adj0, *eid0;
  int32_t *adj, *eid, *len;     // working rows
  int32_t *oadj, *oeid, *olen;  // oriented rows, at the same starts
  uint8_t *elive, *vlive, *vfail;
  const int32_t *list;          // vertices of the pass (null: every one)
  const unsigned int *n_list;
  int32_t *list_out;            // vertices that pass
  unsigned int *n_out;
  unsigned long long *mask;
  int2 *items;                  // (u, run of kItemEdges oriented edges)
  int32_t *big_u, *big_i;       // oriented edges of longer rows, one by one
  unsigned int *n_items, *n_big;
  int32_t *v_sweep;
  DevState *st;
};

constexpr int kFailsShift = 8;

__global__ void vinfo_kernel(const int32_t *__restrict__ rank, const int32_t *__restrict__ col, int32_t n,
                             int2 *__restrict__ vinfo) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    vinfo[v] = make_int2(rank[v], col[v]);
}

__device__ __forceinline__ int64_t list_size(const SparseArgs &a) { return a.list ? (int64_t)*a.n_list : a.n; }

// The kernels over the vertices (1, 2 and 4) give a vertex a warp.  In a pass
// over every vertex of a graph whose mean row has fewer than kShortRow entries
// four vertices share one, eight lanes each, and the warp takes rows of more than
// kLongRow entries afterwards, one after another.  (Later passes are left with
// the core, where four long rows to a warp cost more than short ones gain.)  A
// run on 200,000 vertices, k = 3, mean degree 6: 691 us with a warp each, 559
// so; mean degree 12: 806 and 648; power-law degrees, 300,000, mean 6: 1073 and
// 984; 100,000, mean 20 (a warp each either way): 3330.
constexpr int kShortRow = 16, kLongRow = 64;

// The lanes of a vertex, as one of them sees them: its place among them, the
// first one's lane, and as bits of the warp's lanes all of them and those before
// this one.
template <int LANES>
struct Group {
  static constexpr int kLanes = LANES;
  __device__ __forceinline__ static int lane() { return threadIdx.x & (LANES - 1); }
  __device__ __forceinline__ static int shift() { return LANES == 32 ? 0 : threadIdx.x & 32 - LANES; }
  __device__ __forceinline__ static uint32_t mine() {
    return LANES == 32 ? 0xffffffffu : ((1u << (LANES & 31)) - 1u) << shift();
  }
  __device__ __forceinline__ static uint32_t before() { return mine() & ((1u << (threadIdx.x & 31)) - 1u); }
};

// body(group, vertex, first, end) for the pass's vertices: the bounds that
// row(vertex, first, end) gives.
template <bool SHORT, class Row, class Body>
__device__ __forceinline__ void over_vertices(const SparseArgs &a, Row row, Body body) {
  const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5, total = list_size(a);
  const Group<32> W;
  if constexpr (!SHORT) {
    for (int64_t i = warp0; i < total; i += warps) {
      const int32_t u = a.list ? a.list[i] : (int32_t)i;
      int64_t b, e;
      row(u, b, e);
      body(W, u, b, e);
    }
  } else {
    const Group<8> G;
    for (int64_t i0 = 4 * warp0; i0 < total; i0 += 4 * warps) {
      const int64_t i = i0 + (G.shift() >> 3);
      int32_t u = 0;
      int64_t b = 0, e = 0;
      if (i < total) {
        u = a.list ? a.list[i] : (int32_t)i;
        row(u, b, e);
        if (e - b <= kLongRow) body(G, u, b, e);
      }
      __syncwarp();
      for (uint32_t left = __ballot_sync(0xffffffffu, G.lane() == 0 && e - b > kLongRow); left; left &= left - 1) {
        const int from = __ffs(left) - 1;
        const int32_t v = __shfl_sync(0xffffffffu, u, from);
        body(W, v, __shfl_sync(0xffffffffu, b, from), __shfl_sync(0xffffffffu, e, from));
        __syncwarp();
      }
    }
  }
  __syncwarp();
}

// 1. The vertex rule.
template <bool SHORT>
__global__ void __launch_bounds__(256) vertex_kernel(SparseArgs a) {
  const int64_t sweep_no = a.st->sweeps;
  const int32_t *adj = a.from_input ? a.adj0 : a.adj, *eid = a.from_input ? a.eid0 : a.eid;
  unsigned long long tests = 0, dv = 0;
  const auto row = [&](int32_t u, int64_t &b, int64_t &e) {
    b = a.row0[u];
    e = b + (a.from_input ? a.row0[u + 1] - b : a.len[u]);
  };
  over_vertices<SHORT>(a, row, [&](const auto &G, int32_t u, int64_t b, int64_t e) {
    constexpr int L = std::decay_t<decltype(G)>::kLanes;
    const int32_t ru = a.rank[u];
    unsigned long long cm = 0;
    for (int64_t j = b + G.lane(); j < e; j += L) {
      const int32_t v = adj[j];
      if (a.all_live || a.elive[eid[j]]) {
        const int2 x = a.vinfo[v];  // (another warp may set v's failing bit meanwhile: only rank and colour are read)
        cm |= 1ull << (x.y & 63);
        tests += x.x > ru;
      }
    }
    const uint32_t lo = __reduce_or_sync(G.mine(), (uint32_t)cm), hi = __reduce_or_sync(G.mine(), (uint32_t)(cm >> 32));
    if (G.lane() == 0) {
      cm = ((unsigned long long)hi << 32 | lo) & ~(1ull << a.col[u]);
      const bool fail = a.vlive[u] && __popcll(cm) < a.q - 1;
      a.vfail[u] = fail ? 1 : 0;
      a.vinfo[u].y = a.col[u] | (fail ? 1 << kFailsShift : 0);
      if (fail) {
        dv++;
        if (a.apply) a.vlive[u] = 0;
        a.v_sweep[u] = (int32_t)(sweep_no + 1);  // (a refused sweep's marks lie beyond the count of sweeps)
      }
    }
  });
  for (int o = 16; o > 0; o >>= 1) {
    tests += __shfl_down_sync(0xffffffffu, tests, o);
    dv += __shfl_down_sync(0xffffffffu, dv, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (tests) atomicAdd(&a.st->pass_tests, tests);
    if (dv) atomicAdd(&a.st->pass_dv, dv);
  }
}

// 2. Rows of passing vertices, oriented rows, work items, the next vertex
// list; edges of failing vertices go.  The row shrinks in place behind the
// reads.
template <bool SHORT>
__global__ void __launch_bounds__(256) orient_kernel(SparseArgs a) {
  const int32_t *adj = a.from_input ? a.adj0 : a.adj, *eid = a.from_input ? a.eid0 : a.eid;
  unsigned long long de = 0;
  const auto row = [&](int32_t u, int64_t &b, int64_t &e) {
    b = a.row0[u];
    e = b + (a.from_input ? a.row0[u + 1] - b : a.len[u]);
  };
  over_vertices<SHORT>(a, row, [&](const auto &G, int32_t u, int64_t b, int64_t end) {
    constexpr int L = std::decay_t<decltype(G)>::kLanes;
    const int32_t ru = a.rank[u];
    const bool fu = a.vfail[u] != 0;
    int32_t pl = 0, po = 0;
    for (int64_t base = b; base < end; base += L) {
      const int64_t j = base + G.lane();
      int32_t v = 0, ed = 0;
      bool keep = false, ori = false;
      if (j < end) {
        v = adj[j];
        ed = eid[j];
        if (a.all_live || a.elive[ed]) {
          const int2 x = a.vinfo[v];
          const bool fv = (x.y >> kFailsShift & 1) != 0, up = x.x > ru;
          keep = !fu && !fv;
          ori = up && !(fu && fv);
          if (up && !keep) {
            de++;
            if (a.apply) a.elive[ed] = 0;
          }
          if (up && keep) a.mask[ed] = 0ull;
        }
      }
      __syncwarp(G.mine());  // this step's reads precede its writes, which lie at or before them
      const uint32_t mk = __ballot_sync(G.mine(), keep) & G.mine(), mo = __ballot_sync(G.mine(), ori) & G.mine();
      if (keep && a.apply) {
        a.adj[b + pl + __popc(mk & G.before())] = v;
        a.eid[b + pl + __popc(mk & G.before())] = ed;
      }
      if (ori) {
        a.oadj[b + po + __popc(mo & G.before())] = v;
        a.oeid[b + po + __popc(mo & G.before())] = ed;
      }
      pl += __popc(mk);
      po += __popc(mo);
    }
    const bool live = a.vlive[u] != 0;
    if (G.lane() == 0) {
      a.olen[u] = po;
      if (a.apply) {
        a.len[u] = pl;
        if (live && !fu) a.list_out[atomicAdd(a.n_out, 1u)] = u;
      }
    }
    if (po < 2) return;  // no triangle starts here
    if (po <= kTableKeys) {
      const int parts = (po + kItemEdges - 1) / kItemEdges;
      unsigned int at = 0;
      if (G.lane() == 0) at = atomicAdd(a.n_items, (unsigned int)parts);
      at = __shfl_sync(G.mine(), at, G.shift());
      if (G.lane() < parts) a.items[at + G.lane()] = make_int2(u, G.lane());
    } else {
      unsigned int at = 0;
      if (G.lane() == 0) at = atomicAdd(a.n_big, (unsigned int)po);
      at = __shfl_sync(G.mine(), at, G.shift());
      for (int32_t t = G.lane(); t < po; t += L) {
        a.big_u[at + t] = u;
        a.big_i[at + t] = t;
      }
    }
  });
  for (int o = 16; o > 0; o >>= 1) de += __shfl_down_sync(0xffffffffu, de, o);
  if ((threadIdx.x & 31) == 0 && de) atomicAdd(&a.st->pass_de, de);
}

// OR of bits into a mask; most repeat, so they are looked up first.
__device__ __forceinline__ void or_mask(unsigned long long *mask, int32_t e, unsigned long long bits) {
  if (bits & ~*((volatile unsigned long long *)&mask[e])) atomicOr(&mask[e], bits);
}

// 3. Triangles of the items.  Per warp in shared memory: a bitmap of hashes of
// u's oriented row, its keys in an open-addressed table (at most half full),
// each with its place in the row, its colour and whether it passes, and the
// bits found for the edges (u, .) by place.  The warp reads the oriented rows
// of u's neighbours v 32 entries at a time; an entry whose bit is set (a few
// in a hundred are no neighbour of u) joins a queue, and 32 queued entries at
// a time go through the table, so the divergent probes run with full warps.
// (One table probe per entry, without the bitmap, left 12 of 32 lanes active
// and took 5.5 ms where this takes 1.8; a binary search per entry of the
// shorter row took 3.1.)  COUNT (support schedule): every
// triangle adds its three witnesses to the per-class counts instead.
template <bool COUNT>
__global__ void __launch_bounds__(32 * kTriWarps) triangle_kernel(SparseArgs a, uint32_t *__restrict__ cnt_e) {
  __shared__ uint32_t s_bits[kTriWarps][kBloomWords];
  __shared__ int32_t s_key[kTriWarps][kTableSlots];
  __shared__ uint16_t s_val[kTriWarps][kTableSlots];  // place, colour << 8, passes << 15
  __shared__ uint2 s_mask[kTriWarps][kTableKeys];     // (shared atomics are native on 32-bit words)
  __shared__ int32_t s_qj[kTriWarps][64];             // queue: entry of v's row,
  __shared__ uint8_t s_qv[kTriWarps][64];             // place of v in u's row
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t *bits = s_bits[wib];
  int32_t *key = s_key[wib];
  uint16_t *val = s_val[wib];
  uint32_t *um = reinterpret_cast<uint32_t *>(s_mask[wib]);
  int32_t *qj = s_qj[wib];
  uint8_t *qv = s_qv[wib];
  const int64_t warp0 = ((int64_t)blockIdx.x * kTriWarps) + wib, warps = (int64_t)gridDim.x * kTriWarps;
  const int64_t total = *a.n_items;
  for (int64_t it = warp0; it < total; it += warps) {
    const int2 item = a.items[it];
    const int32_t u = item.x;
    const int64_t ub = a.row0[u];
    const int od = a.olen[u];
    const bool pu = COUNT || !a.vfail[u];
    int slots = 32;
    while (slots < 2 * od) slots <<= 1;
    const uint32_t smask = (uint32_t)slots - 1u;
    const int words = min(slots, kBloomWords);  // 32 bits a slot at most
    const uint32_t bmask = 32u * (uint32_t)words - 1u;
    for (int i = lane; i < slots; i += 32) key[i] = -1;
    for (int i = lane; i < words; i += 32) bits[i] = 0u;
    for (int i = lane; i < 2 * od; i += 32) um[i] = 0u;
    __syncwarp();
    for (int i = lane; i < od; i += 32) {
      const int32_t w = a.oadj[ub + i];
      const bool pw = COUNT || !a.vfail[w];
      const uint32_t hash = (uint32_t)w * 2654435761u;
      atomicOr(&bits[(hash >> 8 & bmask) >> 5], 1u << (hash >> 8 & 31u));
      uint32_t h = hash >> 16 & smask;
      while (atomicCAS(&key[h], -1, w) != -1) h = (h + 1) & smask;
      val[h] = (uint16_t)(i | a.col[w] << 8 | (pw ? 1 << 15 : 0));
    }
    __syncwarp();
    const int cu = a.col[u];
    const unsigned long long bu = 1ull << cu;
    int qn = 0;
    // the last min(qn, 32) entries of the queue through the table
    auto drain = [&]() {
      __syncwarp();
      const int take = min(qn, 32);
      if (lane < take) {
        const int q = qn - take + lane, pvl = qv[q];
        const int32_t v = a.oadj[ub + pvl];
        const int64_t at = a.row0[v] + qj[q];
        const int32_t w = a.oadj[at];
        uint32_t h = (uint32_t)w * 2654435761u >> 16 & smask;
        int32_t found;
        while ((found = key[h]) != w && found != -1) h = (h + 1) & smask;
        if (found == w) {
          const uint32_t x = val[h];
          const int place = x & 255, cw = (x >> 8) & 63, cv = a.col[v];
          if constexpr (COUNT) {
            atomicAdd(&cnt_e[(int64_t)a.oeid[ub + pvl] * a.k + cw], 1u);
            atomicAdd(&cnt_e[(int64_t)a.oeid[ub + place] * a.k + cv], 1u);
            atomicAdd(&cnt_e[(int64_t)a.oeid[at] * a.k + cu], 1u);
          } else {
            const bool pw = x >> 15, pv = !a.vfail[v];
            if (pu && pv) atomicOr(&um[2 * pvl + (cw >> 5)], 1u << (cw & 31));
            if (pu && pw) atomicOr(&um[2 * place + (cv >> 5)], 1u << (cv & 31));
            if (pv && pw) or_mask(a.mask, a.oeid[at], bu);
          }
        }
      }
      __syncwarp();
      // the tail of the queue was taken: nothing moves up
      qn -= take;
      __syncwarp();
    };
    const int v0 = item.y * kItemEdges, v1 = min(od, v0 + kItemEdges);
    for (int vbase = v0; vbase < v1; vbase += 32) {
      // the lanes look up 32 neighbours v at a time
      int32_t lo = 0;
      int64_t lb = 0;
      if (vbase + lane < v1) {
        const int32_t v = a.oadj[ub + vbase + lane];
        lb = a.row0[v];
        lo = a.olen[v];
      }
      const int cnt = min(32, v1 - vbase);
      for (int t = 0; t < cnt; t++) {
        const int32_t ol = __shfl_sync(0xffffffffu, lo, t);
        if (ol == 0) continue;
        const int32_t *vrow = a.oadj + __shfl_sync(0xffffffffu, lb, t);
        int32_t w = vrow[min(lane, ol - 1)];
        for (int j0 = 0; j0 < ol; j0 += 32) {
          const int32_t wn = vrow[min(j0 + 32 + lane, ol - 1)];  // the next 32 are on their way
          const uint32_t ha = (uint32_t)w * 2654435761u >> 8;
          const uint32_t ba = bits[(ha & bmask) >> 5] >> (ha & 31u);
          const bool ca = (ba & 1u) & (j0 + lane < ol);
          const uint32_t ma = __ballot_sync(0xffffffffu, ca);
          if (ma) {
            if (ca) {
              const int p = qn + __popc(ma & lt);
              qj[p] = j0 + lane;
              qv[p] = (uint8_t)(vbase + t);
            }
            qn += __popc(ma);
            if (qn >= 32) drain();
          }
          w = wn;
        }
      }
    }
    while (qn > 0) drain();
    if (!COUNT)
      for (int i = lane; i < od; i += 32) {
        const unsigned long long m = (unsigned long long)um[2 * i + 1] << 32 | um[2 * i];
        if (m) or_mask(a.mask, a.oeid[ub + i], m);
      }
    __syncwarp();
  }
}

// 3, for the oriented edges u -> v of rows too long for a table: one warp per
// edge, lanes walk the shorter of the two oriented rows, two entries at a time,
// and bisect the longer one for both, so that their loads travel together (the
// number of halvings is the same for every entry).  Bound by those chains of
// loads and by the atomics of the edges {u, w} and {v, w}; the classes of {u, v}
// are gathered in registers.  9000 vertices, k = 12, 3.7 million edges, most in
// such rows: 7.7 ms a pass, 14.5 with one entry at a time and three masks looked
// up per triangle.
template <bool COUNT>
__global__ void __launch_bounds__(256) triangle_big_kernel(SparseArgs a, uint32_t *__restrict__ cnt_e) {
  const int lane = threadIdx.x & 31;
  const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t total = *a.n_big;
  for (int64_t x = warp0; x < total; x += warps) {
    const int32_t u = a.big_u[x];
    const int64_t ub = a.row0[u], q = ub + a.big_i[x];
    const int32_t v = a.oadj[q], euv = a.oeid[q];
    const int64_t vb = a.row0[v];
    const int32_t nu = a.olen[u], nv = a.olen[v];
    const bool walk_u = nu <= nv;
    const int32_t walked = walk_u ? nu : nv, searched = walk_u ? nv : nu;
    const int32_t *wadj = a.oadj + (walk_u ? ub : vb), *sadj = a.oadj + (walk_u ? vb : ub);
    const int32_t *weid = a.oeid + (walk_u ? ub : vb), *seid = a.oeid + (walk_u ? vb : ub);
    const bool pu = COUNT || !a.vfail[u], pv = COUNT || !a.vfail[v];
    const int cu = a.col[u], cv = a.col[v];
    unsigned long long muv = 0;
    // entry i of the walked row and entry j of the other hold w
    const auto triangle = [&](int32_t i, int32_t j, int32_t w) {
      const int32_t euw = walk_u ? weid[i] : seid[j], evw = walk_u ? seid[j] : weid[i];
      if constexpr (COUNT) {
        atomicAdd(&cnt_e[(int64_t)euv * a.k + a.col[w]], 1u);
        atomicAdd(&cnt_e[(int64_t)euw * a.k + cv], 1u);
        atomicAdd(&cnt_e[(int64_t)evw * a.k + cu], 1u);
      } else {
        const int cw = a.vinfo[w].y;  // colour, and whether w fails
        muv |= 1ull << (cw & 63);
        if (cw >> kFailsShift & 1) return;
        if (pu) atomicOr(&a.mask[euw], 1ull << cv);
        if (pv) atomicOr(&a.mask[evw], 1ull << cu);
      }
    };
    for (int32_t i = lane; i < walked; i += 64) {
      const int32_t i2 = min(i + 32, walked - 1);
      const int32_t w = wadj[i], w2 = wadj[i2];
      int32_t j = 0, j2 = 0;
      for (int32_t len = searched; len > 1;) {
        const int32_t half = len >> 1;
        const int32_t y = sadj[j + half - 1], y2 = sadj[j2 + half - 1];
        j += y < w ? half : 0;
        j2 += y2 < w2 ? half : 0;
        len -= half;
      }
      if (sadj[j] == w) triangle(i, j, w);
      if (i + 32 < walked && sadj[j2] == w2) triangle(i2, j2, w2);
    }
    if constexpr (!COUNT) {
      const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)muv),
                     hi = __reduce_or_sync(0xffffffffu, (uint32_t)(muv >> 32));
      if (lane == 0 && pu && pv) or_mask(a.mask, euv, (unsigned long long)hi << 32 | lo);
    }
  }
}

// 4. The edge rule on the masks, over the oriented edges of passing vertices.
template <bool SHORT>
__global__ void __launch_bounds__(256) verdict_kernel(SparseArgs a) {
  unsigned long long de = 0;
  const auto row = [&](int32_t u, int64_t &b, int64_t &e) {
    b = a.row0[u];
    e = b + (a.vfail[u] ? 0 : a.olen[u]);
  };
  over_vertices<SHORT>(a, row, [&](const auto &G, int32_t, int64_t b, int64_t e) {
    for (int64_t j = b + G.lane(); j < e; j += G.kLanes) {
      if (a.vfail[a.oadj[j]]) continue;
      const int32_t ed = a.oeid[j];
      if (__popcll(a.mask[ed]) >= a.q - 2) continue;
      de++;
      if (a.apply) a.elive[ed] = 0;
    }
  });
  for (int o = 16; o > 0; o >>= 1) de += __shfl_down_sync(0xffffffffu, de, o);
  if ((threadIdx.x & 31) == 0 && de) atomicAdd(&a.st->pass_de, de);
}

// Of the edges spread over the list, one per CTA: how many are live (found[0])
// and fail the edge rule (found[1]).  The warps take the entries of the shorter
// row 32 at a time and bisect the longer one, until enough classes are covered;
// an edge still open after kSampleWalk entries counts as neither.
constexpr int kSampleWalk = 1024;

__global__ void __launch_bounds__(256) sample_kernel(SparseArgs a, const int32_t *__restrict__ eu,
                                                     const int32_t *__restrict__ ev, int64_t m,
                                                     unsigned long long *found) {
  __shared__ uint32_t s_cover[2];
  const int lane = threadIdx.x & 31;
  const int64_t e = m * blockIdx.x / gridDim.x;
  if (!a.all_live && !a.elive[e]) return;  // (the whole CTA)
  if (threadIdx.x < 2) s_cover[threadIdx.x] = 0u;
  __syncthreads();
  const int32_t *adj = a.from_input ? a.adj0 : a.adj, *eid = a.from_input ? a.eid0 : a.eid;
  const auto length = [&](int32_t x) { return (int32_t)(a.from_input ? a.row0[x + 1] - a.row0[x] : a.len[x]); };
  const int32_t u = eu[e], v = ev[e], nu = length(u), nv = length(v);
  const int32_t walked = min(nu, nv), searched = max(nu, nv);
  const int64_t wb = a.row0[nu <= nv ? u : v], sb = a.row0[nu <= nv ? v : u];
  const auto enough = [&]() {
    return __popc(((volatile uint32_t *)s_cover)[0]) + __popc(((volatile uint32_t *)s_cover)[1]) >= a.q - 2;
  };
  for (int32_t i0 = threadIdx.x - lane; i0 < min(walked, kSampleWalk); i0 += 256) {
    unsigned long long cm = 0;
    const int64_t i = wb + i0 + lane;
    if (i0 + lane < walked && (a.all_live || a.elive[eid[i]])) {
      const int32_t w = adj[i];
      int64_t j = sb;
      for (int32_t len = searched; len > 1;) {
        const int32_t half = len >> 1;
        if (adj[j + half - 1] < w) j += half;
        len -= half;
      }
      if (adj[j] == w && (a.all_live || a.elive[eid[j]])) cm = 1ull << a.col[w];
    }
    __syncwarp();
    const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)cm), hi = __reduce_or_sync(0xffffffffu, (uint32_t)(cm >> 32));
    if (lane < 2) atomicOr(&s_cover[lane], lane ? hi : lo);
    __syncwarp();
    if (__any_sync(0xffffffffu, enough())) break;
  }
  __syncthreads();
  if (threadIdx.x == 0 && (enough() || walked <= kSampleWalk)) {
    atomicAdd(&found[0], 1ull);
    if (!enough()) atomicAdd(&found[1], 1ull);
  }
}

// Closes the pass and empties the counters of the next one (ctr: the two
// lists' lengths, items, long-row edges).  report: whether the run goes on,
// vertices left, live edges before the pass and left.
__global__ void sparse_finish_kernel(DevState *st, unsigned int *ctr, int out, long long *report) {
  const unsigned long long tests = st->pass_tests, de = st->pass_de;
  report[0] = finish_pass(st, st->pass_dv, de, tests);
  report[1] = ctr[out];
  report[2] = (long long)tests;
  report[3] = (long long)(tests - de);
  st->pass_dv = st->pass_de = st->pass_tests = 0;
  ctr[out ^ 1] = ctr[2] = ctr[3] = 0;
}

__global__ void sparse_begin_kernel(DevState *st, int64_t max_sweeps, int64_t passes0, unsigned int *ctr,
                                    long long *report) {
  st->status = KZ_OK;
  st->cont = 1;
  st->sweeps = 0;
  st->passes = passes0;
  st->tests = 0;
  st->max_sweeps = max_sweeps;
  st->pass_dv = st->pass_de = st->pass_tests = 0;
  st->ticket = 0;
  st->bar_count = 0;
  st->bar_abort = 0;
  st->pass_word = 0;
  for (int i = 0; i < 2; i++) st->ppass[i][0] = st->ppass[i][1] = st->ppass[i][2] = 0;
  ctr[0] = ctr[1] = ctr[2] = ctr[3] = 0;
  report[0] = report[1] = 0;  // (sparse_sample counts there)
}

// ---------------------------------------------------------------------------
// the remnant on bitset rows
// ---------------------------------------------------------------------------

// The remnant's vertices are list[0 .. n'), its rows plane-major bitset rows
// (the layout of small_setup) indexed by place in the list, in Scratch::A0;
// its live edges are entries (i << 12 | j), dead ones kDeadEntry, a failing
// one marked by kFailBit between the two halves of a pass.
constexpr uint32_t kDeadEntry = 0xffffffffu, kFailBit = 0x80000000u;
static_assert(noalloc::kMaxN <= 4096, "twelve bits a vertex");
constexpr int kRemWarps = 16;
constexpr int kRemChunk = 8;   // entries a warp takes at a time
constexpr uint32_t kRemSpinLimit = 1u << 24;

struct RemnantArgs {
  noalloc::Scratch *s;
  SparseArgs a;
  const int32_t *list;
  uint32_t *entries;
  int32_t *eids;
  unsigned int *n_entries;
};

__global__ void remnant_colours_kernel(const int32_t *__restrict__ list, int32_t count, const int32_t *__restrict__ col,
                                       int32_t *__restrict__ out, int32_t *__restrict__ local) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  out[i] = col[list[i]];
  local[list[i]] = i;
}

__global__ void remnant_clear_kernel(noalloc::Scratch *s) {
  const int64_t words = (int64_t)s->h.desc.n * s->h.desc.ldw;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < words; i += (int64_t)gridDim.x * blockDim.x)
    s->A0[i] = 0u;
}

// Rows and entries of the live edges, one warp per vertex.
__global__ void remnant_pack_kernel(RemnantArgs r, const int32_t *__restrict__ local) {
  noalloc::Scratch *s = r.s;
  const SparseArgs &a = r.a;
  const int lane = threadIdx.x & 31, i = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (i >= s->h.desc.n) return;
  const int32_t u = r.list[i], ru = a.rank[u];
  const int64_t b = a.row0[u], e = b + a.len[u], at = (int64_t)i * s->h.desc.ldw;
  for (int64_t base = b; base < e; base += 32) {
    const int64_t t = base + lane;
    bool up = false;
    int32_t j = 0, ed = 0;
    if (t < e) {
      ed = a.eid[t];
      if (a.elive[ed]) {
        const int32_t v = a.adj[t];
        j = local[v];
        up = a.rank[v] > ru;
        const int p = s->pos[j];
        atomicOr(&s->A0[at + (p >> 5)], 1u << (p & 31));
      }
    }
    const uint32_t m = __ballot_sync(0xffffffffu, up);
    unsigned int first = 0;
    if (lane == 0 && m) first = atomicAdd(r.n_entries, (unsigned int)__popc(m));
    first = __shfl_sync(0xffffffffu, first, 0) + __popc(m & ((1u << lane) - 1u));
    if (up) {
      r.entries[first] = (uint32_t)i << 12 | (uint32_t)j;
      r.eids[first] = ed;
    }
  }
}

// Grid barrier of the cooperative remnant kernel (thread 0 of every CTA).  The
// last to arrive runs `close` and publishes its word; the others wait,
// bounded.  Returns the word (0 after an abort).
template <class Close>
__device__ __forceinline__ unsigned long long remnant_barrier(DevState *st, Close close) {
  __threadfence();
  const unsigned long long w0 = *((volatile unsigned long long *)&st->pass_word);
  if (atomicAdd(&st->bar_count, 1u) == gridDim.x - 1u) {
    __threadfence();
    const unsigned long long w = close(pass_word_gen(w0) + 1u);
    st->bar_count = 0;
    __threadfence();
    atomicExch(&st->pass_word, w);
    return w;
  }
  for (uint32_t spins = 0;; spins++) {
    const unsigned long long w = *((volatile unsigned long long *)&st->pass_word);
    if (pass_word_gen(w) != pass_word_gen(w0)) {
      __threadfence();
      return w;
    }
    if (*((volatile int32_t *)&st->bar_abort)) return 0;
    if (spins > kRemSpinLimit) {
      atomicCAS(&st->status, (int32_t)KZ_OK, (int32_t)KZ_ERR_TIMEOUT);
      atomicExch(&st->bar_abort, 1);
      return 0;
    }
    __nanosleep(32);
  }
}

// Classes (bit c) with a set bit among this lane's chunk of the AND of two
// rows (one row: y = x); chunk q holds words 4 q ..., of classes c, c + 1, ...
__device__ __forceinline__ uint32_t chunk_classes(const uint32_t *x, const uint32_t *y, int q, int quads, int k, int c) {
  uint32_t cov = 0;
  if (q < quads) {
    const uint4 a = reinterpret_cast<const uint4 *>(x)[q], b = reinterpret_cast<const uint4 *>(y)[q];
    const uint32_t w[4] = {a.x & b.x, a.y & b.y, a.z & b.z, a.w & b.w};
#pragma unroll
    for (int i = 0; i < 4; i++) {
      if (w[i]) cov |= 1u << c;
      if (++c == k) c = 0;
    }
  }
  return cov;
}

// The covered classes of a whole row pair, or at least `enough` of them, given
// those of its first 32 chunks.
__device__ __forceinline__ uint32_t rest_classes(uint32_t all, const uint32_t *x, const uint32_t *y, int quads, int k,
                                                 int c, int cstep, int enough) {
  const int lane = threadIdx.x & 31;
  for (int q0 = 32; q0 < quads && __popc(all) < enough; q0 += 32) {
    c += cstep;
    if (c >= k) c -= k;
    all |= __reduce_or_sync(0xffffffffu, chunk_classes(x, y, q0 + lane, quads, k, c));
  }
  return all;
}

// Every remaining pass in one cooperative launch.  First half: a warp per live
// edge ANDs the two rows (own-class words are zero, so no class needs
// masking), a warp per live vertex ORs its row; barrier, where the last CTA
// closes the pass; second half: the failing edges' bits and vertices go;
// barrier.  Rows, entries and live words stay in L2.
__global__ void __launch_bounds__(32 * kRemWarps, 1) remnant_kernel(RemnantArgs r) {
  __shared__ unsigned long long s_cnt[3], s_word;
  noalloc::Scratch *s = r.s;
  const SparseArgs &a = r.a;
  DevState *st = a.st;
  uint32_t *A = s->A0, *vf = s->A1;  // vf: per vertex, fails in this pass
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int n = s->h.desc.n, ldw = s->h.desc.ldw, k = a.k, quads = ldw / 4;
  const int c0 = 4 * lane % k, cstep = 128 % k;
  const int64_t warps = (int64_t)gridDim.x * kRemWarps, w = (int64_t)wib * gridDim.x + blockIdx.x;
  const int64_t total = *r.n_entries;
  int64_t sweep_no = *((volatile int64_t *)&st->sweeps);
  for (int pass = 0;; pass++) {
    if (threadIdx.x < 3) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    unsigned int tests = 0, de = 0, dv = 0;
    for (int64_t base = w * kRemChunk; base < total; base += warps * kRemChunk) {
      const uint32_t mine = lane < kRemChunk && base + lane < total ? r.entries[base + lane] : kDeadEntry;
      uint32_t todo = __ballot_sync(0xffffffffu, mine != kDeadEntry), failed = 0;
      tests += __popc(todo);
      while (todo) {
        // two edges at a time: their loads travel together
        const int t0 = __ffs(todo) - 1;
        todo &= todo - 1;
        const int t1 = todo ? __ffs(todo) - 1 : t0;
        todo &= todo - 1;
        const uint32_t e0 = __shfl_sync(0xffffffffu, mine, t0), e1 = __shfl_sync(0xffffffffu, mine, t1);
        const uint32_t *x0 = A + (int64_t)(e0 >> 12) * ldw, *y0 = A + (int64_t)(e0 & 4095u) * ldw;
        const uint32_t *x1 = A + (int64_t)(e1 >> 12) * ldw, *y1 = A + (int64_t)(e1 & 4095u) * ldw;
        uint32_t v0 = chunk_classes(x0, y0, lane, quads, k, c0), v1 = chunk_classes(x1, y1, lane, quads, k, c0);
        v0 = rest_classes(__reduce_or_sync(0xffffffffu, v0), x0, y0, quads, k, c0, cstep, a.q - 2);
        v1 = rest_classes(__reduce_or_sync(0xffffffffu, v1), x1, y1, quads, k, c0, cstep, a.q - 2);
        if (__popc(v0) < a.q - 2) failed |= 1u << t0;
        if (__popc(v1) < a.q - 2) failed |= 1u << t1;
      }
      if (failed >> lane & 1u) r.entries[base + lane] = mine | kFailBit;
      de += __popc(failed);
    }
    for (int64_t i = w; i < n; i += warps) {
      const int p = s->pos[i];
      if (!(*((volatile uint32_t *)&s->V0[p >> 5]) >> (p & 31) & 1u)) continue;
      const uint32_t *row = A + i * ldw;
      const uint32_t first = __reduce_or_sync(0xffffffffu, chunk_classes(row, row, lane, quads, k, c0));
      const bool fail = __popc(rest_classes(first, row, row, quads, k, c0, cstep, a.q - 1)) < a.q - 1;
      if (lane == 0) {
        vf[i] = fail ? 1u : 0u;
        if (fail) a.v_sweep[r.list[i]] = (int32_t)(sweep_no + 1);
      }
      dv += fail;
    }
    if (lane == 0) {
      if (tests) atomicAdd(&s_cnt[0], (unsigned long long)tests);
      if (de) atomicAdd(&s_cnt[1], (unsigned long long)de);
      if (dv) atomicAdd(&s_cnt[2], (unsigned long long)dv);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned long long *cnt = st->ppass[pass & 1];
      for (int i = 0; i < 3; i++)
        if (s_cnt[i]) atomicAdd(&cnt[i], s_cnt[i]);
      s_word = remnant_barrier(st, [&](uint32_t gen) {
        const unsigned long long t = atomicAdd(&cnt[0], 0ull), e = atomicAdd(&cnt[1], 0ull), v = atomicAdd(&cnt[2], 0ull);
        const int cont = finish_pass(st, v, e, t);
        cnt[0] = cnt[1] = cnt[2] = 0;
        return pass_word(gen, cont, 0, cont ? sweep_no + 1 : sweep_no);
      });
    }
    __syncthreads();
    if (!pass_word_cont(s_word)) break;
    for (int64_t base = w * kRemChunk; base < total; base += warps * kRemChunk) {
      const uint32_t mine = lane < kRemChunk && base + lane < total ? r.entries[base + lane] : kDeadEntry;
      if (mine == kDeadEntry || !(mine & kFailBit)) continue;
      const uint32_t i = (mine & ~kFailBit) >> 12, j = mine & 4095u;
      const int pi = s->pos[i], pj = s->pos[j];
      atomicAnd(&A[(int64_t)i * ldw + (pj >> 5)], ~(1u << (pj & 31)));
      atomicAnd(&A[(int64_t)j * ldw + (pi >> 5)], ~(1u << (pi & 31)));
      r.entries[base + lane] = kDeadEntry;
    }
    for (int64_t i = w; i < n; i += warps) {
      if (lane != 0) continue;
      const int p = s->pos[i];
      if ((*((volatile uint32_t *)&s->V0[p >> 5]) >> (p & 31) & 1u) && vf[i]) atomicAnd(&s->V0[p >> 5], ~(1u << (p & 31)));
    }
    __syncthreads();
    sweep_no++;
    if (threadIdx.x == 0)
      s_word = remnant_barrier(st, [&](uint32_t gen) { return pass_word(gen, 1, 0, sweep_no); });
    __syncthreads();
    if (!pass_word_cont(s_word)) break;
  }
}

// The survivors back into the flags.
__global__ void remnant_unpack_kernel(RemnantArgs r) {
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = tid; e < (int64_t)*r.n_entries; e += stride)
    if (r.entries[e] == kDeadEntry) r.a.elive[r.eids[e]] = 0;
  for (int64_t i = tid; i < r.s->h.desc.n; i += stride) {
    const int p = r.s->pos[i];
    if (!(r.s->V0[p >> 5] >> (p & 31) & 1u)) r.a.vlive[r.list[i]] = 0;
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

static int sms_here() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return std::max(sms, 1);
}

// The CSR structures of the caller's edges (d_edges: device int32[2 m_in],
// built on the device by sparse_build_csr, kz_csr.cu), the colours and the
// pass scratch.
kz_status sparse_load(kz_graph g, const int32_t *colour, int64_t m_in, const int32_t *d_edges, bool dedup,
                      cudaStream_t s) {
  const int32_t n = g->n;
  KZ_TRY(sparse_build_csr(g, d_edges, m_in, dedup, s));
  const size_t nn = (size_t)std::max(n, 1), mm = (size_t)std::max<int64_t>(g->m, 1);
  KZ_TRY(graph_alloc(g, &g->sp_adj, 2 * mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_eid, 2 * mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_oadj, 2 * mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_oeid, 2 * mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_len, nn, s));
  KZ_TRY(graph_alloc(g, &g->sp_olen, nn, s));
  KZ_TRY(graph_alloc(g, &g->sp_elive, mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_vlive, nn, s));
  KZ_TRY(graph_alloc(g, &g->sp_vfail, nn, s));
  KZ_TRY(graph_alloc(g, &g->sp_list[0], nn, s));
  KZ_TRY(graph_alloc(g, &g->sp_list[1], nn, s));
  KZ_TRY(graph_alloc(g, &g->sp_items, nn + mm / kItemEdges + 1, s));
  KZ_TRY(graph_alloc(g, &g->sp_big[0], mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_big[1], mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_col, nn, s));
  KZ_TRY(graph_alloc(g, &g->sp_vinfo, nn, s));
  KZ_TRY(graph_alloc(g, &g->sp_mask, mm, s));
  KZ_TRY(graph_alloc(g, &g->sp_ctr, 4, s));
  KZ_TRY(graph_alloc(g, &g->sp_report, 4, s));
  KZ_TRY(graph_alloc(g, &g->sp_v_sweep, nn, s));
  if (!g->st) {
    KZ_TRY(graph_alloc(g, &g->st, 1, s));
    KZ_CUDA_TRY(cudaMemsetAsync(g->st, 0, sizeof(DevState), s));
  }
  if (n) {
    KZ_TRY(h2d(g->sp_col, colour, sizeof(int32_t) * n, s));
    vinfo_kernel<<<std::min(8 * sms_here(), (n + 255) / 256), 256, 0, s>>>(g->sp_rank, g->sp_col, n, g->sp_vinfo);
    KZ_CUDA_TRY(cudaGetLastError());
  }
  g->has_csr = true;
  return sparse_reset(g, s);
}

kz_status sparse_reset(kz_graph g, cudaStream_t s) {
  const size_t n = (size_t)g->n, m = (size_t)g->m;
  KZ_CUDA_TRY(cudaMemsetAsync(g->sp_elive, 1, std::max<size_t>(m, 1), s));
  KZ_CUDA_TRY(cudaMemsetAsync(g->sp_vlive, 1, std::max<size_t>(n, 1), s));
  if (n) KZ_CUDA_TRY(cudaMemsetAsync(g->sp_v_sweep, 0, sizeof(int32_t) * n, s));
  g->sp_from_input = g->sp_all_live = true;
  return KZ_OK;
}

static SparseArgs sparse_args(kz_graph g, bool use_list, int in, bool apply) {
  SparseArgs a;
  a.n = g->n;
  a.k = g->k;
  a.q = g->k - g->slack;
  a.from_input = g->sp_from_input ? 1 : 0;
  a.all_live = g->sp_all_live ? 1 : 0;
  a.apply = apply ? 1 : 0;
  a.col = g->sp_col;
  a.rank = g->sp_rank;
  a.vinfo = g->sp_vinfo;
  a.row0 = g->sp_row0;
  a.adj0 = g->sp_adj0;
  a.eid0 = g->sp_eid0;
  a.adj = g->sp_adj;
  a.eid = g->sp_eid;
  a.len = g->sp_len;
  a.oadj = g->sp_oadj;
  a.oeid = g->sp_oeid;
  a.olen = g->sp_olen;
  a.elive = g->sp_elive;
  a.vlive = g->sp_vlive;
  a.vfail = g->sp_vfail;
  a.list = use_list ? g->sp_list[in] : nullptr;
  a.n_list = g->sp_ctr + in;
  a.list_out = g->sp_list[in ^ 1];
  a.n_out = g->sp_ctr + (in ^ 1);
  a.mask = g->sp_mask;
  a.items = g->sp_items;
  a.big_u = g->sp_big[0];
  a.big_i = g->sp_big[1];
  a.n_items = g->sp_ctr + 2;
  a.n_big = g->sp_ctr + 3;
  a.v_sweep = g->sp_v_sweep;
  a.st = g->st;
  return a;
}

static bool short_rows(kz_graph g) { return 2 * g->m < (int64_t)kShortRow * g->n; }

// Working and oriented rows of the live edges, no vertex left out, with the
// triangles' work items (support schedule).
kz_status sparse_orient_live(kz_graph g, cudaStream_t s) {
  KZ_CUDA_TRY(cudaMemsetAsync(g->sp_vfail, 0, (size_t)std::max(g->n, 1), s));
  if (g->n) vinfo_kernel<<<std::min(8 * sms_here(), (g->n + 255) / 256), 256, 0, s>>>(g->sp_rank, g->sp_col, g->n, g->sp_vinfo);
  KZ_CUDA_TRY(cudaMemsetAsync(g->sp_ctr, 0, 4 * sizeof(unsigned int), s));
  const auto orient = short_rows(g) ? orient_kernel<true> : orient_kernel<false>;
  orient<<<16 * sms_here(), 256, 0, s>>>(sparse_args(g, false, 0, true));
  KZ_CUDA_TRY(cudaGetLastError());
  g->sp_from_input = g->sp_all_live = false;
  return KZ_OK;
}

// The oriented rows' triangles into per-class edge counts (support schedule).
kz_status sparse_count_triangles(kz_graph g, uint32_t *cnt_e, cudaStream_t s) {
  const SparseArgs a = sparse_args(g, false, 0, true);
  triangle_kernel<true><<<5 * sms_here(), 32 * kTriWarps, 0, s>>>(a, cnt_e);
  triangle_big_kernel<true><<<8 * sms_here(), 256, 0, s>>>(a, cnt_e);
  return cuda_status(cudaGetLastError());
}

// Share of the edges that is live, and share of those that fail the edge rule
// now, from kSampleEdges of them, after sparse_begin: 8 us of the device at n =
// 80,000 (1.6 million edges), 16 at n = 200,000 (6 million), and a wait.
constexpr int kSampleEdges = 512;

kz_status sparse_sample(kz_graph g, cudaStream_t s, double *live, double *failing) {
  const int32_t samples = (int32_t)std::min<int64_t>(g->m, kSampleEdges);
  unsigned long long found[2] = {0, 0};
  *live = *failing = 0.0;
  if (samples == 0) return KZ_OK;
  unsigned long long *d_found = reinterpret_cast<unsigned long long *>(g->sp_report);
  sample_kernel<<<samples, 256, 0, s>>>(sparse_args(g, false, 0, false), g->sp_eu, g->sp_ev, g->m, d_found);
  KZ_CUDA_TRY(cudaGetLastError());
  KZ_CUDA_TRY(cudaMemcpyAsync(found, d_found, sizeof(found), cudaMemcpyDeviceToHost, s));
  KZ_CUDA_TRY(cudaStreamSynchronize(s));
  *live = (double)found[0] / samples;
  if (found[0]) *failing = (double)found[1] / (double)found[0];
  return KZ_OK;
}

// Whether the whole graph fits the bitset remnant.
bool sparse_fits_small(kz_graph g) {
  return g->n <= noalloc::kMaxN && g->k <= 32 && g->ldw <= noalloc::kMaxLdw &&
         (int64_t)g->n * g->ldw <= noalloc::kMaxWords && g->blocks.size() <= (size_t)noalloc::kMaxBlocks;
}

kz_status sparse_begin(kz_graph g, int64_t max_sweeps, cudaStream_t s) {
  sparse_begin_kernel<<<1, 1, 0, s>>>(g->st, max_sweeps, g->n == 0 ? 1 : 0, g->sp_ctr, g->sp_report);
  g->sp_use_list = false;
  g->sp_in = 0;
  g->sp_sweeps = 0;
  g->sp_tried = 0;
  return cuda_status(cudaGetLastError());
}

kz_status sparse_one_pass(kz_graph g, int64_t max_sweeps, cudaStream_t s, SparseReport *out) {
  const int sms = sms_here(), grid = 16 * sms;
  const bool apply = g->sp_sweeps < max_sweeps;
  const SparseArgs a = sparse_args(g, g->sp_use_list, g->sp_in, apply);
  const bool few = !a.list && short_rows(g);
  (few ? vertex_kernel<true> : vertex_kernel<false>)<<<grid, 256, 0, s>>>(a);
  (few ? orient_kernel<true> : orient_kernel<false>)<<<grid, 256, 0, s>>>(a);
  triangle_kernel<false><<<5 * sms, 32 * kTriWarps, 0, s>>>(a, nullptr);
  triangle_big_kernel<false><<<8 * sms, 256, 0, s>>>(a, nullptr);
  (few ? verdict_kernel<true> : verdict_kernel<false>)<<<grid, 256, 0, s>>>(a);
  sparse_finish_kernel<<<1, 1, 0, s>>>(g->st, g->sp_ctr, g->sp_in ^ 1, g->sp_report);
  KZ_CUDA_TRY(cudaGetLastError());
  long long r[4];
  KZ_CUDA_TRY(cudaMemcpyAsync(r, g->sp_report, sizeof(r), cudaMemcpyDeviceToHost, s));
  KZ_CUDA_TRY(cudaStreamSynchronize(s));
  out->cont = r[0] != 0;
  out->vertices = r[1];
  out->live_before = r[2];
  out->live = r[3];
  if (apply) {
    // the working rows and the vertex list now describe what the pass left
    g->sp_from_input = g->sp_all_live = false;
    g->sp_use_list = true;
    g->sp_in ^= 1;
  }
  if (out->cont) g->sp_sweeps++;
  return KZ_OK;
}

// The rest of the run on bitset rows, when the live vertices fit (*done tells).
// Tried again only once their number has halved: a layout may exceed the
// scratch through uneven classes.
kz_status sparse_finish_small(kz_graph g, int64_t max_sweeps, const SparseReport &r, cudaStream_t s, bool *done) {
  *done = false;
  const int64_t nv = r.vertices;
  if (nv < 1 || nv > noalloc::kMaxN || g->k > 32) return KZ_OK;
  if (g->sp_tried && 2 * nv > g->sp_tried) return KZ_OK;
  g->sp_tried = nv;
  if (!g->sp_small) {
    // without the scratch the passes simply go on
    noalloc::Scratch *p = nullptr;
    if (graph_alloc(g, &p, 1, s) != KZ_OK) return KZ_OK;
    g->sp_small = p;
  }
  noalloc::Scratch *p = static_cast<noalloc::Scratch *>(g->sp_small);
  const int32_t count = (int32_t)nv;
  const int32_t *list = g->sp_list[g->sp_in];
  int32_t *colours = g->sp_list[g->sp_in ^ 1], *local = g->sp_olen;  // free between passes
  remnant_colours_kernel<<<(count + 255) / 256, 256, 0, s>>>(list, count, g->sp_col, colours, local);
  small_setup(p, count, g->k, colours, s);
  KZ_CUDA_TRY(cudaGetLastError());
  int32_t status = 0;
  KZ_CUDA_TRY(cudaMemcpyAsync(&status, &p->h.status, sizeof(status), cudaMemcpyDeviceToHost, s));
  KZ_CUDA_TRY(cudaStreamSynchronize(s));
  if (status != KZ_OK) return KZ_OK;
  RemnantArgs r2;
  r2.s = p;
  r2.a = sparse_args(g, true, g->sp_in, true);
  r2.list = list;
  r2.entries = reinterpret_cast<uint32_t *>(g->sp_big[0]);
  r2.eids = g->sp_big[1];
  r2.n_entries = g->sp_ctr + 3;  // (zero between passes)
  const int sms = sms_here();
  remnant_clear_kernel<<<2 * sms, 256, 0, s>>>(p);
  remnant_pack_kernel<<<(count + 7) / 8, 256, 0, s>>>(r2, local);
  KZ_CUDA_TRY(cudaGetLastError());
  // one CTA per SM, all resident (16 warps and a few bytes of shared memory)
  void *args[] = {&r2};
  KZ_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)remnant_kernel, dim3(sms), dim3(32 * kRemWarps), args, 0, s));
  remnant_unpack_kernel<<<2 * sms, 256, 0, s>>>(r2);
  KZ_CUDA_TRY(cudaGetLastError());
  *done = true;
  return KZ_OK;
}

kz_status sparse_kernelize(kz_graph g, const kz_options &opt, cudaStream_t s) {
  const int64_t max_sweeps = opt.max_sweeps > 0 ? opt.max_sweeps : (int64_t)g->n + g->m + 1;
  KZ_TRY(sparse_begin(g, max_sweeps, s));
  if (g->n == 0) return KZ_OK;
  for (;;) {
    SparseReport r;
    KZ_TRY(sparse_one_pass(g, max_sweeps, s, &r));
    if (!r.cont) return KZ_OK;
    bool done = false;
    KZ_TRY(sparse_finish_small(g, max_sweeps, r, s, &done));
    if (done) return KZ_OK;
  }
}

// ---------------------------------------------------------------------------
// survivors to the host
// ---------------------------------------------------------------------------

constexpr int kFetchThreads = 256;
constexpr int kFetchChunk = 16 * kFetchThreads;  // edges per CTA, 16 flags a thread

__device__ __forceinline__ uint4 fetch_flags(const uint8_t *__restrict__ elive, int64_t m, int64_t at) {
  if (at + 16 <= m) return *reinterpret_cast<const uint4 *>(elive + at);
  uint32_t w[4] = {0, 0, 0, 0};
  for (int i = 0; i < 16 && at + i < m; i++) w[i >> 2] |= (uint32_t)elive[at + i] << (8 * (i & 3));
  return make_uint4(w[0], w[1], w[2], w[3]);
}

__global__ void __launch_bounds__(kFetchThreads) count_live_edges_kernel(const uint8_t *__restrict__ elive, int64_t m,
                                                                         int32_t *__restrict__ counts) {
  __shared__ int s_cnt;
  if (threadIdx.x == 0) s_cnt = 0;
  __syncthreads();
  const uint4 f = fetch_flags(elive, m, (int64_t)blockIdx.x * kFetchChunk + 16 * threadIdx.x);
  const int c = __reduce_add_sync(0xffffffffu, __popc(f.x) + __popc(f.y) + __popc(f.z) + __popc(f.w));
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(&s_cnt, c);
  __syncthreads();
  if (threadIdx.x == 0) counts[blockIdx.x] = s_cnt;
}

// The live edges in order, those below `cap`.
__global__ void __launch_bounds__(kFetchThreads) write_live_edges_kernel(const uint8_t *__restrict__ elive, int64_t m,
                                                                         const int32_t *__restrict__ eu,
                                                                         const int32_t *__restrict__ ev,
                                                                         const int64_t *__restrict__ offset, int64_t cap,
                                                                         int2 *__restrict__ out) {
  __shared__ int s_warp[kFetchThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t at = (int64_t)blockIdx.x * kFetchChunk + 16 * threadIdx.x;
  const uint4 f = fetch_flags(elive, m, at);
  const uint32_t w[4] = {f.x, f.y, f.z, f.w};
  const int mine = __popc(f.x) + __popc(f.y) + __popc(f.z) + __popc(f.w);
  int incl = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  int64_t pos = offset[blockIdx.x] + incl - mine;
  for (int i = 0; i < warp; i++) pos += s_warp[i];
  for (int i = 0; i < 16 && mine; i++)
    if ((w[i >> 2] >> (8 * (i & 3))) & 1u) {
      if (pos < cap) out[pos] = make_int2(eu[at + i], ev[at + i]);
      pos++;
    }
}

// The flags are counted and the survivors gathered on the device, so only
// they travel (a copy of every edge and flag, and a host scan, took 7.3 ms
// for 5.9M edges).  KZ_ERR_OOM when the allocator refuses the lists' memory.
static kz_status fetch_gathered(kz_graph g, uint8_t *vertex_alive, int32_t *edges_out, int64_t cap, int64_t *m_live) {
  const int64_t m = g->m;
  cudaStream_t s = g->stream;
  const int64_t chunks = (m + kFetchChunk - 1) / kFetchChunk;
  if (chunks > INT32_MAX) return KZ_ERR_UNSUPPORTED;
  // counts, offsets (and the total), partial sums of the scan
  const size_t off_at = ((size_t)chunks * 4 + 15) / 16 * 16, sums_at = off_at + 8 * ((size_t)chunks + 2);
  const size_t bytes = sums_at + 8 * ((size_t)chunks / kScanBlock + 2);
  uint8_t *tmp = (uint8_t *)dev_alloc(bytes, s);
  if (!tmp) return KZ_ERR_OOM;
  int32_t *counts = reinterpret_cast<int32_t *>(tmp);
  int64_t *offset = reinterpret_cast<int64_t *>(tmp + off_at), *sums = reinterpret_cast<int64_t *>(tmp + sums_at);
  int2 *d_out = nullptr;
  size_t out_bytes = 0;
  count_live_edges_kernel<<<(unsigned)chunks, kFetchThreads, 0, s>>>(g->sp_elive, m, counts);
  kz_status st = scan_counts(counts, chunks, offset, sums, offset + chunks + 1, s);
  if (st == KZ_OK) st = cuda_status(cudaMemcpyAsync(m_live, offset + chunks, 8, cudaMemcpyDeviceToHost, s));
  if (st == KZ_OK && vertex_alive && g->n)
    st = cuda_status(cudaMemcpyAsync(vertex_alive, g->sp_vlive, (size_t)g->n, cudaMemcpyDeviceToHost, s));
  // (also after a failure: no copy into the caller's memory may outlive the call)
  kz_status waited = cuda_status(cudaStreamSynchronize(s));
  if (st == KZ_OK) st = waited;
  const int64_t take = edges_out ? std::min<int64_t>(*m_live, cap) : 0;
  if (st == KZ_OK && take > 0) {
    out_bytes = (size_t)take * sizeof(int2);
    d_out = (int2 *)dev_alloc(out_bytes, s);
    if (!d_out) st = KZ_ERR_OOM;
    if (st == KZ_OK) {
      write_live_edges_kernel<<<(unsigned)chunks, kFetchThreads, 0, s>>>(g->sp_elive, m, g->sp_eu, g->sp_ev, offset,
                                                                         take, d_out);
      st = cuda_status(cudaGetLastError());
    }
    if (st == KZ_OK) st = cuda_status(cudaMemcpyAsync(edges_out, d_out, out_bytes, cudaMemcpyDeviceToHost, s));
    waited = cuda_status(cudaStreamSynchronize(s));
    if (st == KZ_OK) st = waited;
  }
  if (d_out) dev_free(d_out, out_bytes, s);
  dev_free(tmp, bytes, s);
  return st;
}

// The same without device memory: every edge and flag to the host, and a scan
// there.
static kz_status fetch_scanned(kz_graph g, uint8_t *vertex_alive, int32_t *edges_out, int64_t cap, int64_t *m_live) {
  const size_t m = (size_t)g->m;
  cudaStream_t s = g->stream;
  std::vector<int32_t> ends;
  std::vector<uint8_t> live;
  try {
    ends.resize(2 * m);
    live.resize(m);
  } catch (...) {
    return KZ_ERR_OOM;
  }
  kz_status st = KZ_OK;
  const auto copy = [&](void *dst, const void *src, size_t bytes) {
    if (st == KZ_OK && bytes) st = cuda_status(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, s));
  };
  copy(ends.data(), g->sp_eu, 4 * m);
  copy(ends.data() + m, g->sp_ev, 4 * m);
  copy(live.data(), g->sp_elive, m);
  if (vertex_alive) copy(vertex_alive, g->sp_vlive, (size_t)g->n);
  const kz_status waited = cuda_status(cudaStreamSynchronize(s));
  if (st == KZ_OK) st = waited;
  if (st != KZ_OK) return st;
  int64_t cnt = 0;
  for (size_t e = 0; e < m; e++) {
    if (!live[e]) continue;
    if (cnt < cap && edges_out) {
      edges_out[2 * cnt] = ends[e];
      edges_out[2 * cnt + 1] = ends[m + e];
    }
    cnt++;
  }
  *m_live = cnt;
  return KZ_OK;
}

// Edges up to which everything travels to the host: the gathering takes two
// requests, five launches and two waits, 100 us however few there are, and the
// scan 69 us for 434 edges, 87 for 20,000, 99 for 35,000 and 173 for 120,000.
constexpr int64_t kScanEdges = 32768;

kz_status sparse_fetch(kz_graph g, uint8_t *vertex_alive, int32_t *edges_out, int64_t cap, int64_t *m_live) {
  *m_live = 0;
  kz_status st = g->m > kScanEdges ? fetch_gathered(g, vertex_alive, edges_out, cap, m_live) : KZ_ERR_OOM;
  if (st == KZ_ERR_OOM) st = fetch_scanned(g, vertex_alive, edges_out, cap, m_live);
  return st;
}

kz_status sparse_vertex_alive(kz_graph g, uint8_t *host_alive, int64_t *n_live) {
  const size_t n = (size_t)g->n;
  std::vector<uint8_t> vl(std::max<size_t>(n, 1));
  if (n) KZ_CUDA_TRY(cudaMemcpy(vl.data(), g->sp_vlive, n, cudaMemcpyDeviceToHost));
  int64_t live = 0;
  for (size_t v = 0; v < n; v++) {
    live += vl[v];
    if (host_alive) host_alive[v] = vl[v];
  }
  if (n_live) *n_live = live;
  return KZ_OK;
}

kz_status sparse_v_sweep(kz_graph g, int32_t *host) {
  if (g->n) KZ_CUDA_TRY(cudaMemcpy(host, g->sp_v_sweep, sizeof(int32_t) * g->n, cudaMemcpyDeviceToHost));
  return KZ_OK;
}

}  // namespace kz

namespace kz {

// ---------------------------------------------------------------------------
// moving the live state between the bitset rows and the CSR flags
// ---------------------------------------------------------------------------

__global__ void bitset_to_flags_kernel(const uint32_t *__restrict__ A, const uint32_t *__restrict__ V, int32_t ldw,
                                       int32_t k, const int32_t *__restrict__ inv, const int32_t *__restrict__ coff,
                                       const int32_t *__restrict__ col, const int32_t *__restrict__ eu,
                                       const int32_t *__restrict__ ev, int64_t m, int32_t n,
                                       uint8_t *__restrict__ elive, uint8_t *__restrict__ vlive) {
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = tid; e < m; e += stride) {
    const int32_t x = inv[eu[e]], v = ev[e], y = inv[v];
    const int32_t c = col[v], i = y - coff[c];
    elive[e] = (uint8_t)((A[(int64_t)x * ldw + (i >> 5) * k + c] >> (i & 31)) & 1u);
  }
  for (int64_t v = tid; v < n; v += stride) {
    const int32_t c = col[v], i = inv[v] - coff[c];
    vlive[v] = (uint8_t)((V[(i >> 5) * k + c] >> (i & 31)) & 1u);
  }
}

__global__ void flags_to_bitset_kernel(uint32_t *__restrict__ A, uint32_t *__restrict__ V, int32_t ldw, int32_t k,
                                       const int32_t *__restrict__ inv, const int32_t *__restrict__ coff,
                                       const int32_t *__restrict__ col, const int32_t *__restrict__ eu,
                                       const int32_t *__restrict__ ev, int64_t m, int32_t n,
                                       const uint8_t *__restrict__ elive, const uint8_t *__restrict__ vlive) {
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = tid; e < m; e += stride) {
    if (!elive[e]) continue;
    const int32_t u = eu[e], v = ev[e], x = inv[u], y = inv[v];
    const int32_t cu = col[u], cv = col[v], iu = x - coff[cu], iv = y - coff[cv];
    atomicOr(&A[(int64_t)x * ldw + (iv >> 5) * k + cv], 1u << (iv & 31));
    atomicOr(&A[(int64_t)y * ldw + (iu >> 5) * k + cu], 1u << (iu & 31));
  }
  for (int64_t v = tid; v < n; v += stride) {
    if (!vlive[v]) continue;
    const int32_t c = col[v], i = inv[v] - coff[c];
    atomicOr(&V[(i >> 5) * k + c], 1u << (i & 31));
  }
}

kz_status state_to_sparse(kz_graph g, cudaStream_t s) {
  if (g->owner == KZ_PATH_SPARSE) return KZ_OK;
  if (!g->has_csr || !g->has_bitset) return KZ_ERR_UNSUPPORTED;
  int32_t cur = 0;
  KZ_CUDA_TRY(cudaMemcpyAsync(&cur, &g->st->cur, 4, cudaMemcpyDeviceToHost, s));
  KZ_CUDA_TRY(cudaStreamSynchronize(s));
  bitset_to_flags_kernel<<<4 * sms_here(), 256, 0, s>>>(g->A[cur & 1], g->V[cur & 1], g->ldw, g->k, g->d_inv,
                                                        g->d_coff, g->sp_col, g->sp_eu, g->sp_ev, g->m, g->n,
                                                        g->sp_elive, g->sp_vlive);
  KZ_CUDA_TRY(cudaGetLastError());
  g->owner = KZ_PATH_SPARSE;
  g->sp_all_live = false;  // (the working rows still hold every live edge)
  return KZ_OK;
}

kz_status state_to_bitset(kz_graph g, cudaStream_t s) {
  if (g->owner == KZ_PATH_BITSET) return KZ_OK;
  if (!g->has_csr || !g->has_bitset) return KZ_ERR_UNSUPPORTED;
  int32_t cur = 0;
  KZ_CUDA_TRY(cudaMemcpyAsync(&cur, &g->st->cur, 4, cudaMemcpyDeviceToHost, s));
  KZ_CUDA_TRY(cudaStreamSynchronize(s));
  uint32_t *A = g->A[cur & 1], *V = g->V[cur & 1];
  KZ_CUDA_TRY(cudaMemsetAsync(A, 0, (size_t)g->n * g->ldw * 4, s));
  KZ_CUDA_TRY(cudaMemsetAsync(V, 0, (size_t)g->ldw * 4, s));
  flags_to_bitset_kernel<<<4 * sms_here(), 256, 0, s>>>(A, V, g->ldw, g->k, g->d_inv, g->d_coff, g->sp_col,
                                                        g->sp_eu, g->sp_ev, g->m, g->n, g->sp_elive, g->sp_vlive);
  KZ_CUDA_TRY(cudaGetLastError());
  g->owner = KZ_PATH_BITSET;
  g->ab_synced = false;  // only the current buffer was rebuilt
  return KZ_OK;
}

}  // namespace kz
