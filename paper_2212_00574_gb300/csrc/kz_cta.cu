// kz_cta.cu -- whole-fixpoint-in-one-CTA kernel: the small-graph path and
// the batched persistent launch.
//
// One CTA runs every Jacobi pass of one graph (thesis Section 4.2 rules, see
// kz_rules.cuh) with __syncthreads() between passes, so no pass needs a new
// launch and no CTA ever waits on another.  A persistent grid (one CTA per
// SM) pulls graphs from an atomic queue in longest-first order.  A graph
// whose two ping-pong copies fit in shared memory is copied in once and
// swept there ("shared" mode); a larger one is swept in place in its global
// ping-pong buffers ("global" mode, L2-resident for the sizes of a batch).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include "kz_internal.cuh"
#include "kz_pack_tiles.cuh"
#include "kz_rules.cuh"
#include "kz_small.cuh"
#include "kz_sweep.cuh"

namespace kz {

constexpr int kCtaThreads = 512;
constexpr int kCtaWarps = kCtaThreads / 32;

struct CtaArgs {
  const CtaGraph *graphs;
  const int32_t *order;   // queue order (longest first)
  int32_t count;
  unsigned int *queue;    // next queue slot; null: CTA b takes order[b] only
  int32_t smem_words;     // dynamic shared memory available, in words
  int32_t slack;          // colours minus the clique size sought, every graph (0: the thesis's rules)
  int64_t max_sweeps;     // option value; <= 0 means n + m + 1 per graph
};

// First pair index of the warp's share, then the block X holding it.
__device__ __forceinline__ int find_x(const int32_t *__restrict__ pair_off, int nb, int64_t p) {
  int lo = 0, hi = nb;  // pair_off[lo] <= p < pair_off[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (pair_off[mid] <= p) lo = mid;
    else hi = mid;
  }
  return lo;
}

// The running record of one graph's fixpoint, kept in shared memory while
// its CTA works on it and written to the graph's DevState at the end.
struct CtaRun {
  int64_t sweeps, passes, tests, max_sweeps;
  int32_t cur, status;
};

template <int KMAX, bool SHARED>
__device__ void cta_fixpoint(const CtaGraph &G, int64_t max_sweeps, int slack, uint32_t *smem, unsigned long long *s_cnt,
                             int *s_flag, int32_t *s_rounds, CtaRun *run) {
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int k = G.k, ldw = G.ldw, nb = G.nb;
  DevState *st = G.st;
  int cur = st->cur;
  const size_t words = (size_t)G.n * ldw;

  uint32_t *Ac, *An, *Vc, *Vn;
  if (SHARED) {
    Ac = smem;
    An = smem + words;
    Vc = An + words;
    Vn = Vc + ldw;
    const uint32_t *src = cur ? G.A1 : G.A0;
    const uint32_t *vsrc = cur ? G.V1 : G.V0;
    const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
    uint4 *a4 = reinterpret_cast<uint4 *>(Ac);
    uint4 *n4 = reinterpret_cast<uint4 *>(An);
    for (size_t i = tid; i < words / 4; i += kCtaThreads) {
      const uint4 w = s4[i];
      a4[i] = w;
      n4[i] = w;
    }
    for (int i = tid; i < ldw; i += kCtaThreads) {
      Vc[i] = vsrc[i];
      Vn[i] = vsrc[i];
    }
  } else {
    Ac = cur ? G.A1 : G.A0;
    An = cur ? G.A0 : G.A1;
    Vc = cur ? G.V1 : G.V0;
    Vn = cur ? G.V0 : G.V1;
  }
  for (int c = tid; c < k; c += kCtaThreads) s_rounds[c] = G.rounds[c];
  if (tid == 0) {
    run->sweeps = 0;
    run->passes = G.n == 0 ? 1 : 0;
    run->tests = 0;
    run->max_sweeps = max_sweeps > 0 ? max_sweeps : (int64_t)G.n + G.m + 1;
    run->cur = cur;
    run->status = KZ_OK;
    s_cnt[0] = s_cnt[1] = s_cnt[2] = 0;
  }
  __syncthreads();

  const int64_t npairs = G.pair_off[nb];
  const int64_t share = (npairs + kCtaWarps - 1) / kCtaWarps;
  for (; G.n > 0;) {
    const int64_t sweep_no = run->sweeps;
    unsigned long long my_tests = 0, my_de = 0, my_dv = 0;
    // vertex rule, one warp per block
    for (int x = warp; x < nb; x += kCtaWarps) {
      const BlockDesc X = G.blocks[x];
      const bool valid_u = lane < X.size;
      const int u = X.base + lane;
      const uint32_t *rowu = Ac + (size_t)(valid_u ? u : X.base) * ldw;
      uint32_t Fu[KMAX];
      load_plane0<KMAX>(Fu, rowu, k, valid_u);
      const int wx = X.r * k + X.c;
      const uint32_t vword = Vc[wx];
      const bool live = valid_u && ((vword >> lane) & 1u);
      const uint64_t miss0 = plane0_vertex_missing<KMAX>(Fu, k, X.c);
      int cnt = (k - 1) - __popcll(miss0);
      if (live && cnt < k - 1 - slack) cnt += vertex_cover_beyond_plane0(rowu, k, s_rounds, miss0);
      const bool fail = live && cnt < k - 1 - slack;
      const uint32_t failmask = __ballot_sync(0xffffffffu, fail);
      if (lane == 0) {
        Vn[wx] = vword & ~failmask;
        my_dv += __popc(failmask);
      }
      if (fail && G.v_sweep) G.v_sweep[u] = (int32_t)(sweep_no + 1);
    }
    // edge rule over the warp's contiguous share of block pairs
    const int64_t p0 = (int64_t)warp * share;
    const int64_t p1 = min(npairs, p0 + share);
    if (p0 < p1) {
      int x = find_x(G.pair_off, nb, p0);
      BlockDesc X = G.blocks[x];
      int ybeg = G.boff[X.c + 1];
      bool valid_u = lane < X.size;
      int u = X.base + lane;
      const uint32_t *rowu = Ac + (size_t)(valid_u ? u : X.base) * ldw;
      uint32_t Fu[KMAX], P[KMAX];
      load_plane0<KMAX>(Fu, rowu, k, valid_u);
      int prev_cv = -1;
      for (int64_t p = p0; p < p1; p++) {
        while (p >= G.pair_off[x + 1]) {
          x++;
          X = G.blocks[x];
          ybeg = G.boff[X.c + 1];
          valid_u = lane < X.size;
          u = X.base + lane;
          rowu = Ac + (size_t)(valid_u ? u : X.base) * ldw;
          load_plane0<KMAX>(Fu, rowu, k, valid_u);
          prev_cv = -1;
        }
        const BlockDesc Y = G.blocks[ybeg + (int)(p - G.pair_off[x])];
        if (Y.c != prev_cv) {
          pair_mask<KMAX>(P, k, X.c, Y.c);
          prev_cv = Y.c;
        }
        const int wy = Y.r * k + Y.c;
        const uint32_t adjw = valid_u ? rowu[wy] : 0u;
        my_tests += __popc(adjw);
        const uint32_t *Ybase = Ac + (size_t)Y.base * ldw;
        const uint32_t del = edge_rule_block<KMAX>(
            Fu, P, rowu, adjw, k, slack, s_rounds, X.c, Y.c,
            [&](int b) { return Ybase + (size_t)b * ldw; },
            [&](int b) { return Ybase + (size_t)b * ldw; });
        if (valid_u) An[(size_t)u * ldw + wy] = adjw & ~del;
        my_de += __popc(del);
        const uint32_t delT = transpose_deletions(del);
        if (lane < Y.size) {
          const size_t wi = (size_t)(Y.base + lane) * ldw + X.r * k + X.c;
          An[wi] = Ac[wi] & ~delT;
        }
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      my_tests += __shfl_down_sync(0xffffffffu, my_tests, o);
      my_de += __shfl_down_sync(0xffffffffu, my_de, o);
      my_dv += __shfl_down_sync(0xffffffffu, my_dv, o);
    }
    if (lane == 0) {
      if (my_tests) atomicAdd(&s_cnt[0], my_tests);
      if (my_de) atomicAdd(&s_cnt[1], my_de);
      if (my_dv) atomicAdd(&s_cnt[2], my_dv);
    }
    __syncthreads();
    if (tid == 0) {  // close the pass in shared memory (the trace goes straight out)
      const unsigned long long dv = s_cnt[2], de = s_cnt[1];
      run->passes += 1;
      run->tests += (int64_t)s_cnt[0];
      int cont = 0;
      if (dv + de > 0) {
        if (run->sweeps >= run->max_sweeps) {
          run->status = KZ_ERR_LIMIT;
        } else {
          if (run->sweeps < kTraceCap) {
            st->trace_dv[run->sweeps] = (int64_t)dv;
            st->trace_de[run->sweeps] = (int64_t)de;
          }
          run->sweeps += 1;
          run->cur ^= 1;
          cont = 1;
        }
      }
      *s_flag = cont;
      s_cnt[0] = s_cnt[1] = s_cnt[2] = 0;
    }
    __syncthreads();
    if (!*s_flag) break;
    uint32_t *t = Ac;
    Ac = An;
    An = t;
    t = Vc;
    Vc = Vn;
    Vn = t;
    __syncthreads();
  }
  if (SHARED && G.n > 0) {
    // hand the final state back through buffer 0
    uint4 *d4 = reinterpret_cast<uint4 *>(G.A0);
    const uint4 *a4 = reinterpret_cast<const uint4 *>(Ac);
    for (size_t i = tid; i < words / 4; i += kCtaThreads) d4[i] = a4[i];
    for (int i = tid; i < ldw; i += kCtaThreads) G.V0[i] = Vc[i];
  }
  if (tid == 0) {  // the run's record (global mode: the live buffer is run->cur)
    st->sweeps = run->sweeps;
    st->passes = run->passes;
    st->tests = run->tests;
    st->max_sweeps = run->max_sweeps;
    st->status = run->status;
    st->cont = 0;
    st->cur = SHARED ? 0 : run->cur;
  }
  __syncthreads();
}

template <int KMAX>
__global__ void __launch_bounds__(kCtaThreads, 1) cta_fixpoint_kernel(CtaArgs a) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ unsigned long long s_cnt[3];
  __shared__ int s_flag;
  __shared__ int s_g;
  __shared__ int32_t s_rounds[KMAX];
  __shared__ CtaRun s_run;
  for (int round = 0;; round++) {
    if (threadIdx.x == 0) s_g = a.queue ? (int)atomicAdd(a.queue, 1u) : (round == 0 ? (int)blockIdx.x : a.count);
    __syncthreads();
    const int g = s_g;
    __syncthreads();
    if (g >= a.count) break;
    const CtaGraph G = a.graphs[a.order[g]];
    if (G.k > KMAX) continue;  // never scheduled: the host groups graphs by KMAX
    if (G.smem_words > 0 && G.smem_words <= a.smem_words)
      cta_fixpoint<KMAX, true>(G, a.max_sweeps, a.slack, smem, s_cnt, &s_flag, s_rounds, &s_run);
    else
      cta_fixpoint<KMAX, false>(G, a.max_sweeps, a.slack, smem, s_cnt, &s_flag, s_rounds, &s_run);
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

typedef void (*CtaFn)(CtaArgs);

static CtaFn pick_cta(int k, int &kmax) {
  if (k <= 8) { kmax = 8; return cta_fixpoint_kernel<8>; }
  if (k <= 16) { kmax = 16; return cta_fixpoint_kernel<16>; }
  if (k <= 32) { kmax = 32; return cta_fixpoint_kernel<32>; }
  kmax = 64;
  return cta_fixpoint_kernel<64>;
}

static int device_smem_optin() {
  int dev = 0, v = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return v;
}

// Shared memory words a graph needs for the shared mode (two copies of the
// rows and of the live words).
size_t cta_smem_words(kz_graph g) { return 2 * ((size_t)g->n * g->ldw + (size_t)g->ldw); }

static CtaGraph describe(kz_graph g, int64_t max_sweeps);

// Descriptor of the graph for single-graph in-CTA launches (needs every
// buffer of the graph allocated).
kz_status cta_upload_descriptor(kz_graph g, cudaStream_t s) {
  CtaGraph *d = nullptr;
  KZ_TRY(graph_alloc(g, &d, 1, s));
  g->d_cta_desc = d;
  KZ_TRY(graph_alloc(g, &g->d_zero, 4, s));
  KZ_CUDA_TRY(cudaMemsetAsync(g->d_zero, 0, 16, s));
  CtaGraph h = describe(g, 0);
  // staged (or, outside a load, a copy from pageable memory, which has left
  // the local by the time the call returns)
  KZ_TRY(h2d(d, &h, sizeof(h), s));
  return KZ_OK;
}

static CtaGraph describe(kz_graph g, int64_t max_sweeps) {
  CtaGraph d;
  memset(&d, 0, sizeof(d));
  d.A0 = g->A[0];
  d.A1 = g->A[1];
  d.V0 = g->V[0];
  d.V1 = g->V[1];
  d.v_sweep = g->v_sweep;
  d.st = g->st;
  d.blocks = g->d_blocks;
  d.rounds = g->d_rounds;
  d.pair_off = g->d_pair_off;
  d.boff = g->d_boff;
  d.n = g->n;
  d.k = g->k;
  d.ldw = g->ldw;
  d.nb = (int32_t)g->blocks.size();
  const size_t sw = cta_smem_words(g);
  d.smem_words = sw > (size_t)INT32_MAX ? -1 : (int32_t)sw;
  (void)max_sweeps;
  d.m = g->m;
  // cost estimate for the queue order: block pairs x class words
  d.cost = (int64_t)g->n_pairs * 32 * g->k + (int64_t)g->blocks.size() * g->k;
  return d;
}

bool cta_fits_shared(kz_graph g) {
  const size_t limit = (size_t)(device_smem_optin() / 4);
  return cta_smem_words(g) * 4 + 64 <= limit * 4;
}

// Kernelizes `count` graphs with persistent launches, one per KMAX group
// (one launch when every k <= 32, as in a batch of k-partite graphs).
kz_status cta_kernelize(kz_graph *gs, int count, const kz_options &opt, cudaStream_t s,
                        int force_mode) {
  if (count <= 0) return KZ_OK;
  const int optin = device_smem_optin();
  std::vector<CtaGraph> desc((size_t)count);
  for (int i = 0; i < count; i++) {
    desc[i] = describe(gs[i], opt.max_sweeps);
    if (force_mode == 0) desc[i].smem_words = -1;  // global mode everywhere
  }
  // group by KMAX, longest first inside a group
  int sms = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  CtaGraph *d_desc = (CtaGraph *)dev_alloc(sizeof(CtaGraph) * count, s);
  int32_t *d_order = (int32_t *)dev_alloc(sizeof(int32_t) * count, s);
  unsigned int *d_queue = (unsigned int *)dev_alloc(64, s);
  kz_status st = (d_desc && d_order && d_queue) ? KZ_OK : KZ_ERR_OOM;
  if (st == KZ_OK)
    st = cuda_status(cudaMemcpyAsync(d_desc, desc.data(), sizeof(CtaGraph) * count,
                                     cudaMemcpyHostToDevice, s));
  if (st == KZ_OK) st = cuda_status(cudaMemsetAsync(d_queue, 0, 64, s));
  std::vector<int32_t> order;
  int group = 0;
  for (int kmax_want : {8, 16, 32, 64}) {
    if (st != KZ_OK) break;
    std::vector<int32_t> idx;
    for (int i = 0; i < count; i++) {
      int km = 0;
      pick_cta(desc[i].k, km);
      if (km == kmax_want) idx.push_back(i);
    }
    if (idx.empty()) continue;
    std::sort(idx.begin(), idx.end(), [&](int a, int b) { return desc[a].cost > desc[b].cost; });
    const size_t off = order.size();
    order.insert(order.end(), idx.begin(), idx.end());
    int km = 0;
    CtaFn fn = pick_cta(desc[idx[0]].k, km);
    const int smem_bytes = std::max(0, optin - 1024);  // static shared memory of the kernel
    st = cuda_status(cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          smem_bytes));
    if (st != KZ_OK) break;
    CtaArgs a;
    a.graphs = d_desc;
    a.order = d_order + off;
    a.count = (int32_t)idx.size();
    a.queue = d_queue + 4 * group;  // each group its own 16-byte counter
    a.smem_words = smem_bytes / 4;
    a.slack = 0;  // the fused batch runs the thesis's rules only
    a.max_sweeps = opt.max_sweeps;
    const int grid = std::max(1, std::min<int>((int)idx.size(), sms));
    // order slice must be on the device before the launch
    st = cuda_status(cudaMemcpyAsync(d_order + off, order.data() + off, sizeof(int32_t) * idx.size(),
                                     cudaMemcpyHostToDevice, s));
    if (st != KZ_OK) break;
    fn<<<grid, kCtaThreads, smem_bytes, s>>>(a);
    st = cuda_status(cudaGetLastError());
    group++;
  }
  // (pageable host-to-device copies return once the source is staged, so
  // the host vectors may go out of scope here)
  if (d_desc) dev_free(d_desc, sizeof(CtaGraph) * count, s);
  if (d_order) dev_free(d_order, sizeof(int32_t) * count, s);
  if (d_queue) dev_free(d_queue, 64, s);
  return st;
}

static bool configure_once(CtaFn fn, int kmax, int bytes) {
  static bool done[4] = {false, false, false, false};
  const int slot = kmax == 8 ? 0 : kmax == 16 ? 1 : kmax == 32 ? 2 : 3;
  if (done[slot]) return true;
  if (cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) !=
      cudaSuccess)
    return false;
  done[slot] = true;
  return true;
}

kz_status cta_kernelize_one(kz_graph g, const kz_options &opt, cudaStream_t s) {
  int km = 0;
  CtaFn fn = pick_cta(g->k, km);
  const int max_bytes = std::max(0, device_smem_optin() - 1024);
  if (!configure_once(fn, km, max_bytes)) return KZ_ERR_CUDA;
  // ask only for what this graph's shared mode needs (a small graph should
  // not force the largest shared-memory carve-out)
  const size_t need = cta_smem_words(g) * 4;
  const int smem_bytes = need <= (size_t)max_bytes ? (int)((need + 15) / 16 * 16) : 0;
  CtaArgs a;
  a.graphs = g->d_cta_desc;
  a.order = g->d_zero;
  a.count = 1;
  a.queue = nullptr;
  a.smem_words = smem_bytes / 4;
  a.slack = g->slack;
  a.max_sweeps = opt.max_sweeps;
  fn<<<1, kCtaThreads, smem_bytes, s>>>(a);
  return cuda_status(cudaGetLastError());
}

}  // namespace kz

// ---------------------------------------------------------------------------
// kz_kernelize_dense_noalloc: one graph, start to finish, with no memory
// allocation at all.  Every intermediate lives in one file-scope device array
// (g_noalloc_scratch below) that each GPU loading the library keeps until the
// process exits; the caller passes device buffers for inputs and outputs.
// The fixpoint itself is a cooperative grid kernel (the in-CTA kernel above for
// the smallest graphs), reading its descriptor from that array.
// ---------------------------------------------------------------------------

// The scratch of kz_kernelize_dense_noalloc (about 9 MiB per device).
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(kz::noalloc::Scratch)];

namespace kz {
namespace noalloc {

// Layout of the caller's graph: colour classes, blocks, block pairs, the
// descriptor of the in-CTA kernel, the relabelling and the live words.  One
// CTA; every prefix over blocks is closed-form per class, so the blocks are
// filled in parallel.
__global__ void __launch_bounds__(1024) setup_kernel(Scratch *s, int32_t n, int32_t k,
                                                     const int32_t *__restrict__ colour) {
  Header &h = s->h;
  __shared__ int cnt[64], coff[65], boff[65], fill[64], pairs0[65], units0[65];
  __shared__ int bad, status, ldw_s;
  const int tid = threadIdx.x;
  if (tid < 64) cnt[tid] = 0;
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int v = tid; v < n; v += blockDim.x) {
    const int c = colour[v];
    if (c < 0 || c >= k) atomicExch(&bad, (int)KZ_ERR_COLOUR_RANGE);
    else atomicAdd(&cnt[c], 1);
  }
  __syncthreads();
  if (tid == 0) {
    int R = 1;
    coff[0] = boff[0] = 0;
    for (int c = 0; c < k; c++) {
      const int rounds = (cnt[c] + 31) / 32;
      coff[c + 1] = coff[c] + cnt[c];
      boff[c + 1] = boff[c] + rounds;
      fill[c] = coff[c];
      R = max(R, rounds);
    }
    const int nb = boff[k];
    pairs0[0] = units0[0] = 0;
    for (int c = 0; c < k; c++) {
      const int rounds = boff[c + 1] - boff[c], with = nb - boff[c + 1];  // blocks of higher classes
      pairs0[c + 1] = pairs0[c] + rounds * with;
      units0[c + 1] = units0[c] + rounds * max(with, 1);
    }
    const int64_t ldw = ((int64_t)R * k + 3) / 4 * 4;
    int st = bad;
    if (!st && (ldw > kMaxLdw || (int64_t)n * ldw > kMaxWords || nb > kMaxBlocks)) st = KZ_ERR_UNSUPPORTED;
    if (!st) {
      CtaGraph &d = h.desc;
      d.A0 = s->A0;
      d.A1 = s->A1;
      d.V0 = s->V0;
      d.V1 = s->V1;
      d.v_sweep = s->v_sweep;
      d.st = &s->st;
      d.blocks = h.blocks;
      d.rounds = h.rounds;
      d.pair_off = h.pair_off;
      d.boff = h.boff;
      d.n = n;
      d.k = k;
      d.ldw = (int32_t)ldw;
      d.nb = nb;
      d.smem_words = (int32_t)(2 * ((int64_t)n * ldw + ldw));
      d.m = 0;
      d.cost = 0;
      int64_t cross = 0;
      for (int c = 0; c < k; c++) cross += (int64_t)cnt[c] * coff[c];
      h.cross = cross;
      h.bits = 0;
      h.R = R;
      DevState &ds = s->st;
      ds.cur = 0;
      ds.status = KZ_OK;
      ds.cont = 0;
      ds.sweeps = ds.passes = ds.tests = 0;
      ds.pass_dv = ds.pass_de = ds.pass_tests = 0;
      ds.ticket = 0;
      ds.bar_count = 0;
      ds.bar_abort = 0;
      ds.pass_word = 0;
      for (int i = 0; i < 2; i++) ds.ppass[i][0] = ds.ppass[i][1] = ds.ppass[i][2] = 0;
      h.pair_off[nb] = pairs0[k];
      h.unit_off[nb] = units0[k];
    }
    h.status = st;
    h.illegal = 0;
    status = st;
    ldw_s = (int)ldw;
  }
  __syncthreads();
  if (status) return;
  for (int i = tid; i < ldw_s; i += blockDim.x) s->V0[i] = s->V1[i] = 0u;
  if (tid <= k) {
    h.coff[tid] = coff[tid];
    h.boff[tid] = boff[tid];
    if (tid < k) h.rounds[tid] = boff[tid + 1] - boff[tid];
  }
  __syncthreads();
  const int nb = boff[k];
  for (int b = tid; b < nb; b += blockDim.x) {
    int c = 0;
    while (boff[c + 1] <= b) c++;
    const int r = b - boff[c], with = nb - boff[c + 1];
    BlockDesc d;
    d.c = c;
    d.r = r;
    d.base = coff[c] + 32 * r;
    d.size = min(32, cnt[c] - 32 * r);
    h.blocks[b] = d;
    h.pair_off[b] = pairs0[c] + r * with;
    h.unit_off[b] = units0[c] + r * max(with, 1);
    s->V0[r * k + c] = s->V1[r * k + c] = d.size >= 32 ? 0xffffffffu : ((1u << d.size) - 1u);
  }
  // relabel: every class a contiguous id range (order inside a class is free:
  // the fixpoint and every count reported do not depend on it)
  for (int v = tid; v < n; v += blockDim.x) {
    const int c = colour[v], x = atomicAdd(&fill[c], 1), i = x - coff[c];
    s->inv[v] = x;
    s->perm[x] = v;
    s->pos[v] = (((i >> 5) * k + c) << 5) | (i & 31);
    s->v_sweep[v] = 0;
  }
}

// Caller's dense bit matrix (strict upper triangle) into both copies of the
// block-plane rows (kz_pack_tiles.cuh).
__global__ void __launch_bounds__(kTileThreads) pack_kernel(Scratch *s, const uint64_t *__restrict__ bits,
                                                            int64_t row_words, const int32_t *__restrict__ colour) {
  extern __shared__ __align__(16) uint32_t colw[];  // 32 * ceil(n / 32) column words
  __shared__ int32_t scoff[65];
  Header &h = s->h;
  if (h.status) return;
  const int n = h.desc.n, k = h.desc.k, lane = threadIdx.x & 31;
  if (threadIdx.x <= k) scoff[threadIdx.x] = h.coff[threadIdx.x];
  unsigned long long mine = 0;
  bool bad = false;
  for (int64_t i0 = (int64_t)blockIdx.x * 32; i0 < n; i0 += (int64_t)gridDim.x * 32) {
    const int rows = min(32, n - (int)i0);
    __syncthreads();
    tile_columns(colw, bits, row_words, n, i0, rows);
    __syncthreads();
    const bool valid = lane < rows;
    mine += tile_rows(colw, s->A0, s->A1, nullptr, h.desc.ldw, k, h.R, scoff, s->perm,
                      valid ? s->inv[i0 + lane] : 0, valid ? colour[i0 + lane] : -1, valid, &bad);
  }
  if (bad) atomicCAS(&h.illegal, 0, (int32_t)KZ_ERR_ILLEGAL_COLOURING);
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, o);
  if (lane == 0 && mine) atomicAdd(&h.bits, mine);
}

// The in-CTA fixpoint on the scratch descriptor (k <= 32).
__global__ void __launch_bounds__(kCtaThreads, 1) fixpoint_kernel(Scratch *s, int64_t max_sweeps,
                                                                        int32_t smem_words) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ unsigned long long s_cnt[3];
  __shared__ int s_flag;
  __shared__ int32_t s_rounds[32];
  __shared__ CtaRun s_run;
  if (s->h.status || s->h.illegal) return;
  CtaGraph G = s->h.desc;
  G.m = (int64_t)(s->h.bits / 2);
  if (G.smem_words > 0 && G.smem_words <= smem_words)
    cta_fixpoint<32, true>(G, max_sweeps, 0, smem, s_cnt, &s_flag, s_rounds, &s_run);
  else
    cta_fixpoint<32, false>(G, max_sweeps, 0, smem, s_cnt, &s_flag, s_rounds, &s_run);
}

// The fixpoint over the whole GPU, in one cooperative launch: every warp owns
// a consecutive share of the units (block X against one block Y of a higher
// class, or a block X without partners), runs of one X at a time
// (sweep_item, kz_sweep.cuh: plane 0 of the Y rows staged by asynchronous
// copies, one block ahead), and a grid barrier closes each pass.  The barrier
// wait is bounded; one that runs out records KZ_ERR_TIMEOUT and every CTA
// leaves.
//
// Why a grid: one CTA leaves 151 SMs idle.  A pass of n = 1501, k = 12,
// p = 0.3 (1,100 block pairs) took 2.8 ms on one CTA and takes 26 us here;
// n = 4096, k = 20, p = 0.92: 10.9 ms and 44 us.  Bound by latency: a warp has
// about one unit, and its recounts are chains of loads.  Below density 0.42
// the first test takes two planes (42 to 26 us a pass on the first graph).
constexpr int kGridWarps = 8;
constexpr uint32_t kGridSpinLimit = 1u << 24;
constexpr double kGridTwoPlaneDensity = 0.42;

template <int KMAX>
__global__ void __launch_bounds__(kGridWarps * 32, 1) grid_fixpoint_kernel(Scratch *s, int64_t max_sweeps_opt) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ unsigned long long s_cnt[3];
  __shared__ unsigned long long s_word;
  const Header &h = s->h;
  if (h.status || h.illegal) return;
  DevState *st = &s->st;
  const CtaGraph &d = h.desc;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nb = d.nb;
  uint32_t *buf0 = smem + wib * 2 * 32 * 2 * KMAX;
  uint32_t *buf1 = buf0 + 32 * 2 * KMAX;
  // the two-plane first test below the density where it wins on the
  // single-graph sweep kernels
  const bool two = h.R >= 2 && (double)(h.bits / 2) < kGridTwoPlaneDensity * (double)h.cross;
  const int64_t max_sweeps = max_sweeps_opt > 0 ? max_sweeps_opt : (int64_t)d.n + (int64_t)(h.bits / 2) + 1;
  if (blockIdx.x == 0 && threadIdx.x == 0) st->max_sweeps = max_sweeps;  // the closing CTA reads it behind the barrier
  GraphView G;
  G.blocks = h.blocks;
  G.rounds = h.rounds;
  G.A0 = s->A0;
  G.A1 = s->A1;
  G.V0 = s->V0;
  G.V1 = s->V1;
  G.v_sweep = s->v_sweep;
  G.k = d.k;
  G.ldw = d.ldw;
  const int64_t units = h.unit_off[nb];
  // neighbouring warps of the share order sit on different SMs
  const int64_t warps = (int64_t)gridDim.x * kGridWarps, w = (int64_t)wib * gridDim.x + blockIdx.x;
  const int u0 = (int)(units * w / warps), u1 = (int)(units * (w + 1) / warps);
  const int x0 = u0 < u1 ? find_x(h.unit_off, nb, u0) : 0;
  int cur = 0;
  int64_t sweep_no = 0;
  for (int pass = 0;; pass++) {
    if (threadIdx.x < 3) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    PassCounters pc;
    for (int u = u0, x = x0; u < u1; x++) {
      const int e = min(u1, h.unit_off[x + 1]);
      const int ybeg = min(h.boff[h.blocks[x].c + 1], nb);
      WorkItem item;
      item.x = x;
      item.vflag = u == h.unit_off[x];
      item.y0 = ybeg < nb ? ybeg + (u - h.unit_off[x]) : nb;
      item.y1 = ybeg < nb ? ybeg + (e - h.unit_off[x]) : nb;
      if (two) sweep_item<KMAX, true>(G, item, cur, sweep_no, buf0, buf1, pc);
      else sweep_item<KMAX>(G, item, cur, sweep_no, buf0, buf1, pc);
      u = e;
    }
    for (int o = 16; o > 0; o >>= 1) {
      pc.tests += __shfl_down_sync(0xffffffffu, pc.tests, o);
      pc.de += __shfl_down_sync(0xffffffffu, pc.de, o);
      pc.dv += __shfl_down_sync(0xffffffffu, pc.dv, o);
    }
    if (lane == 0) {
      if (pc.tests) atomicAdd(&s_cnt[0], pc.tests);
      if (pc.de) atomicAdd(&s_cnt[1], pc.de);
      if (pc.dv) atomicAdd(&s_cnt[2], pc.dv);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned long long *cnt = st->ppass[pass & 1];
      for (int i = 0; i < 3; i++)
        if (s_cnt[i]) atomicAdd(&cnt[i], s_cnt[i]);
      __threadfence();
      const unsigned long long w0 = *((volatile unsigned long long *)&st->pass_word);
      unsigned long long word = w0;
      bool abort = false;
      if (atomicAdd(&st->bar_count, 1u) == gridDim.x - 1u) {
        // the last CTA closes the pass and releases the others
        __threadfence();
        const unsigned long long tests = atomicAdd(&cnt[0], 0ull);
        const unsigned long long de = atomicAdd(&cnt[1], 0ull);
        const unsigned long long dv = atomicAdd(&cnt[2], 0ull);
        const int cont = finish_pass(st, dv, de, tests);
        cnt[0] = cnt[1] = cnt[2] = 0;
        st->bar_count = 0;
        word = pass_word(pass_word_gen(w0) + 1u, cont, cont ? cur ^ 1 : cur, cont ? sweep_no + 1 : sweep_no);
        __threadfence();
        atomicExch(&st->pass_word, word);
      } else {
        for (uint32_t spins = 0;; spins++) {
          word = *((volatile unsigned long long *)&st->pass_word);
          if (pass_word_gen(word) != pass_word_gen(w0)) break;
          abort = *((volatile int32_t *)&st->bar_abort) != 0;
          if (!abort && spins > kGridSpinLimit) {
            atomicCAS(&st->status, (int32_t)KZ_OK, (int32_t)KZ_ERR_TIMEOUT);
            atomicExch(&st->bar_abort, 1);
            abort = true;
          }
          if (abort) break;
          __nanosleep(32);
        }
      }
      __threadfence();
      s_word = abort ? 0ull : word;  // a cleared continue bit ends the kernel
    }
    __syncthreads();
    const unsigned long long word = s_word;
    if (!pass_word_cont(word)) break;
    cur = pass_word_cur(word);
    sweep_no = pass_word_sweeps(word);
  }
}

typedef void (*GridFn)(Scratch *, int64_t);

static GridFn pick_grid(int k, int &kmax) {
  if (k <= 8) { kmax = 8; return grid_fixpoint_kernel<8>; }
  if (k <= 16) { kmax = 16; return grid_fixpoint_kernel<16>; }
  if (k <= 24) { kmax = 24; return grid_fixpoint_kernel<24>; }
  kmax = 32;
  return grid_fixpoint_kernel<32>;
}

constexpr size_t grid_smem(int kmax) { return (size_t)kGridWarps * 2 * 32 * 2 * kmax * 4; }

static kz_status configure_grid() {
  for (int kk = 8; kk <= 32; kk += 8) {
    int km = 0, per_sm = 0;
    const GridFn fn = pick_grid(kk, km);
    KZ_CUDA_TRY(cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)grid_smem(km)));
    KZ_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)fn, kGridWarps * 32,
                                                              grid_smem(km)));
    if (per_sm < 1) return KZ_ERR_UNSUPPORTED;
  }
  return KZ_OK;
}

// One CTA per SM at most (all resident, as the grid barrier needs), and no
// more warps than the block pairs the classes can make.
static kz_status launch_grid(Scratch *sp, int32_t n, int32_t k, int64_t max_sweeps, int sms, cudaStream_t s) {
  int km = 0;
  const GridFn fn = pick_grid(k, km);
  const int64_t blocks = n / 32 + k, pairs = blocks * blocks / 2;
  const int ctas = (int)std::max<int64_t>(1, std::min<int64_t>(std::max(sms, 1), (pairs + kGridWarps - 1) / kGridWarps));
  void *args[] = {&sp, &max_sweeps};
  KZ_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)fn, dim3(ctas), dim3(kGridWarps * 32), args, grid_smem(km), s));
  return KZ_OK;
}

// Vertices up to which one CTA runs the fixpoint from shared memory: below
// it a pass is shorter than a grid barrier (n = 100: 9.7 us a pass on one CTA,
// n = 200: 8.1 us on the grid).
constexpr int kOneCtaMaxN = 64;

// Kernel rows back to caller ids: the symmetric bit matrix, the live
// vertices, and (sweeps, passes, edge tests, status).  A CTA stages one
// relabelled row; its warps gather the row's 32 positions of 32 caller
// columns at a time, and a ballot is half an output word.
constexpr int kUnpackThreads = 128;

__global__ void __launch_bounds__(kUnpackThreads) unpack_kernel(Scratch *s, int32_t n_in, uint64_t *__restrict__ out,
                                                                int64_t row_words, uint8_t *__restrict__ alive,
                                                                int64_t *__restrict__ counts) {
  __shared__ uint32_t srow[kMaxLdw];
  const Header &h = s->h;
  const int status = h.status ? h.status : h.illegal;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (status) {
    // a rejected input leaves defined outputs: no vertex, no edge, zero
    // counts and the status
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = tid; i < (int64_t)n_in * row_words; i += stride) out[i] = 0ull;
    for (int64_t v = tid; v < n_in; v += stride) alive[v] = 0;
    if (tid == 0) {
      counts[0] = counts[1] = counts[2] = 0;
      counts[3] = status;
    }
    return;
  }
  const int n = h.desc.n, ldw = h.desc.ldw, cur = s->st.cur;
  const uint32_t *A = cur ? s->A1 : s->A0;
  const uint32_t *V = cur ? s->V1 : s->V0;
  for (int v = blockIdx.x; v < n; v += gridDim.x) {
    __syncthreads();  // the previous row is consumed
    const uint4 *row = reinterpret_cast<const uint4 *>(A + (int64_t)s->inv[v] * ldw);
    for (int i = threadIdx.x; i < ldw / 4; i += kUnpackThreads) reinterpret_cast<uint4 *>(srow)[i] = row[i];
    __syncthreads();
    uint64_t *dst = out + (int64_t)v * row_words;
    for (int64_t w = warp; w < row_words; w += kUnpackThreads / 32) {
      uint32_t half[2];
#pragma unroll
      for (int q = 0; q < 2; q++) {
        const int64_t col = 64 * w + 32 * q + lane;
        const int p = col < n ? s->pos[col] : -1;
        half[q] = __ballot_sync(0xffffffffu, p >= 0 && ((srow[p >> 5] >> (p & 31)) & 1u));
      }
      if (lane == 0) dst[w] = (uint64_t)half[0] | (uint64_t)half[1] << 32;
    }
    if (threadIdx.x == 0) {
      const int p = s->pos[v];
      alive[v] = (uint8_t)((V[p >> 5] >> (p & 31)) & 1u);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    counts[0] = s->st.sweeps;
    counts[1] = s->st.passes;
    counts[2] = s->st.tests;
    counts[3] = s->st.status;
  }
}

}  // namespace noalloc

void small_setup(noalloc::Scratch *s, int32_t n, int32_t k, const int32_t *colour, cudaStream_t stream) {
  noalloc::setup_kernel<<<1, 1024, 0, stream>>>(s, n, k, colour);
}

}  // namespace kz

namespace {

// Device address of the scratch array, looked up once per device (host code
// cannot use the array's name as a device pointer).
std::mutex g_noalloc_mu;
void *g_noalloc_addr[64] = {nullptr};

kz_status noalloc_scratch(void **out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return KZ_ERR_CUDA;
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_addr[dev]) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) return KZ_ERR_CUDA;
    g_noalloc_addr[dev] = p;
  }
  *out = g_noalloc_addr[dev];
  return KZ_OK;
}

}  // namespace

extern "C" kz_status kz_kernelize_dense_noalloc(int32_t n, int32_t k, const int32_t *colour,
                                                const uint64_t *adj_bits, int64_t row_words,
                                                int64_t max_sweeps, uint8_t *vertex_alive,
                                                uint64_t *adj_out, int64_t *counts, void *stream) {
  using namespace kz::noalloc;
  if (n < 0 || k < 1 || k > 32) return KZ_ERR_ARG;
  if (n > kMaxN) return KZ_ERR_UNSUPPORTED;
  if (row_words < (int64_t)((n + 63) / 64) || !counts) return KZ_ERR_ARG;
  if (n > 0 && (!colour || !adj_bits || !vertex_alive || !adj_out)) return KZ_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  void *scratch = nullptr;
  KZ_TRY(noalloc_scratch(&scratch));  // device address of the array on this device
  Scratch *sp = static_cast<Scratch *>(scratch);
  int dev = 0, sms = 1, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int smem_bytes = std::max(0, optin - 1024);
  {
    static std::mutex mu;
    static bool configured[64] = {false};
    std::lock_guard<std::mutex> lk(mu);
    if (!configured[dev]) {
      KZ_CUDA_TRY(cudaFuncSetAttribute((const void *)fixpoint_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes));
      KZ_TRY(configure_grid());  // every width is set up (and loaded) now, so that no later call does
      configured[dev] = true;
    }
  }
  kz::small_setup(sp, n, k, colour, s);
  if (n > 0) pack_kernel<<<(n + 31) / 32, kz::kTileThreads, (size_t)(n + 31) / 32 * 128, s>>>(sp, adj_bits, row_words, colour);
  if (n <= kOneCtaMaxN) {
    fixpoint_kernel<<<1, kz::kCtaThreads, smem_bytes, s>>>(sp, max_sweeps, smem_bytes / 4);
  } else {
    KZ_TRY(launch_grid(sp, n, k, max_sweeps, sms, s));
  }
  unpack_kernel<<<std::max(1, std::min(n, 16 * std::max(sms, 1))), kUnpackThreads, 0, s>>>(sp, n, adj_out, row_words,
                                                                                          vertex_alive, counts);
  KZ_CUDA_TRY(cudaGetLastError());
  // synchronous: the device status decides the return value
  int64_t status = 0;
  KZ_CUDA_TRY(cudaMemcpyAsync(&status, counts + 3, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  KZ_CUDA_TRY(cudaStreamSynchronize(s));
  return (kz_status)status;
}
