// multi.cu -- Skipper over many independent graphs in one persistent launch,
// each graph in its own device buffers (mm_skipper_multi), and the exact
// checker over all of them at once (mm_validate_multi).
//
// Graphs are described by a table of (n, nnz, offsets, nbrs, mate) entries
// copied to the device per call; nothing is repacked.  Every graph is split
// into merge-path units of `grain` rows + entries (as in the single-graph
// sweep, Section IV-C's equal-edge blocks), the units of all graphs are
// numbered consecutively, and persistent warps take them from one counter, so
// large and small graphs share the GPU in a single launch.  The walk of a unit
// is the single-graph walk (walk.cuh) on a view of its graph.
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>
#include <cuda_runtime.h>

#include "internal.h"
#include "skipper.h"
#include "walk.cuh"
#include "checkwalk.cuh"

using namespace skp;

namespace skp {
namespace {

struct MultiParams {
  uint64_t num_graphs;
  const mm_graph_desc* desc;  // [G]
  const uint64_t* ubase;      // [G+1] first unit of each graph
  const uint64_t* vbase;      // [G+1] first vertex of each graph (for the init pass)
  const uint64_t* sbase;      // [G+1] first packed state word of each graph
  uint32_t* state_pool;       // packed state words of all graphs (2- or 8-bit layouts)
  int64_t* part;              // (row, entry) per unit
  uint32_t* gid;              // graph of each unit
  uint64_t units;
  uint64_t grain;
  unsigned long long* work;
  uint32_t* err;
  uint32_t* host_err;         // as SweepParams::host_err
  uint64_t spin_limit;
  uint32_t disperse;          // units handed out in dispersed runs
  unsigned long long* counters;  // checker: kCkCount per graph, then the long rows' count
};

// last g with base[g] <= x, base[0] = 0, base ascending, g < G
__device__ __forceinline__ uint64_t find_graph(const uint64_t* base, uint64_t G, uint64_t x) {
  uint64_t lo = 0, hi = G;
  while (hi - lo > 1) {
    const uint64_t mid = (lo + hi) >> 1;
    if (__ldg(base + mid) <= x) lo = mid; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ SweepParams view(const MultiParams& M, uint64_t g, bool word) {
  const mm_graph_desc d = M.desc[g];
  SweepParams P{};
  P.n = d.n;
  P.nnz = d.nnz;
  P.offsets = d.offsets;
  P.nbrs = d.nbrs;
  P.mate = d.mate;
  P.state = word ? d.mate : M.state_pool + M.sbase[g];
  P.err = M.err;
  P.host_err = M.host_err;
  P.spin_limit = M.spin_limit;
  return P;
}

template <bool kWord>
__global__ void multi_prepare_kernel(MultiParams M) {
  const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t nthreads = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t G = M.num_graphs;
  // every vertex ACC (Algorithm 1 lines 3-4), mate unmatched: a warp fills runs
  // of kFillRun vertices, graph by graph, one search a run
  constexpr uint64_t kFillRun = 1024;
  const uint64_t V = M.vbase[G];
  const unsigned lane = threadIdx.x & 31u;
  for (uint64_t v0 = (tid >> 5) * kFillRun; v0 < V; v0 += (nthreads >> 5) * kFillRun) {
    const uint64_t v1 = v0 + kFillRun < V ? v0 + kFillRun : V;
    uint64_t g = warp_last_at_or_below(M.vbase, G, v0, lane);
    for (uint64_t v = v0; v < v1; ++g) {
      const uint64_t first = __ldg(M.vbase + g), last = __ldg(M.vbase + g + 1);
      const uint64_t stop = last < v1 ? last : v1;
      uint32_t* const mate = M.desc[g].mate;
      for (uint64_t i = v + lane; i < stop; i += 32) mate[i - first] = kNone;  // = the word state ACC
      v = stop;
    }
  }
  if (!kWord)
    for (uint64_t i = tid; i < (M.sbase[G] + 3) / 4; i += nthreads)  // the pool holds whole quads
      reinterpret_cast<uint4*>(M.state_pool)[i] = make_uint4(0u, 0u, 0u, 0u);
  // merge-path units of every graph
  for (uint64_t u = tid; u < M.units; u += nthreads) {
    const uint64_t g = find_graph(M.ubase, G, u);
    const mm_graph_desc d = M.desc[g];
    const int64_t total = (int64_t)(d.n + d.nnz);
    int64_t diag = (int64_t)((u - M.ubase[g]) * M.grain);
    if (diag > total) diag = total;
    const int64_t rows = merge_path_rows(d.offsets, (int64_t)d.n, (int64_t)d.nnz, diag);
    M.part[2 * u] = rows;
    M.part[2 * u + 1] = diag - rows;
    M.gid[u] = (uint32_t)g;
  }
  if (tid == 0) {
    *M.work = 0ull;
    *M.err = 0u;
  }
}

template <class S, bool kWord, bool kSel = false, bool kLean = false>
__global__ void __launch_bounds__(512, kLean ? 4 : 3) multi_sweep_kernel(MultiParams M) {
  const unsigned lane = threadIdx.x & 31u;
  const uint64_t pol = policy_evict_first();
  if (lane == 0) *warp_started() = 0u;
  const UnitOrder order(M.units, M.disperse != 0, (uint64_t)gridDim.x * (blockDim.x >> 5));
  for (;;) {
    const uint32_t c = take_unit(M.work, 0, lane);
    if (c >= order.total) return;
    const uint64_t w = order.unit(c);
    if (w >= M.units) continue;
    const uint32_t g = M.gid[w];
    const SweepParams P = view(M, g, kWord);
    const int64_t row0 = M.part[2 * w];
    const int64_t e_begin = M.part[2 * w + 1];
    const int64_t e_end = (w + 1 < M.units && M.gid[w + 1] == g) ? M.part[2 * w + 3] : (int64_t)P.nnz;
    if (e_begin < e_end) sweep_unit<S, false, false, kSel>(S(P), P, row0, e_begin, e_end, lane, pol);
    if ((c & 15) == 0) {
      uint32_t e = 0;
      if (lane == 0) e = ld_relaxed(M.err);
      if (__shfl_sync(kFull, e, 0) & kErrTimeout) return;
    }
  }
}

template <class S, bool kWord>
__global__ void multi_serial_kernel(MultiParams M) {
  const uint64_t g = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // one warp a graph
  if (g >= M.num_graphs) return;
  const SweepParams P = view(M, g, kWord);
  serial_graph<S>(P, threadIdx.x & 31u);
}

__device__ __forceinline__ void group_add(unsigned long long* c, unsigned peers, uint32_t v) {
  const uint32_t s = __reduce_add_sync(peers, v);
  if ((int)(threadIdx.x & 31) == __ffs(peers) - 1 && s) atomicAdd(c, (unsigned long long)s);
}

// The exact checker (checkwalk.cuh) over every vertex of every graph, one set
// of counters a graph.  A warp takes runs of kCheckRun * 32 consecutive
// vertices of the whole batch: one search finds a run's graph, and its counts go
// to the graph's counters when the warp leaves it, not vertex by vertex.
constexpr uint64_t kCheckRun = 4;  // 8: 195 us for 171 graphs of up to 1e6 edges; 4: 165

__device__ __forceinline__ CheckView multi_check_view(const MultiParams& M, uint64_t g) {
  const mm_graph_desc* d = M.desc + g;
  return CheckView{d->offsets, d->nbrs, d->mate, d->n, d->nnz};
}

__global__ void __launch_bounds__(256, kCheckBlocks) multi_check_kernel(MultiParams M, LongRows queue) {
  const unsigned lane = threadIdx.x & 31u;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint64_t G = M.num_graphs, N = M.vbase[G];
  init_counts(lane);
  uint64_t cur = 0;  // the graph of the warp's counts
  for (uint64_t w0 = warp * 32 * kCheckRun; w0 < N; w0 += nwarps * 32 * kCheckRun) {
    uint64_t g = warp_last_at_or_below(M.vbase, G, w0, lane);
    for (uint64_t v0 = w0; v0 < w0 + 32 * kCheckRun && v0 < N; v0 += 32) {
      const uint64_t i = v0 + lane;
      const bool in = i < N;
      while (in && i >= __ldg(M.vbase + g + 1)) ++g;
      const uint32_t v = (uint32_t)(i - __ldg(M.vbase + g));
      const CheckView V = multi_check_view(M, g);
      const Visit a = check_group<false>(V, in, v, load_vertex(V, in, v), (uint32_t)g, lane, queue);
      const uint64_t g0 = __shfl_sync(kFull, g, 0);
      const unsigned active = __ballot_sync(kFull, in);
      if (__all_sync(kFull, !in || g == g0)) {
        if (g0 != cur) flush_counts(M.counters + cur * kCkCount, lane);
        cur = g0;
        const unsigned matched = __ballot_sync(kFull, a.bits & kVxMatched), pairs = __ballot_sync(kFull, a.bits & kVxPair);
        if (lane == 0) {
          warp_counts()[kCkMatched] += __popc(matched);
          warp_counts()[kCkPairs] += __popc(pairs);
        }
        add_faults(a, v, lane);
      } else if (in) {  // the group spans graphs: each lane counts for its own
        unsigned long long* c = M.counters + g * kCkCount;
        const unsigned peers = __match_any_sync(active, g);
        group_add(c + kCkMatched, peers, a.bits & kVxMatched ? 1u : 0u);
        group_add(c + kCkPairs, peers, a.bits & kVxPair ? 1u : 0u);
        if (a.bits & kVxRange) atomicAdd(c + kCkRange, 1ull);
        if (a.bits & kVxAsym) atomicAdd(c + kCkAsym, 1ull);
        if (a.bits & kVxNonedge) atomicAdd(c + kCkNonedge, a.bits & kVxBothEnds ? 2ull : 1ull);
        if (a.bits & kVxBad) atomicMax(c + kCkFirstBad, ~(unsigned long long)v);
        add_nonzero(c + kCkUncovered, a.uncovered);
        if (~a.first_unc) atomicMax(c + kCkFirstUncovered, ~a.first_unc);
      }
      g = __shfl_sync(kFull, g, 0);
    }
  }
  flush_counts(M.counters + cur * kCkCount, lane);
}

__global__ void multi_check_long_kernel(MultiParams M, LongRows queue) {
  const unsigned long long pieces = queue.size();
  init_counts(threadIdx.x & 31u);
  uint64_t cur = 0;  // the graph of the counts
  for (unsigned long long i = blockIdx.x; i < pieces; i += gridDim.x) {
    const ulonglong2 item = queue.items[i];
    const uint64_t g = item.x >> 32;
    if (g != cur) flush_counts(M.counters + cur * kCkCount, threadIdx.x & 31u);
    cur = g;
    check_piece(multi_check_view(M, g), (uint32_t)item.x, (int64_t)item.y, threadIdx.x & 31u);
  }
  flush_counts(M.counters + cur * kCkCount, threadIdx.x & 31u);
}

// Grow a device buffer to at least `want` elements, ordered on the call's
// stream (cudaFreeAsync / cudaMallocAsync), so growing never waits for the
// whole device; capacity doubles so growth is rare.
template <class T>
cudaError_t grow(T** p, uint64_t* cap, uint64_t want, cudaStream_t s) {
  if (*p && *cap >= want) return cudaSuccess;
  uint64_t n = *cap ? *cap : 64;
  while (n < want) n *= 2;
  if (*p) {
    cudaError_t e = cudaFreeAsync(*p, s);
    if (e != cudaSuccess) return e;
  }
  *p = nullptr;
  *cap = 0;
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(p), n * sizeof(T), s);
  if (e == cudaSuccess) *cap = n;
  return e;
}

thread_local char g_msg[512] = "";

mm_status mfail(mm_status st, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_msg, sizeof g_msg, fmt, ap);
  va_end(ap);
  set_error_message("%s", g_msg);
  return st;
}

#define MTRY(expr)                                                                             \
  do {                                                                                         \
    cudaError_t e_ = (expr);                                                                   \
    if (e_ != cudaSuccess)                                                                     \
      return mfail(e_ == cudaErrorMemoryAllocation ? MM_ERR_OOM : MM_ERR_CUDA, "%s: %s", #expr, \
                   cudaGetErrorString(e_));                                                    \
  } while (0)

}  // namespace
}  // namespace skp

// Device tables of one call ([desc G | ubase G+1 | vbase G+1 | sbase G+1]),
// their pinned staging copy and the partition built on them.  The sweep and
// the checker have one set each, so a checker enqueued right behind a sweep
// never waits for the sweep's staging copy.
struct TableSet {
  unsigned char* tables = nullptr;
  uint64_t tables_cap = 0;
  unsigned char* staging = nullptr;    // pinned host copy of the tables
  uint64_t staging_cap = 0;
  cudaEvent_t staging_free = nullptr;  // the last copy out of `staging` has finished
  bool staging_pending = false;
  int64_t* part = nullptr;
  uint64_t part_cap = 0;
  uint32_t* gid = nullptr;
  uint64_t gid_cap = 0;
};

struct mm_multi {
  int device = 0;
  int num_sms = 0;
  int l2_bytes = 0;
  TableSet sweep, check;
  uint32_t* pool = nullptr;
  uint64_t pool_cap = 0;
  unsigned long long* counters = nullptr;
  uint64_t counters_cap = 0;
  unsigned long long* ctrl = nullptr;  // [0] work, [1] err
  uint32_t* h_err = nullptr;           // pinned
  unsigned long long* h_counters = nullptr;
  uint64_t h_counters_cap = 0;
  uint64_t checked_graphs = 0;         // graphs of the last enqueued check
};

namespace skp {
namespace {

struct Layout {
  uint64_t units = 0;
  uint64_t bytes = 0;
  uint64_t off_ubase = 0, off_vbase = 0, off_sbase = 0;
  uint64_t total_vertices = 0, total_words = 0;
  uint64_t long_rows = 0;              // pieces that long rows can have
};

mm_status stage_tables(TableSet* m, uint64_t G, const mm_graph_desc* h, uint64_t grain, int bits,
                       cudaStream_t s, Layout* L) {
  L->off_ubase = G * sizeof(mm_graph_desc);
  L->off_vbase = L->off_ubase + (G + 1) * 8;
  L->off_sbase = L->off_vbase + (G + 1) * 8;
  L->bytes = L->off_sbase + (G + 1) * 8;
  if (m->staging_pending) {  // the previous call may still be copying out of the staging buffer
    MTRY(cudaEventSynchronize(m->staging_free));
    m->staging_pending = false;
  }
  if (m->staging_cap < L->bytes) {
    uint64_t cap = m->staging_cap ? m->staging_cap : 4096;   // doubling from the old size
    while (cap < L->bytes) cap *= 2;
    if (m->staging) cudaFreeHost(m->staging);
    m->staging = nullptr;
    m->staging_cap = 0;
    MTRY(cudaMallocHost(&m->staging, cap));
    m->staging_cap = cap;
  }
  MTRY(grow(&m->tables, &m->tables_cap, L->bytes, s));
  memcpy(m->staging, h, G * sizeof(mm_graph_desc));
  uint64_t* ub = reinterpret_cast<uint64_t*>(m->staging + L->off_ubase);
  uint64_t* vb = reinterpret_cast<uint64_t*>(m->staging + L->off_vbase);
  uint64_t* sb = reinterpret_cast<uint64_t*>(m->staging + L->off_sbase);
  ub[0] = vb[0] = sb[0] = 0;
  for (uint64_t g = 0; g < G; ++g) {
    ub[g + 1] = ub[g] + (h[g].n + h[g].nnz + grain - 1) / grain;
    vb[g + 1] = vb[g] + h[g].n;
    L->long_rows += long_row_cap(h[g].nnz, false);
    sb[g + 1] = sb[g] + (bits == 32 ? 0 : packed_words(h[g].n, bits) + 1);
  }
  L->units = ub[G];
  L->total_vertices = vb[G];
  L->total_words = sb[G];
  MTRY(cudaMemcpyAsync(m->tables, m->staging, L->bytes, cudaMemcpyHostToDevice, s));
  MTRY(cudaEventRecord(m->staging_free, s));
  m->staging_pending = true;
  return MM_OK;
}

MultiParams params(mm_multi* m, const TableSet& t, uint64_t G, const Layout& L, uint64_t grain,
                   uint64_t spin) {
  MultiParams M{};
  M.num_graphs = G;
  M.desc = reinterpret_cast<const mm_graph_desc*>(t.tables);
  M.ubase = reinterpret_cast<const uint64_t*>(t.tables + L.off_ubase);
  M.vbase = reinterpret_cast<const uint64_t*>(t.tables + L.off_vbase);
  M.sbase = reinterpret_cast<const uint64_t*>(t.tables + L.off_sbase);
  M.state_pool = m->pool;
  M.part = t.part;
  M.gid = t.gid;
  M.units = L.units;
  M.grain = grain;
  M.work = m->ctrl;
  M.err = reinterpret_cast<uint32_t*>(m->ctrl + 1);
  M.spin_limit = spin;
  M.counters = m->counters;
  return M;
}

mm_status check_descs(uint64_t G, const mm_graph_desc* h) {
  for (uint64_t g = 0; g < G; ++g) {
    const mm_graph_desc& d = h[g];
    if (d.n > MM_MAX_VERTICES) return mfail(MM_ERR_ARG, "graph %llu: n too large", (unsigned long long)g);
    if (!d.offsets || (d.nnz && !d.nbrs) || (d.n && !d.mate))
      return mfail(MM_ERR_ARG, "graph %llu: null array", (unsigned long long)g);
    if (d.nnz && (reinterpret_cast<uintptr_t>(d.nbrs) & 15u))
      return mfail(MM_ERR_ARG, "graph %llu: nbrs must be 16-byte aligned", (unsigned long long)g);
  }
  return MM_OK;
}

}  // namespace
}  // namespace skp

extern "C" {

mm_status mm_multi_create(mm_multi** out) {
  if (!out) return mfail(MM_ERR_ARG, "null out");
  *out = nullptr;
  mm_multi* m = new (std::nothrow) mm_multi();
  if (!m) return mfail(MM_ERR_OOM, "host allocation failed");
  cudaError_t e = cudaGetDevice(&m->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&m->num_sms, cudaDevAttrMultiProcessorCount, m->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&m->l2_bytes, cudaDevAttrL2CacheSize, m->device);
  if (e == cudaSuccess) e = cudaMalloc(&m->ctrl, 16 * sizeof(unsigned long long));
  if (e == cudaSuccess) e = cudaMallocHost(&m->h_err, 64);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&m->sweep.staging_free, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&m->check.staging_free, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    mm_multi_destroy(m);
    return mfail(MM_ERR_CUDA, "mm_multi_create: %s", cudaGetErrorString(e));
  }
  *m->h_err = 0;
  *out = m;
  return MM_OK;
}

mm_status mm_skipper_multi(mm_multi* m, uint64_t num_graphs, const mm_graph_desc* h_descs,
                           const mm_options* o, void* cuda_stream) {
  if (!m) return mfail(MM_ERR_ARG, "null handle");
  if (!num_graphs) return MM_OK;
  if (!h_descs) return mfail(MM_ERR_ARG, "null descriptors");
  mm_status st = check_descs(num_graphs, h_descs);
  if (st != MM_OK) return st;
  mm_options d;
  mm_default_options(&d);
  if (!o) o = &d;
  const uint32_t bits = o->status_bits ? o->status_bits : 8u;
  if (bits != 2 && bits != 8 && bits != 32) return mfail(MM_ERR_ARG, "status_bits must be 2, 8 or 32");
  const bool word = bits == 32;
  if (o->grain % 128 || o->grain > (1u << 24)) return mfail(MM_ERR_ARG, "bad grain");
  if (o->unit_order > MM_ORDER_DISPERSED) return mfail(MM_ERR_ARG, "unit_order must be 0, 1 or 2");
  const int block = o->block_threads ? (int)o->block_threads : 512;
  if (block < 32 || block > 512 || block % 32) return mfail(MM_ERR_ARG, "bad block_threads");
  if (o->id_loads > MM_ID_LOADS_SELECTIVE) return mfail(MM_ERR_ARG, "id_loads must be 0, 1 or 2");
  const bool sel = o->id_loads == MM_ID_LOADS_SELECTIVE;   // automatic: eager
  if (o->timing || o->use_graph || o->poison_vertex || o->l2_persist)
    return mfail(MM_ERR_UNSUPPORTED, "timing, use_graph, poison_vertex and l2_persist are not "
                                     "available in multi-graph calls");
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  // work split as for one graph of all their rows and entries
  uint64_t rows = 0, items = 0;
  for (uint64_t g = 0; g < num_graphs; ++g) {
    rows += h_descs[g].n;
    items += h_descs[g].n + h_descs[g].nnz;
  }
  const uint64_t state_bytes = word ? 4 * rows : rows * bits / 8;
  const bool fits = 2 * state_bytes <= (uint64_t)m->l2_bytes;
  const bool disperse = o->unit_order == MM_ORDER_DISPERSED || (o->unit_order == MM_ORDER_AUTO && fits);
  const uint64_t grain = o->grain ? o->grain : choose_grain(rows, items, (uint64_t)m->num_sms * (fits ? 64 : 48), disperse, word);
  Layout L;
  if ((st = stage_tables(&m->sweep, num_graphs, h_descs, grain, (int)bits, s, &L)) != MM_OK) return st;
  MTRY(grow(&m->sweep.part, &m->sweep.part_cap, 2 * (L.units + 1), s));
  MTRY(grow(&m->sweep.gid, &m->sweep.gid_cap, L.units + 1, s));
  if (!word) MTRY(grow(&m->pool, &m->pool_cap, L.total_words + 4, s));
  MultiParams M = params(m, m->sweep, num_graphs, L, grain, o->spin_limit ? o->spin_limit : (1ull << 20));
  M.disperse = disperse ? 1u : 0u;
  m->h_err[1] = 0;  // a call that waits has its kernels report here
  M.host_err = o->nosync ? nullptr : m->h_err + 1;

  const int prep_grid = m->num_sms * 8;
  if (word) multi_prepare_kernel<true><<<prep_grid, 256, 0, s>>>(M);
  else multi_prepare_kernel<false><<<prep_grid, 256, 0, s>>>(M);
  MTRY(cudaGetLastError());
  if (o->serial) {
    const unsigned grid = (unsigned)((num_graphs + kSerialGraphsPerBlock - 1) / kSerialGraphsPerBlock);
    constexpr int threads = 32 * (int)kSerialGraphsPerBlock;
    if (bits == 32) multi_serial_kernel<WordState, true><<<grid, threads, 0, s>>>(M);
    else if (bits == 2) multi_serial_kernel<TwoBitState, false><<<grid, threads, 0, s>>>(M);
    else multi_serial_kernel<ByteState, false><<<grid, threads, 0, s>>>(M);
  } else if (L.units) {
    // 64 warps an SM (32 registers) where the states stay in L2, as in the
    // single-graph sweep; selective loads wait on the host link all the same
    const bool lean = !sel && (o->blocks_per_sm ? o->blocks_per_sm > 3 : fits);
    void (*kernel)(MultiParams) = nullptr;
#define SKP_MULTI(S, W)                                                                    \
  (sel ? multi_sweep_kernel<S, W, true> : lean ? multi_sweep_kernel<S, W, false, true>     \
                                               : multi_sweep_kernel<S, W>)
    kernel = bits == 32 ? SKP_MULTI(WordState, true) : bits == 2 ? SKP_MULTI(TwoBitState, false) : SKP_MULTI(ByteState, false);
#undef SKP_MULTI
    int per_sm = (int)o->blocks_per_sm;
    if (per_sm <= 0) {
      const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, 0);
      if (e != cudaSuccess || per_sm < 1) per_sm = 1;
    }
    kernel<<<m->num_sms * per_sm, block, 0, s>>>(M);
  }
  MTRY(cudaGetLastError());
  if (o->nosync) {
    MTRY(cudaMemcpyAsync(m->h_err, M.err, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    return MM_OK;
  }
  MTRY(cudaStreamSynchronize(s));
  m->h_err[0] = *static_cast<volatile uint32_t*>(m->h_err + 1);
  return mm_multi_sync(m, cuda_stream);
}

mm_status mm_multi_sync(mm_multi* m, void* cuda_stream) {
  if (!m) return mfail(MM_ERR_ARG, "null handle");
  MTRY(cudaStreamSynchronize(static_cast<cudaStream_t>(cuda_stream)));
  const uint32_t e = *static_cast<volatile uint32_t*>(m->h_err);
  if (e & kErrTimeout) return mfail(MM_ERR_TIMEOUT, "a wait on a reserved vertex ran past spin_limit");
  if (e & kErrBadId) return mfail(MM_ERR_BAD_GRAPH, "a neighbour id >= n was met");
  return MM_OK;
}

mm_status mm_validate_multi_async(mm_multi* m, uint64_t num_graphs, const mm_graph_desc* h_descs,
                                  void* cuda_stream) {
  if (!m) return mfail(MM_ERR_ARG, "null handle");
  m->checked_graphs = 0;
  if (!num_graphs) return MM_OK;
  if (!h_descs) return mfail(MM_ERR_ARG, "null descriptors");
  mm_status st = check_descs(num_graphs, h_descs);
  if (st != MM_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  Layout L;
  if ((st = stage_tables(&m->check, num_graphs, h_descs, (uint64_t)kPiece, 32, s, &L)) != MM_OK) return st;
  const uint64_t words = num_graphs * kCkCount;
  MTRY(grow(&m->counters, &m->counters_cap, words + 1, s));
  MTRY(grow(&m->check.part, &m->check.part_cap, 2 * L.long_rows + 2, s));
  if (m->h_counters_cap < words) {
    // the previous check's counters may still be on their way into the old buffer
    MTRY(cudaStreamSynchronize(s));
    if (m->h_counters) cudaFreeHost(m->h_counters);
    m->h_counters = nullptr;
    uint64_t cap = m->h_counters_cap ? m->h_counters_cap : 64 * kCkCount;
    while (cap < words) cap *= 2;
    m->h_counters_cap = 0;
    MTRY(cudaMallocHost(&m->h_counters, cap * sizeof(unsigned long long)));
    m->h_counters_cap = cap;
  }
  const MultiParams M = params(m, m->check, num_graphs, L, (uint64_t)kPiece, 1);
  const LongRows queue{m->counters + words, reinterpret_cast<ulonglong2*>(m->check.part), L.long_rows};
  MTRY(cudaMemsetAsync(m->counters, 0, (words + 1) * sizeof(unsigned long long), s));
  if (L.total_vertices) {
    multi_check_kernel<<<check_grid(L.total_vertices, m->num_sms), 256, 0, s>>>(M, queue);
    if (L.long_rows) multi_check_long_kernel<<<m->num_sms * 4, 256, 0, s>>>(M, queue);
  }
  MTRY(cudaGetLastError());
  MTRY(cudaMemcpyAsync(m->h_counters, m->counters, words * sizeof(unsigned long long),
                       cudaMemcpyDeviceToHost, s));
  m->checked_graphs = num_graphs;
  return MM_OK;
}

mm_status mm_multi_verdicts(mm_multi* m, uint64_t num_graphs, mm_verdict* h_out) {
  if (!m || (num_graphs && !h_out)) return mfail(MM_ERR_ARG, "null argument");
  if (num_graphs != m->checked_graphs)
    return mfail(MM_ERR_ARG, "%llu verdicts asked, the last check covered %llu graphs",
                 (unsigned long long)num_graphs, (unsigned long long)m->checked_graphs);
  for (uint64_t g = 0; g < num_graphs; ++g) {
    const unsigned long long* c = m->h_counters + g * kCkCount;
    mm_verdict v{};
    v.n_matched = c[kCkMatched];
    v.n_pairs = c[kCkPairs];
    v.n_bad_range = c[kCkRange];
    v.n_asym = c[kCkAsym];
    v.n_nonedge = c[kCkNonedge];
    v.n_uncovered = c[kCkUncovered];
    v.n_pairs_bad = 0;
    v.first_bad_vertex = ~c[kCkFirstBad];
    v.first_uncovered = ~c[kCkFirstUncovered];
    if (v.n_bad_range) v.flags |= MM_V_RANGE;
    if (v.n_asym) v.flags |= MM_V_ASYM;
    if (v.n_nonedge) v.flags |= MM_V_NONEDGE;
    if (v.n_uncovered) v.flags |= MM_V_UNCOVERED;
    h_out[g] = v;
  }
  return MM_OK;
}

mm_status mm_validate_multi(mm_multi* m, uint64_t num_graphs, const mm_graph_desc* h_descs,
                            mm_verdict* h_out, void* cuda_stream) {
  if (!m || (num_graphs && !h_out)) return mfail(MM_ERR_ARG, "null argument");
  mm_status st = mm_validate_multi_async(m, num_graphs, h_descs, cuda_stream);
  if (st != MM_OK) return st;
  MTRY(cudaStreamSynchronize(static_cast<cudaStream_t>(cuda_stream)));
  return mm_multi_verdicts(m, num_graphs, h_out);
}

mm_status mm_multi_destroy(mm_multi* m) {
  if (!m) return MM_OK;
  for (TableSet* t : {&m->sweep, &m->check}) {
    if (t->staging_pending && t->staging_free) cudaEventSynchronize(t->staging_free);
    if (t->staging_free) cudaEventDestroy(t->staging_free);
    if (t->tables) cudaFree(t->tables);
    if (t->staging) cudaFreeHost(t->staging);
    if (t->part) cudaFree(t->part);
    if (t->gid) cudaFree(t->gid);
  }
  if (m->pool) cudaFree(m->pool);
  if (m->counters) cudaFree(m->counters);
  if (m->ctrl) cudaFree(m->ctrl);
  if (m->h_err) cudaFreeHost(m->h_err);
  if (m->h_counters) cudaFreeHost(m->h_counters);
  delete m;
  return MM_OK;
}

}  // extern "C"
