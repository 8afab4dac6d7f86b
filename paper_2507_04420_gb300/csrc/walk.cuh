// walk.cuh -- the per-warp walk of Skipper's single pass (Algorithm 1) over
// one merge-path work unit, shared by the single-graph sweep (sweep.cu) and
// the multi-graph sweep (multi.cu).  Every function here takes the graph it
// works on through a SweepParams view, so one unit of any graph is walked the
// same way.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "internal.h"
#include "state.cuh"

namespace skp {
namespace {

// a[j] for a run-time j without local-memory indexing
template <class T>
__device__ __forceinline__ T pick4(const T (&a)[4], int j) {
  T r = a[0];
#pragma unroll
  for (int i = 1; i < 4; ++i) r = j == i ? a[i] : r;
  return r;
}

// Merge-path split of diagonal d over the row ends offsets[1..n] and the entry
// indices 0..nnz-1 (a row end equal to an entry index is taken first): returns
// the number of rows finished before the split; entry index = d - rows.
__device__ __forceinline__ int64_t merge_path_rows(const int64_t* offsets, int64_t n, int64_t nnz,
                                                   int64_t d) {
  int64_t lo = d - nnz > 0 ? d - nnz : 0;
  int64_t hi = d < n ? d : n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (offsets[mid + 1] <= d - mid - 1)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// number of lanes k whose ascending value rel_k is <= p (32-bit); the caller
// guarantees rel_31 > p for the lanes whose answer it uses.
__device__ __forceinline__ int count_le(int rel, int p) {
  int c = 0;
#pragma unroll
  for (int step = 16; step >= 1; step >>= 1) {
    const int v = __shfl_sync(kFull, rel, c + step - 1);
    if (v <= p) c += step;
  }
  return c;
}

// Four neighbour ids from entry e0 on (one aligned 128-bit load when all four
// exist, else the ones below nnz).
__device__ __forceinline__ void load_quad(const SweepParams& P, int64_t e0, uint64_t pol,
                                          uint32_t (&y)[4]) {
  if (e0 + 4 <= (int64_t)P.nnz) {
    const uint4 q = ld_stream_v4(P.nbrs + e0, pol);
    y[0] = q.x; y[1] = q.y; y[2] = q.z; y[3] = q.w;
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (e0 + j < (int64_t)P.nnz) y[j] = ld_stream(P.nbrs + e0 + j, pol);
  }
}

// Shared-memory tile of one 32-row window (kTile instances, opt-in), filled
// by one bulk copy (TMA, cp.async.bulk with an mbarrier) while the warp still
// works on the window before it: the window's row ends (34 int64 from an even
// index, 272 bytes) and the state words of its rows (12 words from a multiple
// of 4, 48 bytes).  Both copies start 16-byte aligned (the host enables the
// instances only for 16-byte aligned arrays in device memory) and stay inside
// their arrays (n + 1 row ends, ceil(n / per word) state words); a window for
// which they would not is loaded directly.  The state words are a snapshot one
// window old: a row matched since then reads as unmatched, which costs an
// extra filter read, never a wrong result (MCHD is absorbing, and every
// transition is a CAS on the current word).  Every wait on the barrier is
// bounded.
struct alignas(16) WindowTile {
  int64_t ends[36];
  uint32_t st[16];
  unsigned long long bar;
  unsigned long long pad;
};
constexpr uint32_t kTileEnds = 34, kTileWords = 12;
constexpr uint32_t kTileBytes = kTileEnds * 8 + kTileWords * 4;
__shared__ WindowTile g_window_tiles[16];       // one per warp of a block of <= 512 threads

// the warp's tile barrier (one arrival per copy); once per warp before its first unit
__device__ __forceinline__ void init_window_tile(unsigned lane) {
  if (lane == 0) {
    mbar_init(&g_window_tiles[threadIdx.x >> 5].bar, 1);
    fence_mbar_init();
  }
  __syncwarp();
}

// One work unit: entries [e_begin, e_end), the first of which lies in row >= row0.
//
// The warp keeps a window of 32 consecutive rows: lane k holds the end offset
// of row wbase+k and the word holding that row vertex's state, both loaded in
// one coalesced step, and `mchd` has bit k set when row wbase+k is known to be
// matched.  Matched rows are jumped over with bit arithmetic, so a matched
// source costs no load of its own (Skipper leaves the rest of a matched row;
// SGMM does the same in CSR order, Section II-B).  The unmatched entries are
// read in chunks of up to 128 (one aligned 128-bit load per lane); the state
// of the row at the head of each chunk is re-read alongside, so a long row
// matched by another warp is left after at most one more chunk.
//
// kMesh (graphs of few entries a row, most of them lattices, meshes and road
// networks): where ids have locality the rows of a window name each other, as x
// names x - 1 all along it; tried at once, each holds what the next one waits
// for.  So a chunk that names rows of its own window is visited twice, the odd
// rows waiting for the second visit.
//
// kTile: windows come from the warp's shared-memory tile (WindowTile above).
//
// kSel (selective id loads): a lane loads its quad only after the row search,
// and only when the quad holds an entry of a row not known matched.  The
// eager walk issues every load of the chunk first, so that its latency
// overlaps the search; the selective walk moves fewer bytes (on R-MAT, well
// under half the quads of a chunk are in rows not known matched), which pays
// where the bytes cross the host link.
template <class S, bool kStats = false, bool kSym = false, bool kSel = false, bool kTile = false, bool kMesh = false>
__device__ __forceinline__ void sweep_unit(const S& s, const SweepParams& P, int64_t row0,
                                           const int64_t e_begin, const int64_t e_end,
                                           const unsigned lane, const uint64_t pol_stream,
                                           uint32_t* phase = nullptr) {
  const uint32_t n32 = (uint32_t)P.n;
  // Positions are entry indices relative to e_begin (a unit holds at most
  // 2^24 items, so 32 bits suffice).  Row ends are clamped to [0, ue]: a row
  // that ends before the unit reads as ending at 0, one that ends after it as
  // ending at ue, which changes no comparison the walk makes.
  const int ue = (int)(e_end - e_begin);
  const int align = (int)(e_begin & 3);     // base of a chunk: ((pos + align) & ~3) - align
  auto rel_end = [&](int64_t end) -> int {
    const int64_t d = end - e_begin;
    return d < 0 ? 0 : (d > (int64_t)ue ? ue : (int)d);
  };
  int64_t wbase = row0;
  int my_end;
  uint32_t my_st;
  unsigned mchd;
  int pos = 0;
  bool again = false;                           // second visit to a chunk (kMesh)
  bool pending = false;                         // a copy of the next window's tile is in flight
  auto tile = [&]() { return &g_window_tiles[threadIdx.x >> 5]; };
  auto t_s = [&](int64_t w) { return (w + 1) & ~(int64_t)1; };
  auto t_sw = [&](int64_t w) { return (w / (int64_t)S::kPerWord) & ~(int64_t)3; };
  auto issue_next = [&](int64_t w) {
    if (!kTile) return;
    const int64_t sidx = t_s(w), sw = t_sw(w);
    // both copies stay inside their arrays: n + 1 row offsets, ceil(n / per word) state words
    if (sidx + (int64_t)kTileEnds > (int64_t)P.n + 1 ||
        sw + (int64_t)kTileWords > (int64_t)((P.n + S::kPerWord - 1) / S::kPerWord))
      return;
    if (lane == 0) {
      fence_proxy_async_smem();   // this warp's reads of the tile come before the copy's writes
      mbar_expect_tx(&tile()->bar, kTileBytes);
      bulk_to_smem(tile()->ends, P.offsets + sidx, kTileEnds * 8, &tile()->bar);
      bulk_to_smem(tile()->st, P.state + sw, kTileWords * 4, &tile()->bar);
    }
    pending = true;
  };
  // bounded wait for the copy in flight; false when it ran past the limit
  auto wait_tile = [&]() -> bool {
    for (uint32_t i = 0; i < (1u << 22); ++i)
      if (mbar_try_wait(&tile()->bar, *phase)) {
        *phase ^= 1u;
        pending = false;
        return true;
      }
    return false;
  };
  {
    const int64_t r = wbase + lane;
    const bool in = r < (int64_t)P.n;
    my_end = in ? rel_end(__ldg(P.offsets + r + 1)) : ue;
    my_st = in ? s.peek((uint32_t)r) : 0u;
    mchd = __ballot_sync(kFull, !in || S::matched(my_st, (uint32_t)r));  // rows past n hold no entries
    issue_next(wbase + 32);
  }
  while (pos < ue) {
    if (kMesh && again) {  // what the first visit left open
      if (wbase + lane < (int64_t)P.n) my_st = s.peek((uint32_t)wbase + lane);
      mchd |= __ballot_sync(kFull, S::matched(my_st, (uint32_t)wbase + lane));
    }
    // rows of the window with entries at or after pos that are not known matched
    const unsigned open = __ballot_sync(kFull, my_end > pos) & ~mchd;
    if (open == 0u) {  // the window is exhausted: continue after its last row
      const int win_end = __shfl_sync(kFull, my_end, 31);
      if (win_end >= ue) break;
      if (win_end > pos) pos = win_end;
      if (kMesh) again = false;
      wbase += 32;
      const int64_t r = wbase + lane;
      const bool in = r < (int64_t)P.n;
      bool from_tile = false;
      if (kTile && pending) {
        from_tile = wait_tile();
        if (!from_tile) {            // the copy did not land: stop, after a last bounded wait
          if (lane == 0) report(P.err, P.host_err, kErrTimeout);
          wait_tile();
          return;
        }
      }
      if (from_tile) {
        my_end = in ? rel_end(tile()->ends[wbase + 1 + lane - t_s(wbase)]) : ue;
        my_st = in ? tile()->st[(r / (int64_t)S::kPerWord) - t_sw(wbase)] : 0u;
        __syncwarp();
      } else {
        my_end = in ? rel_end(__ldg(P.offsets + r + 1)) : ue;
        my_st = in ? s.peek((uint32_t)r) : 0u;
      }
      mchd = __ballot_sync(kFull, !in || S::matched(my_st, (uint32_t)r));
      issue_next(wbase + 32);
      if (kStats && lane == 0) atomicAdd(P.stats + kStWindows, 1ull);
      continue;
    }
    const int k1 = __ffs(open) - 1;
    if (k1 > 0) {  // row k1 starts where row k1-1 ends
      const int st = __shfl_sync(kFull, my_end, k1 - 1);
      if (st > pos) pos = st;
    }
    if (pos >= ue) break;
    const int win_end = __shfl_sync(kFull, my_end, 31);
    const int base = ((pos + align) & ~3) - align;
    int cend = base + 128;
    if (cend > ue) cend = ue;
    if (cend > win_end) cend = win_end;
    // chunk-relative coordinates: entry base+p, p in [lo_r, hi_r)
    const int lo_r = pos - base;
    const int hi_r = cend - base;
    if (kStats && lane == 0) {
      atomicAdd(P.stats + kStChunks, 1ull);
      atomicAdd(P.stats + kStEntries, (unsigned long long)(hi_r - lo_r));
    }
    int rel = my_end - base;
    rel = rel < 0 ? -1 : (rel > 129 ? 129 : rel);

    // neighbour ids (one aligned 128-bit load per lane) and, in parallel, a
    // fresh read of the head row's state
    const int p0 = 4 * (int)lane;
    const int64_t e0 = e_begin + base + p0;
    uint32_t y[4] = {0u, 0u, 0u, 0u};
    if (!kSel && p0 < hi_r) load_quad(P, e0, pol_stream, y);
    const uint32_t wb32 = (uint32_t)wbase;
    const uint32_t x1 = wb32 + (uint32_t)k1;
    uint32_t head = 0;
    if (lane == 0) head = s.peek(x1);  // consumed after the row search, so both loads overlap it

    // row of each entry within the window
    int k[4];
    k[0] = count_le(rel, p0);
    k[3] = count_le(rel, p0 + 3);
    if (__any_sync(kFull, k[0] != k[3])) {
      k[1] = count_le(rel, p0 + 1);
      k[2] = count_le(rel, p0 + 2);
    } else {
      k[1] = k[0];
      k[2] = k[0];
    }
    head = __shfl_sync(kFull, head, 0);
    if (S::matched(head, x1)) mchd |= 1u << k1;
    if (lane == (unsigned)k1) my_st = head;
    uint32_t xs[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) xs[j] = wb32 + (uint32_t)k[j];
    if (kSel || kStats) {
      // does this lane's quad hold an entry of a row not known matched?
      bool open_quad = false;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int p = p0 + j;
        open_quad |= p >= lo_r && p < hi_r && !(mchd >> (k[j] & 31) & 1u);
      }
      if (kSel && open_quad) load_quad(P, e0, pol_stream, y);
      if (kStats) {
        const unsigned issued = __ballot_sync(kFull, p0 < hi_r);
        const unsigned wanted = __ballot_sync(kFull, open_quad);
        if (lane == 0) {
          atomicAdd(P.stats + kStIdLoads, (unsigned long long)__popc(issued));
          atomicAdd(P.stats + kStIdLoadsOpen, (unsigned long long)__popc(wanted));
        }
      }
    }

    // filter (the line-10 read): candidates have both endpoints unmatched.  A
    // row whose snapshot word reads MCHD has its bit in mchd (set when the
    // window or the head word was read), so the row test is the mask alone.
    // Loops are skipped (lines 6-7); on a symmetric CSR so is every (x, y) with
    // y < x, which row y holds as (y, x) (each edge tested once).
    bool want[4];
    bool bad = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int p = p0 + j;
      want[j] = p >= lo_r && p < hi_r && !(mchd >> (k[j] & 31) & 1u) &&
                (kSym ? y[j] > xs[j] : y[j] != xs[j]);
      bad |= want[j] && y[j] >= n32;
      want[j] = want[j] && y[j] < n32;
    }
    if (__any_sync(kFull, bad) && bad) report_bad_id(P.err, P.host_err);
    uint32_t ry[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (want[j]) ry[j] = s.peek(y[j]);
    uint32_t cand = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (want[j] && !S::matched(ry[j], y[j])) cand |= 1u << j;

    if (kMesh) {
      bool near = false;
#pragma unroll
      for (int j = 0; j < 4; ++j) near |= (cand >> j & 1u) && y[j] - wb32 < 32u;
      again = !again && __any_sync(kFull, near);
      if (again) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (k[j] & 1) cand &= ~(1u << j);
      }
    }

    // resolve candidates: per row, one lane at a time
    for (;;) {
      const bool have = cand != 0u;
      if (!__any_sync(kFull, have)) break;
      const int j = have ? __ffs(cand) - 1 : 0;
      const uint32_t key = have ? pick4(xs, j) : kNone;
      const uint32_t rxj = __shfl_sync(kFull, my_st, (key - wb32) & 31);
      const unsigned peers = __match_any_sync(kFull, key);
      const int leader = __ffs(peers) - 1;
      unsigned done = 0u;
      if (have && (int)lane == leader) {
        cand &= ~(1u << j);
        if (resolve_edge<S, kStats>(s, key, pick4(y, j), rxj, pick4(ry, j), P))
          done = 1u << (key - wb32);
      }
      done = __reduce_or_sync(kFull, done);  // rows that are now matched
      mchd |= done;
#pragma unroll
      for (int jj = 0; jj < 4; ++jj)
        if (done >> (k[jj] & 31) & 1u) cand &= ~(1u << jj);
    }
    if (!kMesh || !again) pos = cend;
  }
  if (kTile && pending && !wait_tile()) {   // the tile is reused by the next unit
    if (lane == 0) report(P.err, P.host_err, kErrTimeout);
    wait_tile();
  }
}

// Which vertices of one graph are matched, a bit each in shared memory: all the
// state that serial mode needs of a graph whose ids start at 0.  A chunk's states
// then take tens of nanoseconds instead of a round trip to L2: 4096 graphs of 100
// to 10,000 edges 844 -> 630 us a call, 64 of 1000 to 10,000 edges 612 -> 446.
constexpr uint32_t kSerialBits = 32768;  // vertices; 4 KB a warp leaves 14 blocks of 4 warps an SM
struct SerialBits {
  static constexpr bool kAlone = true;
  uint32_t* words;
  uint32_t* mate;
  __device__ __forceinline__ uint32_t raw(uint32_t v) const { return words[v >> 5] >> (v & 31u) & 1u; }
  __device__ static __forceinline__ bool matched(uint32_t raw, uint32_t) { return raw != 0u; }
  __device__ static __forceinline__ bool reserved(uint32_t, uint32_t) { return false; }
  __device__ __forceinline__ void match_alone(uint32_t u, uint32_t v) const {
    mate[u] = v;
    mate[v] = u;
    atomicOr(words + (u >> 5), 1u << (u & 31u));
    atomicOr(words + (v >> 5), 1u << (v & 31u));
  }
};

// Rows [r0, r1) in sequential greedy order (Section II-B: rows ascending,
// neighbours in stored order, the first free one taken), walked by one warp
// that is the only one to touch these vertices' states.
//
// Greedy order is a chain of decisions, bound by latency: one thread paid two
// dependent memory round trips for every entry.  Here the warp reads a window
// of 32 rows and then up to 128 entries at a time -- the ids one chunk ahead,
// the window's row states beside the first chunk's -- so a chunk costs one
// round trip, for the states of its vertices, and its decisions are made in
// registers: the first entry, in stored order, whose two vertices are both
// free is a pair, and every entry of the chunk that names either is dropped.
// A call on 4096 graphs of 100 to 10,000 edges (22 M entries, byte states):
// 16.5 ms with one thread a graph, 0.88 ms with one warp (0.63 with SerialBits);
// one Erdos-Renyi graph of 2 M entries 330 -> 28 ms.
template <class S>
__device__ __forceinline__ void serial_rows(const S& s, const SweepParams& P, uint64_t r0,
                                            uint64_t r1, const unsigned lane) {
  const uint64_t pol = policy_evict_first();
  const uint32_t n32 = (uint32_t)P.n;
  uint32_t next[4] = {0u, 0u, 0u, 0u};  // ids at next_at + 4 * lane
  int64_t next_at = -256;
  int64_t begin = 0, end = 0;           // row ends of the window after this one
  bool told = false;                    // the lane has reported an id out of range
  if (r0 + lane < r1) {
    begin = __ldg(P.offsets + r0 + lane);
    end = __ldg(P.offsets + r0 + lane + 1);
  }
  for (uint64_t wb = r0; wb < r1; wb += 32) {
    const bool in = wb + lane < r1;
    const int64_t my_begin = clamp_end(begin, P.nnz), my_end = clamp_end(end, P.nnz);  // not on the load's heels
    if (wb + 32 + lane < r1) {
      begin = __ldg(P.offsets + wb + 32 + lane);
      end = __ldg(P.offsets + wb + 32 + lane + 1);
    }
    // the row states arrive beside the first chunk's: until then every row reads as open
    const uint32_t my_st = in ? s.raw((uint32_t)(wb + lane)) : 0u;
    unsigned done = __ballot_sync(kFull, !in);  // vertices of the window that are matched (or past the last row)
    bool fresh = true;
    const int rows = r1 - wb < 32 ? (int)(r1 - wb) : 32;
    const int64_t win_end = __shfl_sync(kFull, my_end, rows - 1);
    const uint32_t wb32 = (uint32_t)wb;
    int64_t pos = 0;
    for (;;) {
      const unsigned open = __ballot_sync(kFull, my_end > pos) & ~done;
      if (open == 0u) break;
      const int64_t st = __shfl_sync(kFull, my_begin, __ffs(open) - 1);
      if (st > pos) pos = st;
      if (pos >= win_end) break;  // only empty rows were left
      const bool loaded = pos >= next_at && pos < next_at + 128;
      const int64_t base = loaded ? next_at : pos & ~(int64_t)3;
      const int64_t cend = base + 128 < win_end ? base + 128 : win_end;
      const int lo_r = (int)(pos - base), hi_r = (int)(cend - base), p0 = 4 * (int)lane;
      uint32_t y[4] = {next[0], next[1], next[2], next[3]};
      if (!loaded && p0 < hi_r) load_quad(P, base + p0, pol, y);
      next_at = base + 128 <= win_end ? base + 128 : win_end & ~(int64_t)3;
      load_quad(P, next_at + p0, pol, next);
      const int64_t d = my_end - base;
      const int rel = lane >= (unsigned)rows || d > 129 ? 129 : d < 0 ? -1 : (int)d;
      int k[4];
      uint32_t ry[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int j = 0; j < 4; ++j) k[j] = count_le(rel, p0 + j) & 31;
      uint32_t cand = 0;  // entries of open rows, loops apart; an id out of range stays, to be reported in its turn
      uint32_t bits[4];   // the window's rows that an entry names: its own, and y's if y is one of them
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int p = p0 + j;
        bits[j] = 1u << k[j] | (y[j] < n32 && y[j] - wb32 < 32u ? 1u << (y[j] - wb32) : 0u);
        if (p < lo_r || p >= hi_r || (done >> k[j] & 1u) || y[j] == wb32 + (uint32_t)k[j]) continue;
        cand |= 1u << j;
        if (y[j] < n32) ry[j] = s.raw(y[j]);
      }
      if (fresh) {
        done |= __ballot_sync(kFull, in && S::matched(my_st, wb32 + lane));
        fresh = false;
      }
      bool odd = in && S::reserved(my_st, wb32 + lane);  // entries that take the slow way below
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if ((bits[j] & done) || (y[j] < n32 && S::matched(ry[j], y[j]))) cand &= ~(1u << j);
        odd |= (cand >> j & 1u) && (y[j] >= n32 || S::reserved(ry[j], y[j]));
      }
      const bool any_odd = __any_sync(kFull, odd);
      uint32_t sx = 0, sy = 0;  // the chunk's i-th pair, on lane i
      int pairs = 0;
      for (;;) {
        const unsigned have = __ballot_sync(kFull, cand != 0u);
        if (have == 0u) break;
        const int first = __ffs(have) - 1;
        const int j = __ffs(cand) - 1;  // -1, and pick4's first, on the lanes without one
        const uint32_t yv = __shfl_sync(kFull, pick4(y, j), first);
        const int kx = __shfl_sync(kFull, pick4(k, j), first);
        const uint32_t xv = wb32 + (uint32_t)kx;
        if (any_odd) {  // an id out of range, or a poisoned vertex: wait for it, as any thread would
          uint32_t got = 0;
          if ((int)lane == first) {
            cand &= cand - 1u;
            if (yv >= n32) {
              if (!told) report(P.err, P.host_err, kErrBadId);
              told = true;
            } else if constexpr (S::kAlone) {  // both ends are free, or the entry had been dropped
              s.match_alone(xv, yv);
              got = 1u;
            } else {
              got = resolve_edge(s, xv, yv, s.raw(xv), s.raw(yv), P) ? 1u : 0u;
              got |= ld_relaxed(P.err) & kErrTimeout ? 2u : 0u;
            }
          }
          got = __shfl_sync(kFull, got, first);
          if (got & 2u) return;
          if (!(got & 1u)) continue;
        } else {
          if ((int)lane == pairs) {
            sx = xv;
            sy = yv;
          }
          ++pairs;  // at most one a row of the window
        }
        done |= 1u << kx | (yv - wb32 < 32u ? 1u << (yv - wb32) : 0u);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if ((bits[i] & done) || y[i] == yv) cand &= ~(1u << i);
      }
      if ((int)lane < pairs) s.match_alone(sx, sy);
      __syncwarp();  // the chunk's states are written before the next reads
      pos = cend;
    }
  }
}

// The whole graph of the view P in that order, with its states on the chip if they fit.
template <class S>
__device__ __forceinline__ void serial_graph(const SweepParams& P, unsigned lane) {
  __shared__ uint32_t bits[kSerialGraphsPerBlock][kSerialBits / 32];
  if (P.n > kSerialBits) {
    serial_rows(S(P), P, 0, P.n, lane);
    return;
  }
  uint32_t* const words = bits[threadIdx.x >> 5];
  for (uint32_t i = lane; i < (P.n + 31) / 32; i += 32) words[i] = 0u;
  __syncwarp();
  serial_rows(SerialBits{words, P.mate}, P, 0, P.n, lane);
}

}  // namespace
}  // namespace skp
