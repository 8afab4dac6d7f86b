// checkwalk.cuh -- the exact checker's walk (Section II-B: every graph edge
// touches an output edge; each output edge is a graph edge; no vertex is in
// two), shared by the single-graph, packed-batch and multi-graph checkers.
//
// One warp takes 32 consecutive vertices, one a lane (check_group), and does
// all of a vertex's checking in one visit:
//   v matched to m: m in range, mate[m] == v, and an edge between them, stored
//     in row v or in row m (the CSR may hold an edge for one endpoint only):
//     the shorter row is searched first and left at the first hit; a symmetric
//     pair is searched once, by its lower endpoint, and counts for both.
//   v unmatched: every entry (v, y), y != v, must have mate[y] set (an entry of
//     a matched row is covered).
// Counting rules are those of the host checker.
//
// The visit is bound by latency -- mate[v], then mate[m] and m's row ends, then
// ids, then their mates -- and most rows it reads are a few entries long, so a
// lane reads its own row, 8 entries a step, which keeps 32 rows in flight a
// warp; a row of more than kLaneQuads quads is read by the whole warp, 256
// entries a step.  A row of an unmatched vertex longer than long_row entries
// is cut into pieces, which a second kernel hands to the GPU's blocks.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "state.cuh"

namespace skp {

// counters of one verdict, in mm_verdict's order after the flags.  The two
// "first offender" fields hold the complement of the index and grow
// (atomicMax), so that a block of zeros is a fresh set of counters.
enum CheckSlot : int { kCkMatched = 0, kCkPairs, kCkRange, kCkAsym, kCkNonedge, kCkUncovered, kCkPairsBad,
                       kCkFirstBad, kCkFirstUncovered, kCkCount,
                       // control words behind them: long rows queued, blocks done
                       kCkLong = kCkCount, kCkDone, kCkWords };
constexpr int64_t kPiece = 8192;     // entries of a piece of a long row, at most (4096, 2048: 18 and 33% slower)
// Entries from which a row is long: over one graph a warp keeps up with up to a
// piece; over many, where it also fetches each row's graph from another lane, with
// less (40,000 rows of 3000 entries: 1560 us by warps, 690 in pieces).
__host__ __device__ constexpr int64_t long_row(bool one) { return one ? kPiece : 2048; }
// Resident blocks of 256 threads an SM.  4 / 5 / 6: a 4096 x 4096 grid 211 / 186 /
// 188 us, R-MAT 24 713 / 688 / 719.  Over many graphs, where a lane carries a graph of
// its own and spills (176 bytes of stores in the batch kernel, 216 in the multi-graph
// one; 56 at 4 blocks), the 4096-graph batch 474 / 492 / 496, 171 graphs 424 / 408 / 426.
constexpr int kCheckBlocks = 5;

namespace {

// 8 / 16 / 32 quads: the 4096-graph batch's check 339 / 324 / 320 us, R-MAT 22's 170 / 174 / 185
constexpr int64_t kLaneQuads = 16;

// a graph as the checker reads it (nbrs 16-byte aligned, nnz entries in all).  Row
// ends that were never checked may lie anywhere: a position outside the entries
// holds no id (check_quad), and rows longer than a lane takes are clamped before
// they are walked.  Clamping every row as it is loaded cost 12 to 17% on lattices.
struct CheckView {
  const int64_t* offsets;
  const uint32_t* nbrs;
  const uint32_t* mate;
  uint64_t n, nnz;
};

// what one visit found: the vertex's bits, and the uncovered entries this lane met
enum : uint32_t { kVxMatched = 1u, kVxPair = 2u, kVxRange = 4u, kVxAsym = 8u, kVxNonedge = 16u,
                  kVxBothEnds = 32u /* a missing edge of a symmetric pair: counts for both ends */,
                  kVxBad = kVxRange | kVxAsym | kVxNonedge };
struct Visit {
  uint32_t bits = 0, uncovered = 0;
  unsigned long long first_unc = ~0ull;
};

// Pieces of long rows of unmatched vertices, left to the second kernel: graph <<
// 32 | vertex, and the number of the piece in its row.  A row spread over the
// whole grid a row at a time kept only the blocks its length reached at work, and
// all of them walking the queue: 39,000 rows of 17,000 to 22,000 entries 44.5 ms,
// in pieces 1.25.  cap counts the pieces of rows that do not overlap; row ends
// that were never checked may, and what does not fit is read at once.
struct LongRows {
  unsigned long long* count;
  ulonglong2* items;
  uint64_t cap;
  // the whole warp queues the k pieces of a row; returns how many fitted
  __device__ __forceinline__ int64_t push(uint64_t row, int64_t k, unsigned lane) const {
    unsigned long long at = 0;
    if (lane == 0) at = atomicAdd(count, (unsigned long long)k);
    at = __shfl_sync(kFull, at, 0);
    const int64_t fit = at >= cap ? 0 : (uint64_t)k < cap - at ? k : (int64_t)(cap - at);
    for (int64_t i = lane; i < fit; i += 32) items[at + i] = make_ulonglong2(row, (unsigned long long)i);
    return fit;
  }
  __device__ __forceinline__ unsigned long long size() const { return *count < cap ? *count : cap; }
};

// a row of `len` entries in pieces of at most kPiece, all but the last of one length
__device__ __forceinline__ int64_t long_pieces(int64_t len) { return (len + kPiece - 1) / kPiece; }
__device__ __forceinline__ int64_t piece_length(int64_t len) {
  const int64_t k = long_pieces(len);
  return (len + k - 1) / k;
}

// last g < G with base[g] <= x (base ascending, base[0] = 0 <= x < base[G]), found by the whole warp;
// some g < G whatever base holds
template <class T>
__device__ __forceinline__ uint64_t warp_last_at_or_below(const T* base, uint64_t G, uint64_t x, unsigned lane) {
  uint64_t lo = 0, hi = G;
  while (hi - lo > 1) {
    const uint64_t step = (hi - lo + 31) / 32, at = lo + lane * step;
    const unsigned below = __ballot_sync(kFull, at < hi && (uint64_t)__ldg(base + at) <= x);
    lo += (uint64_t)(below ? __popc(below) - 1 : 0) * step;
    hi = lo + step < hi ? lo + step : hi;
  }
  return lo;
}

__device__ __forceinline__ void lower(unsigned long long& first, unsigned long long at) {
  if (at < first) first = at;
}

__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(kFull, v, d);
  return v;
}

__device__ __forceinline__ unsigned long long warp_min64(unsigned long long v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    const unsigned long long o = __shfl_xor_sync(kFull, v, d);
    v = o < v ? o : v;
  }
  return v;
}

// the ids at [q, q + 4), q a multiple of 4 below `e`; kNone, which is no vertex, where no entry is
__device__ __forceinline__ uint4 check_quad(const uint32_t* nbrs, uint64_t nnz, int64_t q, int64_t e) {
  uint4 y = make_uint4(kNone, kNone, kNone, kNone);
  if (q >= e) return y;
  const uint64_t whole = nnz & ~3ull;  // entries in whole quads
  if ((uint64_t)q < whole) return __ldg(reinterpret_cast<const uint4*>(nbrs + q));
  if ((uint64_t)q != whole) return y;
  if (whole < nnz) y.x = __ldg(nbrs + q);
  if (whole + 1 < nnz) y.y = __ldg(nbrs + q + 1);
  if (whole + 2 < nnz) y.z = __ldg(nbrs + q + 2);
  return y;
}

__device__ __forceinline__ bool quad_has(const uint4& y, int64_t q, int64_t s, int64_t e, uint32_t t) {
  return (y.x == t && q >= s && q < e) || (y.y == t && q + 1 >= s && q + 1 < e) ||
         (y.z == t && q + 2 >= s && q + 2 < e) || (y.w == t && q + 3 >= s && q + 3 < e);
}

// entries of the quad in [s, e) that leave the edge {x, y} uncovered (x is unmatched)
__device__ __forceinline__ void quad_scan(const uint4& y4, int64_t q, int64_t s, int64_t e, uint32_t x,
                                          const uint32_t* mate, uint64_t n, Visit& a) {
  const uint32_t y[4] = {y4.x, y4.y, y4.z, y4.w};
  bool free_y[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const bool live = q + j >= s && q + j < e && y[j] != x && y[j] < n;
    free_y[j] = live && __ldg(mate + (live ? y[j] : 0u)) == kNone;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (free_y[j]) {
      ++a.uncovered;
      lower(a.first_unc, (unsigned long long)(q + j));
    }
}

// Does [s, e) hold the id t?  The whole warp reads, 256 entries a step.
__device__ __forceinline__ bool warp_row_has(const uint32_t* nbrs, uint64_t nnz, int64_t s, int64_t e,
                                             uint32_t t, unsigned lane) {
  for (int64_t b = s & ~(int64_t)3; b < e; b += 256) {
    const int64_t q = b + 4 * (int64_t)lane;
    const uint4 y0 = check_quad(nbrs, nnz, q, e), y1 = check_quad(nbrs, nnz, q + 128, e);
    if (__any_sync(kFull, quad_has(y0, q, s, e, t) || quad_has(y1, q + 128, s, e, t))) return true;
  }
  return false;
}

template <class T>
__device__ __forceinline__ T* shfl_ptr(T* p, int j) {
  return reinterpret_cast<T*>(__shfl_sync(kFull, reinterpret_cast<unsigned long long>(p), j));
}

// Vertex v of the graph V with what load_vertex read of it, one a lane (`in`: the lane has one); `graph` is the
// graph's number in the queue.  kOne: all lanes read one graph, and an
// uncovered entry may be counted by any lane.
struct VertexRow {
  uint32_t m = kNone;    // mate[v]
  int64_t s = 0, e = 0;  // row v
};
__device__ __forceinline__ VertexRow load_vertex(const CheckView& V, bool in, uint32_t v) {
  VertexRow r;
  if (in) {
    r.m = __ldg(V.mate + v);
    r.s = __ldg(V.offsets + v);
    r.e = __ldg(V.offsets + v + 1);
  }
  return r;
}

template <bool kOne>
__device__ __forceinline__ Visit check_group(const CheckView& V, bool in, uint32_t v, const VertexRow& row,
                                             uint32_t graph, unsigned lane, const LongRows& queue) {
  Visit a;
  const uint32_t m = row.m;
  int64_t s = row.s, e = row.e;            // what is left of the row to read
  uint32_t t = m;                          // the id searched for in it
  const uint32_t other = v ^ m;            // t ^ other: the row's own vertex
  bool find = false, again = true;         // search for t; the other row is still to come
  if (m != kNone) {
    if (m >= V.n || m == v) {
      a.bits = kVxRange;
    } else {
      const bool sym = __ldg(V.mate + m) == v;
      a.bits = kVxMatched | (sym ? kVxBothEnds | (v < m ? kVxPair : 0u) : kVxAsym);
      find = !sym || v < m;
      if (find) {
        const int64_t s2 = __ldg(V.offsets + m), e2 = __ldg(V.offsets + m + 1);
        if (e2 - s2 < e - s) {             // the shorter row first
          s = s2;
          e = e2;
          t = v;
        }
      }
    }
  }
  bool todo = find || (in && m == kNone && s < e);
  for (;;) {  // short rows: one a lane
    const bool mine = todo && ((e - 1) >> 2) - (s >> 2) < kLaneQuads;
    if (!__any_sync(kFull, mine)) break;
    if (!mine) continue;
    const int64_t q = s & ~(int64_t)3;
    const uint4 y0 = check_quad(V.nbrs, V.nnz, q, e), y1 = check_quad(V.nbrs, V.nnz, q + 4, e);
    if (find) {
      if (quad_has(y0, q, s, e, t) || quad_has(y1, q + 4, s, e, t)) {
        todo = false;
        continue;
      }
    } else {
      quad_scan(y0, q, s, e, v, V.mate, V.n, a);
      quad_scan(y1, q + 4, s, e, v, V.mate, V.n, a);
    }
    s = q + 8;
    if (s < e) continue;
    if (find && again) {
      again = false;
      s = __ldg(V.offsets + t);
      e = __ldg(V.offsets + t + 1);
      t ^= other;
    } else {
      todo = false;
      if (find) a.bits |= kVxNonedge;
    }
  }
  unsigned left = __ballot_sync(kFull, todo);
  while (left) {  // longer rows: the warp reads one at a time
    const int j = __ffs(left) - 1;
    left &= left - 1;
    const uint32_t* nbrs = kOne ? V.nbrs : shfl_ptr(V.nbrs, j);
    const uint64_t nnz = kOne ? V.nnz : __shfl_sync(kFull, V.nnz, j);
    int64_t sj = clamp_end(__shfl_sync(kFull, s, j), nnz);
    const int64_t ej = clamp_end(__shfl_sync(kFull, e, j), nnz);
    if (__shfl_sync(kFull, find ? 1 : 0, j)) {
      const uint32_t tj = __shfl_sync(kFull, t, j), oj = __shfl_sync(kFull, other, j);
      bool hit = warp_row_has(nbrs, nnz, sj, ej, tj, lane);
      if (!hit && __shfl_sync(kFull, again ? 1 : 0, j)) {
        const int64_t* offsets = kOne ? V.offsets : shfl_ptr(V.offsets, j);
        hit = warp_row_has(nbrs, nnz, row_end(offsets, tj, nnz), row_end(offsets, (uint64_t)tj + 1, nnz), tj ^ oj, lane);
      }
      if (!hit && (int)lane == j) a.bits |= kVxNonedge;
    } else {
      const uint32_t xj = __shfl_sync(kFull, v, j);
      if (ej - sj > long_row(kOne)) {
        const int64_t k = long_pieces(ej - sj);
        const int64_t fit = queue.push((uint64_t)__shfl_sync(kFull, graph, j) << 32 | xj, k, lane);
        if (fit == k) continue;
        sj += fit * piece_length(ej - sj);
      }
      const uint32_t* mate = kOne ? V.mate : shfl_ptr(V.mate, j);
      const uint64_t n = kOne ? V.n : __shfl_sync(kFull, V.n, j);
      Visit part;
      for (int64_t b = sj & ~(int64_t)3; b < ej; b += 256) {
        const int64_t q = b + 4 * (int64_t)lane;
        const uint4 y0 = check_quad(nbrs, nnz, q, ej), y1 = check_quad(nbrs, nnz, q + 128, ej);
        quad_scan(y0, q, sj, ej, xj, mate, n, part);
        quad_scan(y1, q + 128, sj, ej, xj, mate, n, part);
      }
      if (kOne) {
        a.uncovered += part.uncovered;
        lower(a.first_unc, part.first_unc);
      } else if (__any_sync(kFull, part.uncovered != 0u)) {
        const uint32_t total = __reduce_add_sync(kFull, part.uncovered);
        const unsigned long long first = warp_min64(part.first_unc);
        if ((int)lane == j) {
          a.uncovered += total;
          lower(a.first_unc, first);
        }
      }
    }
  }
  return a;
}

__device__ __forceinline__ void add_nonzero(unsigned long long* c, unsigned long long v) {
  if (v) atomicAdd(c, v);
}

// What a warp has counted so far, in shared memory (blocks of 256 threads):
// added to the verdict's counters when it is done, not group by group -- a wrong
// matching has faults in every group, and 2.5 M pairs of atomics on two words
// took most of the check of an empty matching of a 9000 x 9000 grid.
__device__ __forceinline__ unsigned long long* warp_counts() {
  __shared__ unsigned long long counts[8][kCkCount];
  return counts[threadIdx.x >> 5];
}
__device__ __forceinline__ void init_counts(unsigned lane) {
  if (lane < kCkCount) warp_counts()[lane] = 0ull;
  __syncwarp();
}

// The faults of one visit, each lane's vertex reported as index `at`, into the
// warp's counts (every lane takes part).
__device__ __forceinline__ void add_faults(const Visit& a, unsigned long long at, unsigned lane) {
  if (!__any_sync(kFull, (a.bits & kVxBad) != 0u || a.uncovered != 0u)) return;
  const uint32_t range = __popc(__ballot_sync(kFull, a.bits & kVxRange));
  const uint32_t asym = __popc(__ballot_sync(kFull, a.bits & kVxAsym));
  const unsigned missing = __ballot_sync(kFull, a.bits & kVxNonedge);
  const uint32_t nonedge = __popc(missing) + __popc(missing & __ballot_sync(kFull, a.bits & kVxBothEnds));
  const uint32_t uncovered = __reduce_add_sync(kFull, a.uncovered);
  const unsigned long long bad = warp_min64(a.bits & kVxBad ? at : ~0ull), unc = warp_min64(a.first_unc);
  if (lane == 0) {
    unsigned long long* const c = warp_counts();
    c[kCkRange] += range;
    c[kCkAsym] += asym;
    c[kCkNonedge] += nonedge;
    c[kCkUncovered] += uncovered;
    if (~bad > c[kCkFirstBad]) c[kCkFirstBad] = ~bad;
    if (~unc > c[kCkFirstUncovered]) c[kCkFirstUncovered] = ~unc;
  }
}

// The warp's counts into counters `c`, and the warp's left at zero.
__device__ __forceinline__ void flush_counts(unsigned long long* c, unsigned lane) {
  __syncwarp();
  if (lane < kCkCount) {
    const unsigned long long v = warp_counts()[lane];
    if (v) lane < kCkFirstBad ? atomicAdd(c + lane, v) : atomicMax(c + lane, v);
    warp_counts()[lane] = 0ull;
  }
  __syncwarp();
}

// One queued piece of row x, read by a block.
__device__ __forceinline__ void check_piece(const CheckView& V, uint32_t x, int64_t piece, unsigned lane) {
  const int64_t s0 = row_end(V.offsets, x, V.nnz), e0 = row_end(V.offsets, (uint64_t)x + 1, V.nnz);
  const int64_t step = piece_length(e0 - s0), s = s0 + piece * step, e = s + step < e0 ? s + step : e0;
  Visit a;
  for (int64_t q = (s & ~(int64_t)3) + 4 * (int64_t)threadIdx.x; q < e; q += 8 * (int64_t)blockDim.x) {
    const int64_t p = q + 4 * (int64_t)blockDim.x;
    const uint4 y0 = check_quad(V.nbrs, V.nnz, q, e), y1 = check_quad(V.nbrs, V.nnz, p, e);
    quad_scan(y0, q, s, e, x, V.mate, V.n, a);
    quad_scan(y1, p, s, e, x, V.mate, V.n, a);
  }
  add_faults(a, 0, lane);
}

// A block's counts, with its matched vertices and pairs (each warp's on all its
// lanes), added once a block: added a warp at a time, the counts of 16.8 M
// vertices took most of a 0.69 ms pass.
__device__ __forceinline__ void add_block(unsigned long long* c, uint32_t matched, uint32_t pairs) {
  if ((threadIdx.x & 31u) == 0) {
    warp_counts()[kCkMatched] += matched;
    warp_counts()[kCkPairs] += pairs;
  }
  __syncthreads();
  if (threadIdx.x < kCkCount) {
    const unsigned long long* const at = warp_counts() + threadIdx.x;  // the first warp's; the others' lie behind
    unsigned long long t = 0;
    for (unsigned w = 0; w < blockDim.x >> 5; ++w) {
      const unsigned long long v = at[w * kCkCount];
      t = threadIdx.x < kCkFirstBad ? t + v : v > t ? v : t;
    }
    if (t) threadIdx.x < kCkFirstBad ? atomicAdd(c + threadIdx.x, t) : atomicMax(c + threadIdx.x, t);
  }
}

// The last block of the launch to get here writes the finished counters to
// page-locked host memory and leaves the device's zeroed for the next check:
// no launch before to clear them, no copy after to fetch them.  With long rows
// still queued (host[kCkLong] != 0) the counters stay as they are, for the
// kernel that reads those rows (kFinal).
template <bool kFinal>
__device__ __forceinline__ void publish_counters(unsigned long long* c, unsigned long long* host) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(c + kCkDone, 1ull) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  const unsigned long long rows = kFinal ? 0ull : atomicAdd(c + kCkLong, 0ull);
  if (threadIdx.x == 0) host[kCkLong] = rows;
  if (rows) {
    if (threadIdx.x == 0) c[kCkDone] = 0ull;
  } else {
    __syncthreads();  // every thread has read kCkLong
    if (threadIdx.x < kCkWords) {
      const unsigned long long v = atomicExch(c + threadIdx.x, 0ull);
      if (threadIdx.x < kCkCount) host[threadIdx.x] = threadIdx.x >= kCkFirstBad ? ~v : v;
    }
  }
  __threadfence_system();
}

}  // namespace
}  // namespace skp
