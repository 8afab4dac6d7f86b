// check.cu -- CSR input check, the exact maximal-matching checker and the
// ordered pair-list compaction, on the device.
//
// The checker follows the validation rule of Section II-B (every edge touches
// an output edge; no two output edges share an endpoint) with the counting
// rules stated in skipper.h, so its verdict can be compared field by field
// with a host checker.  Counters are summed per block and added with 64-bit
// atomics; "first offender" fields take the minimum, so every field is
// independent of thread timing.
#include <cstdint>
#include <cuda_runtime.h>

#include "internal.h"
#include "checkwalk.cuh"
#include "walk.cuh"

namespace skp {

namespace {

__global__ void zero_u64_kernel(unsigned long long* p, uint64_t words, unsigned long long v) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words;
       i += (uint64_t)gridDim.x * blockDim.x)
    p[i] = v;
}

__global__ void zero_u32_kernel(uint32_t* p, uint64_t words) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words;
       i += (uint64_t)gridDim.x * blockDim.x)
    p[i] = 0u;
}

__global__ void csr_check_kernel(uint64_t n, uint64_t nnz, const int64_t* __restrict__ offsets,
                                 const uint32_t* __restrict__ nbrs, unsigned long long* bad) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long local = 0;
  if (tid == 0 && (offsets[0] != 0 || offsets[n] != (int64_t)nnz)) ++local;
  for (uint64_t i = tid; i < n; i += stride)
    if (offsets[i] > offsets[i + 1]) ++local;
  for (uint64_t i = tid; i < nnz; i += stride)
    if (nbrs[i] >= n) ++local;
  if (local) atomicAdd(bad, local);
}

// edge-list input: every endpoint id < n
__global__ void coo_check_kernel(uint64_t n, uint64_t m, const uint32_t* __restrict__ src,
                                 const uint32_t* __restrict__ dst, unsigned long long* bad) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  unsigned long long local = 0;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride)
    local += (src[i] >= n) + (dst[i] >= n);
  if (local) atomicAdd(bad, local);
}

__device__ __forceinline__ void warp_add(unsigned long long* c, uint32_t v) {
  const uint32_t s = __reduce_add_sync(kFull, v);
  if ((threadIdx.x & 31) == 0 && s) atomicAdd(c, (unsigned long long)s);
}

// The checker over a CSR (checkwalk.cuh): one warp per 32 consecutive vertices.
// Bound by the latency of dependent reads (four round trips a vertex), so it
// takes as many warps as fit without spills (the kernels over many graphs spill at
// that count: kCheckBlocks); reading the next group's mates and
// row ends ahead spilled and cost 5 to 12%.  The whole check, against a
// partition, an edge pass, an existence pass with one warp a pair and a vertex
// pass: R-MAT 22 in 170 us (579 before), a 4096 x 4096 grid in 245 us (1645).
__global__ void __launch_bounds__(256, kCheckBlocks) check_csr_kernel(CheckView V, LongRows queue,
                                                            unsigned long long* __restrict__ c,
                                                            unsigned long long* __restrict__ host) {
  const unsigned lane = threadIdx.x & 31u;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  uint32_t matched = 0, pairs = 0;
  init_counts(lane);
  for (uint64_t v0 = warp * 32; v0 < V.n; v0 += nwarps * 32) {
    const bool in = v0 + lane < V.n;
    const uint32_t v = (uint32_t)v0 + lane;
    const Visit a = check_group<true>(V, in, v, load_vertex(V, in, v), 0, lane, queue);
    matched += __popc(__ballot_sync(kFull, a.bits & kVxMatched));
    pairs += __popc(__ballot_sync(kFull, a.bits & kVxPair));
    add_faults(a, v0 + lane, lane);
  }
  add_block(c, matched, pairs);
  publish_counters<false>(c, host);
}

// the queued pieces of unmatched vertices' rows, one a block
__global__ void check_csr_long_kernel(CheckView V, LongRows queue, unsigned long long* __restrict__ c,
                                      unsigned long long* __restrict__ host) {
  const unsigned long long pieces = queue.size();
  init_counts(threadIdx.x & 31u);
  for (unsigned long long i = blockIdx.x; i < pieces; i += gridDim.x) {
    const ulonglong2 item = queue.items[i];
    check_piece(V, (uint32_t)item.x, (int64_t)item.y, threadIdx.x & 31u);
  }
  add_block(c, 0, 0);
  publish_counters<true>(c, host);
}

// edge pass over an edge list: edge i = (x, y), x != y, both ids < n, is
// uncovered when both endpoints are unmatched; mate[x] == y marks found[x] and
// mate[y] == x marks found[y] (the listed edge is the output edge of x / y)
__global__ void validate_coo_edges_kernel(uint64_t n, uint64_t m, const uint32_t* __restrict__ src,
                                          const uint32_t* __restrict__ dst,
                                          const uint32_t* __restrict__ mate,
                                          unsigned char* __restrict__ found,
                                          unsigned long long* __restrict__ c) {
  const unsigned lane = threadIdx.x & 31u;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  unsigned long long unc = 0, first = ~0ull;
  for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x; i0 < m; i0 += stride) {
    const uint64_t i = i0 + threadIdx.x;
    if (i < m) {
      const uint32_t x = __ldg(src + i), y = __ldg(dst + i);
      if (x != y && x < n && y < n) {
        const uint32_t mx = __ldg(mate + x), my = __ldg(mate + y);
        if (mx == kNone && my == kNone) {
          ++unc;
          if (i < first) first = i;
        }
        if (mx == y) found[x] = 1;
        if (my == x) found[y] = 1;
      }
    }
  }
  unc = warp_sum64(unc);
  first = warp_min64(first);
  if (lane == 0) {
    if (unc) atomicAdd(c + kCkUncovered, unc);
    if (~first) atomicMax(c + kCkFirstUncovered, ~first);
  }
}

// vertex pass of an edge list: range and symmetry of each named partner, and
// its existence (the edge pass marks every vertex whose partner edge it met)
__global__ void validate_coo_vertex_kernel(uint64_t n, const uint32_t* __restrict__ mate,
                                           const unsigned char* __restrict__ found,
                                           unsigned long long* __restrict__ c,
                                           unsigned long long* __restrict__ host) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const unsigned lane = threadIdx.x & 31u;
  uint32_t matched = 0, pairs = 0;
  init_counts(lane);
  for (uint64_t v0 = (uint64_t)blockIdx.x * blockDim.x; v0 < n; v0 += stride) {
    const uint64_t v = v0 + threadIdx.x;
    const uint32_t m = v < n ? mate[v] : kNone;
    Visit a;
    if (m != kNone) {
      if (m >= n || m == v) {
        a.bits = kVxRange;
      } else {
        a.bits = kVxMatched | (mate[m] != (uint32_t)v ? kVxAsym : v < m ? kVxPair : 0u);
        if (!found[v] && !found[m]) a.bits |= kVxNonedge;  // the edge may be listed either way
      }
    }
    matched += __popc(__ballot_sync(kFull, a.bits & kVxMatched));
    pairs += __popc(__ballot_sync(kFull, a.bits & kVxPair));
    add_faults(a, v, lane);
  }
  add_block(c, matched, pairs);
  publish_counters<true>(c, host);
}

__global__ void validate_pairs_kernel(uint64_t n, const uint32_t* __restrict__ mate,
                                      const uint32_t* __restrict__ pairs, uint64_t count,
                                      uint32_t* __restrict__ seen, unsigned long long* __restrict__ c) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t j0 = (uint64_t)blockIdx.x * blockDim.x; j0 < count; j0 += stride) {
    const uint64_t j = j0 + threadIdx.x;
    uint32_t bad = 0;
    if (j < count) {
      const uint32_t a = pairs[2 * j], b = pairs[2 * j + 1];
      const bool valid = a < b && b < n && mate[a] == b && mate[b] == a;
      if (!valid) {
        bad = 1;
      } else {
        const uint32_t bit = 1u << (a & 31u);
        if (atomicOr(seen + (a >> 5), bit) & bit) bad = 1;  // a repeat of a valid pair
      }
    }
    warp_add(c + kCkPairsBad, bad);
  }
}

// ---- ordered compaction of (u, mate[u]), u < mate[u] ----
// One pass (a single-pass scan with decoupled look-back, Merrill and Garland 2016):
// a block takes the next tile of 16384 vertices (a ticket keeps the
// tiles in order), counts its pairs, learns how many come before them from the
// tiles before it -- each publishes its own count at once and the running total
// as soon as it knows it, in one 64-bit word -- and writes them.  Bound by
// memory: the mates are read once, in 128-bit loads, and the pairs written once.
// R-MAT 27 (134 M vertices): 573 us as a count, a scan and a scatter that read the
// mates twice, a thread 16 in a row; 291 us in one pass (tiles of 4096 vertices:
// 381, held up by the look back).
constexpr int kCompactThreads = 512, kCompactQuads = 8, kCompactWarps = kCompactThreads / 32;
static_assert(kCompactTile == 4 * kCompactQuads * kCompactThreads, "a thread takes eight quads of a tile");
static_assert(kCompactQuads * kCompactWarps == 128, "a lane of the scan takes four of the tile's parts");
constexpr uint64_t kTileOwn = 1ull << 62, kTileTotal = 2ull << 62, kTileValue = kTileOwn - 1;
constexpr uint32_t kTilePolls = 1u << 24;

__device__ __forceinline__ uint64_t ld_tile(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_tile(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// pairs before tile t: the totals and counts of the tiles before it, 32 at a
// time (the whole warp); a wait that runs out sets `err` and answers with less
__device__ __forceinline__ uint64_t pairs_before(const uint64_t* tiles, int64_t t, unsigned lane, uint32_t* err,
                                                 uint32_t* host_err) {
  uint64_t before = 0;
  for (int64_t p = t - 1; p >= 0; p -= 32) {
    const int64_t i = p - lane;
    uint64_t v = i >= 0 ? ld_tile(tiles + i) : kTileTotal;
    for (uint32_t polls = 0; __any_sync(kFull, v <= kTileValue); ++polls) {
      if (polls > kTilePolls) {
        if (lane == 0) report(err, host_err, kErrTimeout);
        return before;
      }
      if (v <= kTileValue) v = ld_tile(tiles + i);
    }
    const unsigned known = __ballot_sync(kFull, v >= kTileTotal);
    const int last = known ? __ffs(known) - 1 : 31;   // the nearest tile that knows its total
    uint64_t x = (int)lane <= last ? v & kTileValue : 0;
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) x += __shfl_xor_sync(kFull, x, d);
    before += x;
    if (known) break;
  }
  return before;
}

// state: [ticket | a word per tile], zero before the launch
__global__ void __launch_bounds__(kCompactThreads, 2) compact_kernel(uint64_t n, const uint32_t* __restrict__ mate,
                                                                  uint32_t* __restrict__ pairs, uint64_t cap,
                                                                  uint64_t* __restrict__ count,
                                                                  uint64_t* __restrict__ state, uint32_t* err,
                                                                     uint32_t* host_err) {
  __shared__ uint32_t tile_s;
  __shared__ __align__(16) uint32_t sub[128];   // pairs before each 128 vertices of the tile
  __shared__ uint64_t before_s;
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) tile_s = atomicAdd(reinterpret_cast<uint32_t*>(state), 1u);
  __syncthreads();
  const uint64_t t = tile_s, base = t * kCompactTile + 4 * threadIdx.x;
  const bool wide = (reinterpret_cast<uintptr_t>(mate) & 15u) == 0;
  uint32_t m[kCompactQuads][4];
#pragma unroll
  for (int i = 0; i < kCompactQuads; ++i) {  // quad i: vertices base + 2048 i on
    const uint64_t u = base + 4 * kCompactThreads * i;
    if (wide && u + 4 <= n) {
      const uint4 q = *reinterpret_cast<const uint4*>(mate + u);
      m[i][0] = q.x; m[i][1] = q.y; m[i][2] = q.z; m[i][3] = q.w;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) m[i][j] = u + j < n ? mate[u + j] : kNone;
    }
  }
  uint32_t take = 0, cnt[2] = {0, 0};  // a bit per vertex; a byte per quad
#pragma unroll
  for (int i = 0; i < kCompactQuads; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (m[i][j] != kNone && m[i][j] < n && base + 4 * kCompactThreads * i + j < m[i][j]) {
        take |= 1u << (4 * i + j);
        cnt[i / 4] += 1u << (8 * (i % 4));
      }
  uint32_t upto[2] = {cnt[0], cnt[1]};  // four sums over the lanes at once, each at most 128
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y0 = __shfl_up_sync(kFull, upto[0], d), y1 = __shfl_up_sync(kFull, upto[1], d);
    if ((int)lane >= d) {
      upto[0] += y0;
      upto[1] += y1;
    }
  }
  if (lane == 31)
#pragma unroll
    for (int i = 0; i < kCompactQuads; ++i) sub[kCompactWarps * i + warp] = upto[i / 4] >> (8 * (i % 4)) & 255u;
  __syncthreads();
  if (warp == 0) {
    const uint4 part = reinterpret_cast<const uint4*>(sub)[lane];
    const uint32_t own = part.x + part.y + part.z + part.w;
    uint32_t x = own;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, x, d);
      if ((int)lane >= d) x += y;
    }
    const uint32_t first = x - own;
    reinterpret_cast<uint4*>(sub)[lane] =
        make_uint4(first, first + part.x, first + part.x + part.y, first + part.x + part.y + part.z);
    const uint64_t total = __shfl_sync(kFull, x, 31);
    uint64_t* tiles = state + 1;
    if (lane == 0 && t) st_tile(tiles + t, kTileOwn | total);
    const uint64_t before = pairs_before(tiles, (int64_t)t, lane, err, host_err);
    if (lane == 0) {
      st_tile(tiles + t, kTileTotal | (before + total));
      before_s = before;
      if (count && t == gridDim.x - 1) *count = before + total;
    }
  }
  if (!pairs) return;
  __syncthreads();
  const bool wide_pairs = (reinterpret_cast<uintptr_t>(pairs) & 7u) == 0;
#pragma unroll
  for (int i = 0; i < kCompactQuads; ++i) {
    uint64_t pos = before_s + sub[kCompactWarps * i + warp] + ((upto[i / 4] - cnt[i / 4]) >> (8 * (i % 4)) & 255u);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (take >> (4 * i + j) & 1u) {
        const uint32_t u = (uint32_t)(base + 4 * kCompactThreads * i + j);
        if (pos < cap) {
          if (wide_pairs) {
            *reinterpret_cast<uint2*>(pairs + 2 * pos) = make_uint2(u, m[i][j]);
          } else {
            pairs[2 * pos] = u;
            pairs[2 * pos + 1] = m[i][j];
          }
        }
        ++pos;
      }
  }
}

}  // namespace

// pieces that the long rows of a CSR with nnz entries can have: those that a row fills,
// and one more a row
uint64_t long_row_cap(uint64_t nnz, bool one) {
  const uint64_t row = (uint64_t)long_row(one);
  return nnz > row ? nnz / (uint64_t)kPiece + nnz / row : 0;
}

// blocks of 256 threads for n vertices: no more than their groups of 32 fill, or than are resident
int check_grid(uint64_t n, int sms) {
  const uint64_t blocks = (n + 255) / 256;
  return blocks < (uint64_t)sms * kCheckBlocks ? (int)(blocks ? blocks : 1) : sms * kCheckBlocks;
}

cudaError_t launch_csr_check(uint64_t n, uint64_t nnz, const int64_t* offsets,
                             const uint32_t* nbrs, unsigned long long* bad, int grid,
                             cudaStream_t s) {
  zero_u64_kernel<<<1, 32, 0, s>>>(bad, 1, 0ull);
  csr_check_kernel<<<grid, 256, 0, s>>>(n, nnz, offsets, nbrs, bad);
  return cudaGetLastError();
}

cudaError_t launch_validate(uint64_t n, uint64_t nnz, const int64_t* offsets, const uint32_t* nbrs,
                            const uint32_t* mate, const uint32_t* pairs, uint64_t count,
                            const CheckScratch& cs, int sms, cudaStream_t s) {
  const int grid = sms * 8;
  if (pairs && count) {
    zero_u32_kernel<<<grid, 256, 0, s>>>(cs.seen_bits, (n + 31) / 32);
    validate_pairs_kernel<<<grid, 256, 0, s>>>(n, mate, pairs, count, cs.seen_bits, cs.counters);
  }
  const CheckView V{offsets, nbrs, mate, n, nnz};
  const LongRows queue{cs.counters + kCkLong, cs.long_rows, long_row_cap(nnz, true)};
  check_csr_kernel<<<check_grid(n, sms), 256, 0, s>>>(V, queue, cs.counters, cs.host);
  return cudaGetLastError();
}

bool validate_needs_long(const CheckScratch& cs) { return cs.host[kCkLong] != 0; }

cudaError_t launch_validate_long(uint64_t n, uint64_t nnz, const int64_t* offsets, const uint32_t* nbrs,
                                 const uint32_t* mate, const CheckScratch& cs, int sms, cudaStream_t s) {
  check_csr_long_kernel<<<sms * 4, 256, 0, s>>>(CheckView{offsets, nbrs, mate, n, nnz},
                                                LongRows{cs.counters + kCkLong, cs.long_rows, long_row_cap(nnz, true)},
                                                cs.counters, cs.host);
  return cudaGetLastError();
}

cudaError_t launch_coo_check(uint64_t n, uint64_t m, const uint32_t* src, const uint32_t* dst,
                             unsigned long long* bad, int grid, cudaStream_t s) {
  zero_u64_kernel<<<1, 32, 0, s>>>(bad, 1, 0ull);
  if (m) coo_check_kernel<<<grid, 256, 0, s>>>(n, m, src, dst, bad);
  return cudaGetLastError();
}

cudaError_t launch_validate_coo(uint64_t n, uint64_t m, const uint32_t* src, const uint32_t* dst,
                                const uint32_t* mate, const uint32_t* pairs, uint64_t count,
                                const CheckScratch& cs, int sms, cudaStream_t s) {
  const int grid = sms * 8;
  if (pairs && count) {
    zero_u32_kernel<<<grid, 256, 0, s>>>(cs.seen_bits, (n + 31) / 32);
    validate_pairs_kernel<<<grid, 256, 0, s>>>(n, mate, pairs, count, cs.seen_bits, cs.counters);
  }
  if (n) zero_u32_kernel<<<grid, 256, 0, s>>>(reinterpret_cast<uint32_t*>(cs.found), (n + 3) / 4);
  if (n && m) validate_coo_edges_kernel<<<grid, 256, 0, s>>>(n, m, src, dst, mate, cs.found, cs.counters);
  validate_coo_vertex_kernel<<<grid, 256, 0, s>>>(n, mate, cs.found, cs.counters, cs.host);
  return cudaGetLastError();
}

namespace {

// Census of a state array: out[0..3] = ACC, RSVD, MCHD, other field values.
__global__ void census_kernel(const uint32_t* __restrict__ state, uint64_t n, int bits,
                              unsigned long long* __restrict__ out) {
  unsigned long long c[4] = {0, 0, 0, 0};
  const uint64_t per = bits == 32 ? 1 : 32u / (uint32_t)bits;
  const uint32_t mask = bits == 32 ? 0u : (1u << bits) - 1u;
  for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t w = state[v / per];
    int k;
    if (bits == 32) {
      k = w == kWAcc ? 0 : (w == kWRsvd ? 1 : 2);
    } else {
      const uint32_t f = (w >> ((v % per) * (uint32_t)bits)) & mask;
      k = f == kAcc ? 0 : f == kRsvd ? 1 : f == kMchd ? 2 : 3;
    }
    ++c[k];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const unsigned long long t = warp_sum64(c[k]);
    if ((threadIdx.x & 31) == 0 && t) atomicAdd(out + k, t);
  }
}

}  // namespace

cudaError_t launch_census(const uint32_t* state, uint64_t n, int bits, unsigned long long* out,
                          int grid, cudaStream_t s) {
  zero_u64_kernel<<<1, 32, 0, s>>>(out, 4, 0ull);
  if (n) census_kernel<<<grid, 256, 0, s>>>(state, n, bits, out);
  return cudaGetLastError();
}

uint64_t compact_words(uint64_t n) { return (n + kCompactTile - 1) / kCompactTile + 1; }

cudaError_t launch_compact(uint64_t n, const uint32_t* mate, uint32_t* pairs, uint64_t cap, uint64_t* count,
                           uint64_t* state, uint32_t* err, uint32_t* host_err, cudaStream_t s) {
  if (n == 0) {
    if (count) zero_u64_kernel<<<1, 32, 0, s>>>(reinterpret_cast<unsigned long long*>(count), 1, 0ull);
    return cudaGetLastError();
  }
  compact_kernel<<<(unsigned)(compact_words(n) - 1), kCompactThreads, 0, s>>>(n, mate, cap ? pairs : nullptr, cap, count,
                                                                             state, err, host_err);
  return cudaGetLastError();
}

}  // namespace skp
