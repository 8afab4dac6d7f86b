// chip.cu -- Skipper over graphs whose vertex states fit in one SM's shared
// memory: one block walks a whole graph.
//
// The sweep's time on small graphs, and on graphs whose ids have locality, goes
// into reservations (Algorithm 1 lines 11 to 18): two dependent atomics an
// attempt, and waits on reservations that other warps hold.  In global memory
// each of those steps is a round trip to L2 of 0.5 to 0.8 us; in shared memory
// it is some tens of nanoseconds.  So where a graph's states fit, a block
// keeps them on the chip: it zeroes them, walks the graph's rows with the same
// per-warp walk as the sweep (walk.cuh, the same state machine and waits, one
// byte or 2 bits a vertex), and writes the mates of the vertices that stayed
// unmatched.  There is no state array to prepare, no partition and, for a single
// graph, no second launch.
//
// Windows of 32 rows are handed to the block's warps on demand from a shared
// counter; a window of more than kLongWindow entries is put aside and cut into
// pieces for all warps once the others are done.
#include <cstdint>
#include <cuda_runtime.h>

#include "chip.cuh"
#include "walk.cuh"

namespace skp {

namespace {

constexpr int kSingleThreads = 1024;
constexpr int64_t kLongWindow = 8192, kPiece = 2048;  // entries
constexpr uint32_t kMaxLong = 512;

__device__ __forceinline__ uint32_t lds(uint32_t at) {
  uint32_t v;
  asm volatile("ld.relaxed.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
  return v;
}

// Packed states in shared memory (see PackedState for the transitions).
template <int kBits>
struct ChipState {
  static constexpr bool kNear = true;
  static constexpr uint32_t kPerWord = 32u / kBits;
  static constexpr uint32_t kMask = (1u << kBits) - 1u;
  uint32_t words;   // shared-memory address
  uint32_t* mate;
  __device__ __forceinline__ uint32_t at(uint32_t v) const { return words + 4 * (v / kPerWord); }
  __device__ static __forceinline__ uint32_t shift(uint32_t v) { return (v % kPerWord) * kBits; }
  __device__ __forceinline__ uint32_t raw(uint32_t v) const { return lds(at(v)); }
  __device__ __forceinline__ uint32_t peek(uint32_t v) const { return lds(at(v)); }
  __device__ static __forceinline__ bool matched(uint32_t raw, uint32_t v) { return (raw >> shift(v)) & kMchd; }
  __device__ __forceinline__ uint32_t take(uint32_t v) const {
    uint32_t old;
    asm volatile("atom.relaxed.cta.shared::cta.or.b32 %0, [%1], %2;"
                 : "=r"(old)
                 : "r"(at(v)), "r"(kRsvd << shift(v))
                 : "memory");
    return (old >> shift(v)) & kMask;
  }
  __device__ __forceinline__ void put_back(uint32_t v, uint32_t was) const {
    if (!(was & kRsvd))
      asm volatile("red.relaxed.cta.shared::cta.and.b32 [%0], %1;" ::"r"(at(v)), "r"(~(kRsvd << shift(v))) : "memory");
  }
  __device__ __forceinline__ void commit_both(uint32_t u, uint32_t v) const {
    mate[u] = v;
    mate[v] = u;
    flip(u, kRsvd ^ kMchd);
    flip(v, kRsvd ^ kMchd);
  }
  __device__ __forceinline__ bool cas(uint32_t v, uint32_t expect, uint32_t desired, uint32_t& cur,
                                      const SweepParams& P) const {
    const uint32_t a = at(v), sh = shift(v);
    for (uint64_t tries = 0;; ++tries) {
      if (((cur >> sh) & kMask) != expect) return false;
      const uint32_t next = (cur & ~(kMask << sh)) | (desired << sh);
      uint32_t old;
      asm volatile("atom.relaxed.cta.shared::cta.cas.b32 %0, [%1], %2, %3;"
                   : "=r"(old)
                   : "r"(a), "r"(cur), "r"(next)
                   : "memory");
      if (old == cur) {
        cur = next;
        return true;
      }
      cur = old;
      if (tries > P.spin_limit) {
        report(P.err, P.host_err, kErrTimeout);
        return false;
      }
    }
  }
  __device__ __forceinline__ bool try_reserve(uint32_t u, uint32_t& ru, const SweepParams& P) const {
    return cas(u, kAcc, kRsvd, ru, P);
  }
  __device__ __forceinline__ bool try_claim(uint32_t v, uint32_t, uint32_t& rv, const SweepParams& P) const {
    return cas(v, kAcc, kMchd, rv, P);
  }
  __device__ __forceinline__ void flip(uint32_t v, uint32_t bits) const {
    asm volatile("red.relaxed.cta.shared::cta.xor.b32 [%0], %1;" ::"r"(at(v)), "r"(bits << shift(v)) : "memory");
  }
  __device__ __forceinline__ void commit(uint32_t u, uint32_t v) const {
    mate[u] = v;
    mate[v] = u;
    flip(u, kRsvd ^ kMchd);
  }
  __device__ __forceinline__ void release(uint32_t u) const { flip(u, kRsvd ^ kAcc); }
};

struct ChipShared {
  uint32_t next;              // next window
  uint32_t nlong;
  uint32_t longs[kMaxLong];   // windows put aside
};

extern __shared__ __align__(16) uint32_t g_chip_words[];

// The whole pass over one graph (the view P: n vertices, row ends from
// P.offsets[0], mates from P.mate[0]) by the calling block.
template <int kBits, bool kSym>
__device__ __forceinline__ void chip_graph(const SweepParams& P, ChipShared& sh, const uint64_t pol) {
  using S = ChipState<kBits>;
  const unsigned lane = threadIdx.x & 31u;
  const uint32_t n = (uint32_t)P.n, words = (uint32_t)packed_words(n, kBits);
  for (uint32_t i = threadIdx.x; i < words; i += blockDim.x) g_chip_words[i] = 0u;
  if (threadIdx.x == 0) sh.next = sh.nlong = 0;
  __syncthreads();
  const S s{smem_u32(g_chip_words), P.mate};
  const uint32_t windows = (n + 31) / 32;
  for (;;) {
    uint32_t w = 0;
    if (lane == 0) w = atomicAdd(&sh.next, 1u);
    w = __shfl_sync(kFull, w, 0);
    if (w >= windows) break;
    const uint32_t r0 = 32 * w, r1 = r0 + 32 < n ? r0 + 32 : n;
    const int64_t e0 = row_end(P.offsets, r0, P.nnz), e1 = row_end(P.offsets, r1, P.nnz);
    if (e1 - e0 > kLongWindow) {
      uint32_t k = 0;
      if (lane == 0) k = atomicAdd(&sh.nlong, 1u);
      k = __shfl_sync(kFull, k, 0);
      if (k < kMaxLong) {
        if (lane == 0) sh.longs[k] = w;
        continue;
      }
    }
    if (e0 < e1) sweep_unit<S, false, kSym>(s, P, r0, e0, e1, lane, pol);
  }
  __syncthreads();
  const uint32_t nlong = sh.nlong < kMaxLong ? sh.nlong : kMaxLong;
  for (uint32_t k = 0; k < nlong; ++k) {
    const uint32_t r0 = 32 * sh.longs[k], r1 = r0 + 32 < n ? r0 + 32 : n;
    const int64_t e1 = row_end(P.offsets, r1, P.nnz);
    for (int64_t e = row_end(P.offsets, r0, P.nnz) + kPiece * (threadIdx.x >> 5); e < e1; e += kPiece * (blockDim.x >> 5))
      sweep_unit<S, false, kSym>(s, P, r0, e, e + kPiece < e1 ? e + kPiece : e1, lane, pol);
  }
  if (nlong) __syncthreads();
  for (uint32_t v = threadIdx.x; v < n; v += blockDim.x)
    if (!S::matched(lds(s.at(v)), v)) P.mate[v] = kNone;
}

// One graph, one launch.  P.state (packed layouts) receives the states as the
// sweep would have left them.
template <int kBits, bool kSym>
__global__ void __launch_bounds__(kSingleThreads, 1) chip_single_kernel(SweepParams P) {
  __shared__ ChipShared sh;
  if (threadIdx.x == 0) *P.err = 0u;
  for (uint64_t i = threadIdx.x; P.tiles && i < P.tile_words; i += blockDim.x) P.tiles[i] = 0ull;
  chip_graph<kBits, kSym>(P, sh, policy_evict_first());
  if (P.state != P.mate) {
    const uint32_t words = (uint32_t)packed_words(P.n, kBits);
    for (uint32_t i = threadIdx.x; i < words; i += blockDim.x) P.state[i] = g_chip_words[i];
  }
}

}  // namespace

cudaError_t launch_chip_single(const SweepParams& P, int bits, cudaStream_t s) {
  const int layout = bits == 2 ? 2 : 8;  // word states are the mates themselves: bytes on the chip
  const size_t bytes = 4 * (packed_words(P.n, layout) + 4);
  static_assert(kChipSingleItems + 16 <= (40u << 10), "the states of the largest graph fit without opting in to more");
  void (*const kernel)(SweepParams) =
      layout == 2 ? (P.sym ? chip_single_kernel<2, true> : chip_single_kernel<2, false>)
                  : (P.sym ? chip_single_kernel<8, true> : chip_single_kernel<8, false>);
  kernel<<<1, kSingleThreads, bytes, s>>>(P);
  return cudaGetLastError();
}

}  // namespace skp
