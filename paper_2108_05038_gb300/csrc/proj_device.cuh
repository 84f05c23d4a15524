// Device helpers shared by the projected DFS (proj_kernels.cu) and its small-subtree form (proj_sub.cu).
#pragma once

#include "fim_internal.cuh"

namespace fim {
namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr uint64_t kNotProjected = ~0ull;
constexpr uint32_t kGroupWords = 4;      // bitmap words (128 transactions) that a warp gathers together
constexpr uint32_t kIdentity = 0xffffffffu;  // row list: every row of the region, in order
constexpr uint32_t kNoop = 0xffffffffu;  // queue item that carries no work (its region did not fit)

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Exclusive block-wide scan.  tmp: 33 shared elements; tmp[32] receives the
// block total.  Two barriers inside; the caller barriers before reusing tmp.
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T* tmp) {
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  T x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(kFull, x, o);
    if (lane >= (uint32_t)o) x += y;
  }
  if (lane == 31) tmp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const T w = lane < nw ? tmp[lane] : T(0);
    T wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T y = __shfl_up_sync(kFull, wi, o);
      if (lane >= (uint32_t)o) wi += y;
    }
    if (lane < nw) tmp[lane] = wi - w;
    if (lane == 31) tmp[32] = wi;
  }
  __syncthreads();
  return tmp[warp] + x - v;
}

__host__ __device__ inline uint32_t words_of(uint32_t supp) { return (supp + 31) / 32; }
__host__ __device__ inline uint32_t padded_words(uint32_t supp) { return (words_of(supp) + 3) & ~3u; }

__device__ __forceinline__ uint32_t ld_volatile(const uint32_t* a) { return *(volatile const uint32_t*)a; }

struct RegionView {
  const uint32_t* R;     // header
  const uint32_t* rids;  // item id of each row
  const uint32_t* Y;     // rows
  uint32_t k, Wp, xlen, W, cls;
};

__device__ __forceinline__ RegionView region_view(const uint32_t* R) {
  RegionView v;
  v.R = R;
  v.k = R[0];
  v.Wp = R[1];
  v.xlen = R[2];
  v.W = R[3];
  v.cls = R[4];
  v.rids = R + 8 + ((v.xlen + 3) & ~3u);
  v.Y = R + region_rows_off(v.xlen, v.k);
  return v;
}

constexpr unsigned long long kPhaseIdleNs = 2000000000ull;

// The end of a phase whose `total` units the warps of the grid claim one after the other: the CTA adds the units that it has
// finished (mine: this warp's, given by lane 0) to *done and waits until all are.  False when the kernel is to end: an error
// in `stop` was set, or the wait ran out (no unit finished, claimed (*head) or reported alive (*progress) for 2 s:
// DEV_ERR_TIMEOUT).
// A CTA waits only for units that running CTAs have claimed, and these finish them without waiting, so the CTAs that are
// resident get through the phases however few they are, and one that starts late goes past what is over.  That is why
// these kernels need no cooperative launch, which starts only when all its CTAs fit and so waits for the longest kernel on
// any other stream (three threads of steps on 100 items beside another thread's mines of 60 ms: 57 ms a step with
// cooperative launches).
// s_done is 0 on entry and on return.  meanwhile(): called by thread 0 once the units are added (claims ahead of that fence
// would hold them back).
template <typename F>
__device__ inline bool phase_wait(uint32_t mine, uint32_t* done, uint32_t total, const uint32_t* head, const uint32_t* progress,
                                  uint32_t* err, uint32_t stop, uint32_t* s_done, F&& meanwhile) {
  __shared__ uint32_t s_ok;
  if ((threadIdx.x & 31) == 0 && mine) atomicAdd(s_done, mine);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (*s_done) atomicAdd(done, *s_done);
    *s_done = 0;
    meanwhile();
    uint32_t ok = 1, seen = kFull, taken = kFull, alive = kFull;
    unsigned long long t0 = 0;
    for (uint32_t poll = 0;; ++poll) {
      const uint32_t a = ld_volatile(done);
      if (a >= total) break;
      if (poll < 32) continue;  // (a microsecond or two: levels are short)
      __nanosleep(40);
      if (poll & 15u) continue;
      if (ld_volatile(err) & (stop | DEV_ERR_TIMEOUT)) {
        ok = 0;
        break;
      }
      const uint32_t h = ld_volatile(head), g = ld_volatile(progress);
      const unsigned long long now = global_ns();
      if (a != seen || h != taken || g != alive) {
        seen = a;
        taken = h;
        alive = g;
        t0 = now;
      } else if (now - t0 > kPhaseIdleNs) {
        atomicOr(err, DEV_ERR_TIMEOUT);
        ok = 0;
        break;
      }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

}  // namespace
}  // namespace fim
