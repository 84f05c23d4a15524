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

constexpr unsigned long long kBarrierIdleNs = 2000000000ull;

// All CTAs of a cooperative grid meet (epoch: barriers passed so far); false when the wait ran out: no CTA arrived and
// *progress did not change for 2 s, or another CTA gave up.
__device__ inline bool grid_barrier(uint32_t* arrived, const uint32_t* progress, uint32_t* err, uint32_t& epoch) {
  __shared__ uint32_t s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(arrived, 1u);
    const uint32_t want = (epoch + 1) * gridDim.x;
    uint32_t ok = 1, seen = kFull, taken = kFull;
    unsigned long long t0 = 0;
    for (uint32_t poll = 0;; ++poll) {
      const uint32_t a = ld_volatile(arrived);
      if (a >= want) break;
      if (poll < 32) continue;  // (a microsecond or two: levels are short)
      __nanosleep(40);
      if (poll & 15u) continue;
      if (ld_volatile(err) & DEV_ERR_TIMEOUT) {
        ok = 0;
        break;
      }
      const uint32_t h = ld_volatile(progress);
      const unsigned long long now = global_ns();
      if (a != seen || h != taken) {
        seen = a;
        taken = h;
        t0 = now;
      } else if (now - t0 > kBarrierIdleNs) {
        atomicOr(err, DEV_ERR_TIMEOUT);
        ok = 0;
        break;
      }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  ++epoch;
  return s_ok != 0;
}

}  // namespace
}  // namespace fim
