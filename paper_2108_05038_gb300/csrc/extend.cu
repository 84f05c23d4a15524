// Supports of the one-item extensions of an itemset: the AND + popcount step of
// a class node (App. B.3.2, Eclat-DFS-Computation: |t(P u {a_j})| from t(P) and
// t({a_j})) as a standalone query.  t(P) is the AND of the rows of P's items
// (one row: used in place); every candidate row is streamed once against it, read
// only under nonzero words of t(P).  With a dense t(P) this is a pure stream of
// the candidate rows, the bandwidth-bound form of the DFS's counting step.
#include <algorithm>
#include <cstring>
#include <vector>

#include "fim_internal.cuh"

namespace fim {
namespace {

__device__ __forceinline__ bool nz4(const uint4& v) { return (v.x | v.y | v.z | v.w) != 0u; }

// Prefixes of at most kExtInline rows are ANDed word by word inside the counting kernel while the extra rows' reads (from
// the L2) stay below kExtInlineBytes over all candidates, about 10 us; else t(P) is built once.
constexpr uint32_t kExtInline = 8;
constexpr uint64_t kExtInlineBytes = 64ull << 20;

// dst[w] = AND of rows[0..n) at word w (the row list in the host's memory: each CTA reads it once, 256 rows at a time)
__global__ void __launch_bounds__(256) k_and_rows(const uint4* __restrict__ bits4, uint32_t stride4, const uint32_t* rows,
                                                  uint32_t n, uint4* dst) {
  __shared__ uint32_t s_rows[256];
  for (uint32_t k0 = 0; k0 < n; k0 += 256) {
    const uint32_t m = min(256u, n - k0);
    __syncthreads();
    if (threadIdx.x < m) s_rows[threadIdx.x] = rows[k0 + threadIdx.x];
    __syncthreads();
    for (uint32_t w = blockIdx.x * blockDim.x + threadIdx.x; w < stride4; w += gridDim.x * blockDim.x) {
      uint4 a = k0 ? dst[w] : make_uint4(~0u, ~0u, ~0u, ~0u);
      for (uint32_t k = 0; k < m && nz4(a); ++k) {
        const uint4 b = __ldg(bits4 + (size_t)s_rows[k] * stride4 + w);
        a = make_uint4(a.x & b.x, a.y & b.y, a.z & b.z, a.w & b.w);
      }
      dst[w] = a;
    }
  }
}

// out[c] = popc(row(pre[0]) & .. & row(pre[n_pre - 1]) & row(cand[c])), or, with t(P) given (pre4), popc(t(P) & row(cand[c])).
// kS warps of a CTA share a candidate, eight 16-byte loads per lane in flight; a candidate whose row is absent (kNoRow)
// has no common transaction with anything.  The row lists are read from, and the counts written to, the host's pinned
// memory: a call is one kernel, without the copies that moving them took and without a kernel for a short prefix (1,000
// candidates of 12.5 KB, two prefix items: 35 us a call before, 22 now).  Bound by HBM once the rows exceed the L2: every
// candidate's warps run at once, so that no last round of a few candidates leaves most of the chip idle (4,001 rows of
// 125 KB: 102 us a call, 117 with a CTA per candidate and 4.4 rounds).
constexpr uint32_t kNoRow = 0xffffffffu;
constexpr uint32_t kExtThreads = 256, kExtWarps = kExtThreads / 32;
template <uint32_t kS>
__global__ void __launch_bounds__(kExtThreads) k_extension_counts(const uint4* __restrict__ bits4, uint32_t stride4,
                                                                  const uint4* __restrict__ pre4, const uint32_t* pre,
                                                                  uint32_t n_pre, const uint32_t* cand, uint32_t n_cand,
                                                                  uint32_t* out) {
  __shared__ uint32_t wsum[kExtWarps];
  __shared__ uint32_t s_pre[kExtInline];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, part = warp % kS;
  if (!pre4 && threadIdx.x < n_pre) s_pre[threadIdx.x] = pre[threadIdx.x];
  __syncthreads();
  for (uint32_t c0 = blockIdx.x * (kExtWarps / kS); c0 < n_cand; c0 += gridDim.x * (kExtWarps / kS)) {
    const uint32_t c = c0 + warp / kS;
    const uint32_t row = c < n_cand ? cand[c] : kNoRow;
    uint32_t s = 0;
    if (row != kNoRow) {
      const uint4* r4 = bits4 + (size_t)row * stride4;
      const uint4* p4 = pre4 ? pre4 : bits4 + (size_t)s_pre[0] * stride4;
      constexpr uint32_t U = 8;
      for (uint32_t w0 = part * 32 + lane; w0 < stride4; w0 += U * kS * 32) {
        uint4 a[U], b[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
          const uint32_t w = w0 + u * kS * 32;
          a[u] = w < stride4 ? __ldg(p4 + w) : make_uint4(0u, 0u, 0u, 0u);
        }
        if (!pre4)
          for (uint32_t t = 1; t < n_pre; ++t) {
            const uint4* q4 = bits4 + (size_t)s_pre[t] * stride4;
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) {
              const uint4 x = nz4(a[u]) ? __ldg(q4 + w0 + u * kS * 32) : make_uint4(0u, 0u, 0u, 0u);
              a[u] = make_uint4(a[u].x & x.x, a[u].y & x.y, a[u].z & x.z, a[u].w & x.w);
            }
          }
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) b[u] = nz4(a[u]) ? __ldcs(r4 + w0 + u * kS * 32) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (uint32_t u = 0; u < U; ++u)
          s += __popc(a[u].x & b[u].x) + __popc(a[u].y & b[u].y) + __popc(a[u].z & b[u].z) + __popc(a[u].w & b[u].w);
      }
    }
    s = __reduce_add_sync(0xffffffffu, s);
    if (kS == 1) {
      if (lane == 0 && c < n_cand) out[c] = s;
    } else {
      if (lane == 0) wsum[warp] = s;
      __syncthreads();
      if (lane == 0 && part == 0 && c < n_cand) {
        uint32_t t = 0;
#pragma unroll
        for (uint32_t k = 0; k < kS; ++k) t += wsum[warp + k];
        out[c] = t;
      }
      __syncthreads();
    }
  }
}

template <uint32_t kS>
cudaError_t launch_counts(const uint4* bits4, uint32_t stride4, const uint4* pre4, const uint32_t* pre, uint32_t n_pre,
                          const uint32_t* cand, uint32_t n_cand, uint32_t* out, uint32_t ctas, cudaStream_t st) {
  const uint32_t per = kExtWarps / kS, need = (n_cand + per - 1) / per;
  k_extension_counts<kS><<<std::min(need, ctas), kExtThreads, 0, st>>>(bits4, stride4, pre4, pre, n_pre, cand, n_cand, out);
  note_launch();
  return cudaGetLastError();
}

// resident CTAs per SM of the counting kernel (its forms differ in the reduction alone), asked once
uint32_t ext_ctas_per_sm() {
  static const int occ = [] {
    int o = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_extension_counts<8>, (int)kExtThreads, 0) != cudaSuccess) o = 1;
    return std::max(1, o);
  }();
  return (uint32_t)occ;
}

}  // namespace
}  // namespace fim

using namespace fim;

extern "C" {

fim_status fim_extension_supports(fim_db* db, const uint32_t* prefix_items, uint32_t n_prefix,
                                  const uint32_t* cand_items, uint32_t n_cand, uint32_t* supports_out) {
  if (!db) return fail(FIM_ERR_INVALID, "db is NULL");
  if (n_prefix == 0 || !prefix_items) return fail(FIM_ERR_INVALID, "the prefix needs at least one item");
  if (n_cand == 0) return FIM_OK;
  if (!cand_items || !supports_out) return fail(FIM_ERR_INVALID, "candidates or supports_out is NULL");
  // items -> rows; an item dropped by the prefilter has no row, so its supports are unknown
  auto row_of = [&](uint32_t item, uint32_t* row) -> fim_status {
    if (item >= db->N) return fail(FIM_ERR_INVALID, "an item id is >= N");
    const int32_t r = db->item_rank[item];
    if (r < 0) return fail(FIM_ERR_INVALID, "an item was dropped by the build's prefilter");
    *row = (uint32_t)r;
    return FIM_OK;
  };
  std::vector<uint32_t> rows(n_prefix + n_cand);
  for (uint32_t k = 0; k < n_prefix; ++k) FIM_TRY(row_of(prefix_items[k], &rows[k]));
  for (uint32_t k = 0; k < n_cand; ++k) FIM_TRY(row_of(cand_items[k], &rows[n_prefix + k]));
  cudaStream_t st = db->stream;
  const uint32_t stride4 = db->stride / 4;
  const uint4* bits4 = reinterpret_cast<const uint4*>(db->d_bits);
  // rows, then the counts, in the pinned staging buffer, which the kernels read and write in place
  void* h = nullptr;
  FIM_TRY(stage_get(db, (rows.size() + n_cand) * 4, &h));
  uint32_t* const h_rows = static_cast<uint32_t*>(h);
  uint32_t* const h_out = h_rows + rows.size();
  std::memcpy(h_rows, rows.data(), rows.size() * 4);
  const uint4* pre4 = nullptr;
  if (n_prefix == 1) {
    pre4 = bits4 + (size_t)rows[0] * stride4;
  } else if (n_prefix > kExtInline || (uint64_t)n_cand * stride4 * 16 * (n_prefix - 1) > kExtInlineBytes) {
    uint4* d_pre = nullptr;
    FIM_TRY(ws_get(db->ws, WS_QUERY_PREFIX, stride4, &d_pre));
    const uint32_t threads = 256;
    const uint32_t grid = std::min<uint32_t>((stride4 + threads - 1) / threads, (uint32_t)db->num_sms * 8);
    k_and_rows<<<std::max<uint32_t>(1, grid), threads, 0, st>>>(bits4, stride4, h_rows, n_prefix, d_pre);
    note_launch();
    FIM_CUDA(cudaGetLastError());
    pre4 = d_pre;
  }
  // warps per candidate: as many as still let every candidate's warps be resident at once; more candidates than
  // that are taken eight warps at a time, so that the last round is short
  const uint32_t ctas = (uint32_t)db->num_sms * ext_ctas_per_sm();
  const uint64_t slots = (uint64_t)ctas * kExtWarps;
  const uint32_t* const c = h_rows + n_prefix;
  if (n_cand > slots || 8ull * n_cand <= slots)
    FIM_CUDA(launch_counts<8>(bits4, stride4, pre4, h_rows, n_prefix, c, n_cand, h_out, ctas, st));
  else if (4ull * n_cand <= slots)
    FIM_CUDA(launch_counts<4>(bits4, stride4, pre4, h_rows, n_prefix, c, n_cand, h_out, ctas, st));
  else if (2ull * n_cand <= slots)
    FIM_CUDA(launch_counts<2>(bits4, stride4, pre4, h_rows, n_prefix, c, n_cand, h_out, ctas, st));
  else
    FIM_CUDA(launch_counts<1>(bits4, stride4, pre4, h_rows, n_prefix, c, n_cand, h_out, ctas, st));
  FIM_TRY(stream_sync(db));
  std::memcpy(supports_out, h_out, (size_t)n_cand * 4);
  return FIM_OK;
}

}  // extern "C"
