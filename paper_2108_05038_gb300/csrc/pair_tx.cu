// K5 from the transactions: level-2 supports counted by walking the horizontal
// database instead of the bitmap rows.
//
// supp({a,b}) is the number of transactions that hold both items (Ch. 2), so the
// supports of all pairs are one pass over the transactions that adds 1 to the
// counter of every pair of frequent items of each transaction.  That costs one
// addition per (transaction, pair in it), sum_t k_t (k_t - 1) / 2 in all, where
// the bitmap forms cost n1 (n1 - 1) / 2 x D bit pairs whatever the transactions
// hold: on sparse data the transactions hold few of the pairs (large_sparse: 181 M
// additions for 7.7 M pairs x 1 M transactions).
//
// The counters are C2[i * n1 + j] (i < j, frequent-row indices) in device memory,
// resident in L2, and the additions are reductions without a return value.  Two
// things bound them on GB300: the L2's rate for scattered 32-bit reductions, about
// 180 G/s (300,000 transactions with 16.8 M pairs of uniform items: 93 us), and the
// reductions that fall on few lines: with large_sparse's Zipf items, 181 M of them
// run at 96 G/s (1.88 ms) because the pairs of its most frequent items take up to
// 760,000 additions each.  Those rows are dense bitmaps, where the tensor-core product
// is at its best, so the pairs with one of the last (most frequent) kTxDenseRows rows
// are left to it (launch_pair_mma_fused on that block of columns) and this kernel drops
// those items while it reads: 17.5 M additions remain.
//
// A warp takes a group of consecutive transactions (or draws of the estimate's
// sample): the lanes hold the group's offsets, the items of transaction u + 2 are
// in flight while those of u + 1 are mapped to rows and the pairs of u are added, so
// no transaction waits for its own loads.  The kept rows of a transaction are
// compacted to k entries of shared memory, written twice in a row, and lane l adds
// the pairs (l, l + d) for d = 1 .. k / 2: every pair once, all k lanes busy.
#include <algorithm>

#include "fim_internal.cuh"

namespace fim {
namespace {

constexpr uint32_t kFull = 0xffffffffu;
constexpr uint32_t kTxThreads = 512;
constexpr uint32_t kTxCtasPerSm = 4;
constexpr uint32_t kNoItem = 0xffffffffu;

__device__ __forceinline__ void add_pair(uint32_t* C2, uint32_t n1, uint32_t a, uint32_t b) {
  atomicAdd(C2 + (size_t)min(a, b) * n1 + max(a, b), 1u);
}

__global__ void __launch_bounds__(kTxThreads, kTxCtasPerSm) k_pair_tx(const TxPairs p, const uint32_t n1, const uint32_t lim, const uint32_t group, uint32_t* __restrict__ C2) {
  __shared__ uint32_t s_rows[kTxThreads / 32][64];
  const uint32_t lane = threadIdx.x & 31;
  uint32_t* const rows = s_rows[threadIdx.x >> 5];
  const uint32_t warps = gridDim.x * (kTxThreads / 32);
  // row index of an item among the rows that take part, or a value >= lim
  auto row_of = [&](uint32_t it) { return it != kNoItem ? (uint32_t)(__ldg(p.map + it) - p.base) : kFull; };
  for (uint64_t t0 = (uint64_t)(blockIdx.x * (kTxThreads / 32) + (threadIdx.x >> 5)) * group; t0 < p.n;
       t0 += (uint64_t)warps * group) {
    const uint32_t nt = min(group, (uint32_t)(p.n - t0));
    uint32_t tb = 0, tl = 0;
    if (lane < nt) {
      const uint32_t t = p.sample ? sample_draw(p.seed, t0 + lane, p.D) : (uint32_t)t0 + lane;
      tb = __ldg(p.off + t);
      tl = __ldg(p.off + t + 1) - tb;
    }
    auto item_of = [&](uint32_t u) {  // (u up to nt + 1: lanes past the group hold length 0)
      const uint32_t b = __shfl_sync(kFull, tb, u & 31), n = __shfl_sync(kFull, tl, u & 31);
      return u < nt && lane < n ? __ldg(p.items + b + lane) : kNoItem;
    };
    uint32_t f = row_of(item_of(0)), it1 = item_of(1);
    for (uint32_t u = 0; u < nt; ++u) {
      const uint32_t it2 = item_of(u + 2);
      const uint32_t f1 = row_of(it1);
      const bool keep = f < lim;
      const uint32_t bal = __ballot_sync(kFull, keep), k = __popc(bal);
      const uint32_t len = __shfl_sync(kFull, tl, u);
      if (len > 32) {
        // a long transaction, 32 items at a time: the pairs inside each chunk, and with every later chunk
        const uint32_t b = __shfl_sync(kFull, tb, u);
        for (uint32_t c0 = 0; c0 < len; c0 += 32) {
          const uint32_t fa = c0 + lane < len ? row_of(__ldg(p.items + b + c0 + lane)) : kFull;
          for (uint32_t c1 = c0; c1 < len; c1 += 32) {
            const uint32_t fb = c1 == c0 ? fa : (c1 + lane < len ? row_of(__ldg(p.items + b + c1 + lane)) : kFull);
            for (uint32_t m = __ballot_sync(kFull, fb < lim); m; m &= m - 1) {
              const uint32_t s = __ffs(m) - 1;
              const uint32_t g = __shfl_sync(kFull, fb, s);
              if (fa < lim && (c1 != c0 || lane < s)) add_pair(C2, n1, fa, g);
            }
          }
        }
      } else if (k >= 2) {
        const uint32_t pos = __popc(bal & ((1u << lane) - 1u));
        if (keep) rows[pos] = rows[pos + k] = f;
        __syncwarp();
        const uint32_t fa = rows[lane];
        const uint32_t half = (k - 1) / 2;  // distances at which every lane has a pair of its own
        if (lane < k) {
          for (uint32_t d = 1; d <= half; ++d) add_pair(C2, n1, fa, rows[lane + d]);
          if ((k & 1u) == 0 && lane < k / 2) add_pair(C2, n1, fa, rows[lane + k / 2]);
        }
        __syncwarp();
      }
      f = f1;
      it1 = it2;
    }
  }
}

// map[item] = index of the item's row among frows (ascending), or -1: the rows of a mine that are not
// consecutive (an estimate's sample)
__global__ void k_tx_map(const int32_t* __restrict__ item_rank, uint32_t N, const uint32_t* __restrict__ frows,
                         uint32_t n1, int32_t* __restrict__ map) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    const int32_t r = item_rank[i];
    uint32_t lo = 0, hi = n1;  // first index with frows >= r
    while (r >= 0 && lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (__ldg(frows + mid) < (uint32_t)r) lo = mid + 1;
      else hi = mid;
    }
    map[i] = r >= 0 && lo < n1 && __ldg(frows + lo) == (uint32_t)r ? (int32_t)lo : -1;
  }
}

}  // namespace

// Modelled time.  Reading and mapping: 0.06 ns per transaction and 3.5 ps per item (large_sparse: 0.13 ms); the
// additions 180 G/s, half of the shorter of the two hidden behind the longer; the additions to the fullest 128-byte
// line of counters, which the L2 takes one after the other, 0.7 ns each.  The number of additions is that of
// the transactions' pairs of any items (known from the build), times the square of the share of item occurrences
// that the rows hold; a row's line is taken as full as independent items would make it (measured against the
// model on GB300: 0.3 M transactions of uniform items 97 us of 102; Zipf items, 1 M transactions all rows 2.07 ms
// of 2.0, all but 256 rows 0.15 ms of 0.19; 0.07 M transactions all rows 0.143 ms of 0.145).
double pair_tx_cost_us(const fim_db* db, const TxPairs& p, const uint32_t* frows, uint32_t r0, uint32_t n1,
                       uint32_t lim) {
  if (db->tx_distinct == 0) return 1e300;
  const double scale = (double)p.n / db->D, all = (double)db->tx_distinct;
  double kept = 0.0, hot = 0.0, top = 0.0;
  for (uint32_t k = lim; k-- > 0;) {
    const double s = db->supp[frows ? frows[k] : r0 + k];
    kept += s;
    hot = std::max(hot, s * top / db->D);  // row k against the (at most 32) last rows after it
    if (lim - k <= 32) top += s;
  }
  const double share = kept / all;
  const double add_us = (double)db->tx_pairs * scale * share * share / 180e3;
  const double read_us = ((double)p.n * 0.06 + all * scale * 0.0035) * 1e-3;
  return 5.0 + std::max(add_us, read_us) + 0.5 * std::min(add_us, read_us) + hot * scale * 0.7e-3 +
         (double)n1 * n1 * 4 / 5e6;  // (clearing the counters)
}

cudaError_t launch_tx_map(const int32_t* item_rank, uint32_t N, const uint32_t* frows, uint32_t n1, int32_t* map,
                          cudaStream_t st) {
  k_tx_map<<<std::min<uint32_t>((N + 255) / 256, 1024), 256, 0, st>>>(item_rank, N, frows, n1, map);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_pair_tx(const TxPairs& p, uint32_t n1, uint32_t lim, uint32_t* C2, int num_sms, cudaStream_t st) {
  if (p.n == 0) return cudaSuccess;
  const uint64_t warps = (uint64_t)num_sms * kTxCtasPerSm * (kTxThreads / 32);
  // up to 32 transactions per group, fewer when that would leave warps without one
  const uint32_t group = (uint32_t)std::min<uint64_t>(32, std::max<uint64_t>(1, p.n / warps));
  const uint64_t ctas = ((p.n + group - 1) / group + kTxThreads / 32 - 1) / (kTxThreads / 32);
  k_pair_tx<<<(uint32_t)std::min<uint64_t>(ctas, (uint64_t)num_sms * kTxCtasPerSm), kTxThreads, 0, st>>>(p, n1, lim,
                                                                                                       group, C2);
  note_launch();
  return cudaGetLastError();
}

}  // namespace fim
