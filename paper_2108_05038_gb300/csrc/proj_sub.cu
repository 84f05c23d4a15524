// K4, projected mode, small subtrees: Eclat on database parts that fit the
// shared memory of one warp.
//
// The walk of k_dfs_proj expands one class node at a time: a node with its 3.6
// candidates (large_sparse, 700,000 nodes) costs about 1,070 warp instructions, most
// of them per node and not per word.  Most nodes, though, lie below a two-item
// prefix X whose database part (its n survivors' bitmaps over t(X), ceil(supp(X) / 32)
// words each) is a few KB: of large_sparse's 300,000 frames with two or more survivors
// 95% have at most 128 words and none more than 31 survivors.  So k_sub walks subtrees in
// shared memory, and counts supports many pairs at a time.  It works in rounds:
//
//   pairs   the supports of all pairs of a part's candidate rows (round 0: the rows of every
//           class region, i.e. the candidates of all its two-item classes, the first step
//           of Phase 4): a warp takes 8 x 8 rows and up to 512 words, lanes over words, 64
//           running counts, so every word read serves eight pairs.
//   walk    one warp per extension X of a part by one of its rows: X's survivors are read off
//           the pair supports; when their database part fits, it is built in shared memory (gather
//           and ballot) and the whole subtree is walked there a frame at a time: the frame's
//           prefix is the AND of a few rows, the supports of all its survivor pairs are counted
//           together, a lane (or a group of lanes) per pair, and children of two survivors, half
//           of all frames, are counted with their parent.  Itemsets are sets of rows, i.e. masks,
//           kept in a small buffer and written up to 64 at a time behind one reservation.  A part
//           that does not fit goes to the next round with its candidates (and the class region's
//           rows, masked by the prefix), and so does what is left of a subtree that has taken
//           kSubCycles (without room there it goes to k_dfs_proj): no warp keeps a round waiting for long.
//
// One launch runs all rounds.  The warps claim the units, tiles and items of a phase one after the other, and a CTA goes on
// to the next phase when all are finished (phase_wait; bounded: no progress anywhere for 2 s ends the kernel with
// DEV_ERR_TIMEOUT).
// Whatever finds no room in the queues is left to k_dfs_proj, which takes any frame.  The classes,
// nodes, candidates and records are those of k_dfs_proj.
#include <algorithm>
#include <map>
#include <mutex>
#include <type_traits>

#include "proj_device.cuh"

namespace fim {
namespace {

constexpr uint32_t kSubThreads = 256;
constexpr uint32_t kSubWarps = kSubThreads / 32;
constexpr uint32_t kSubCtasPerSm = 2;
constexpr uint32_t kSubPool = 2576;      // words per warp: rows, prefix, child masks
constexpr uint32_t kSubRows = 32;        // rows of a part held in shared memory (with the prefix ids at most 64)
constexpr uint32_t kUnitWords = 512;      // words of a region that a unit of a part's rows covers
constexpr uint32_t kSubAll = 5;          // at most so many survivors: every subset of them counted in one pass

// words of k_sub's shared memory per warp ahead of the pool
struct SubSmem {
  uint32_t pos[288];              // positions of the prefix's set bits; later todo and survivor masks per depth
                                  // (before both: unsorted ids)
  unsigned long long rec[64];     // itemsets not yet written, as sets of `ids` positions
  uint32_t rsupp[64];             // their supports
  uint32_t ids[64];               // the ids that occur (prefix and rows), ascending
  unsigned long long pids[32];    // prefix of the frame at each depth, as positions in `ids`
  uint32_t path[32];              // the same as a set of the part's rows (the part's own prefix not among them)
  uint32_t lrow[64], lsup[64];    // survivors: row of the region, support
  uint32_t prow[64];              // the part's prefix rows (rows of the region)
  uint8_t at[64];                 // row -> position in ids
  uint8_t idx[32];                // rows of the frame being counted
  uint8_t two[32];                // its children with two survivors
  uint32_t pool[kSubPool];
};
static_assert(sizeof(SubSmem) % 8 == 0, "every warp's block keeps the 64-bit arrays aligned");

__host__ __device__ inline uint32_t gram_row_off(uint32_t m, uint32_t k) { return m * k - m * (m + 1) / 2; }  // of (m, m + 1)

// words of the pool that n rows of W words need: the rows (odd stride), the prefix, the child masks of every depth
__host__ __device__ inline uint32_t sub_pool_words(uint32_t n, uint32_t W) {
  return n * (W | 1u) + W + n * (n + 1) / 2;
}
__device__ __forceinline__ bool sub_fits(uint32_t n, uint32_t xlen, uint32_t W) {
  return n <= kSubRows && n + xlen <= 64 && W <= kSubPool && sub_pool_words(n, W) <= kSubPool;
}

__device__ __forceinline__ uint32_t ld_cg(const uint32_t* a) { return __ldcg(a); }

// ---------------------------------------------------------------------------
// Pair supports of one 8 x 8 tile of a part's rows over words [w0, w1), by one warp, under the part's prefix rows (list:
// prefix rows, then the part's rows; NULL: no prefix, every row of the region): written to G, the triangle of pairs and
// then the rows' own supports (added atomically when the words are split).
__device__ __noinline__ void gram_tile(const RegionView& V, const uint32_t* list, uint32_t path_len, uint32_t n,
                                          uint32_t* G, uint32_t ba, uint32_t bb, uint32_t w0, uint32_t w1, bool split) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t acc[kGramRows][kGramRows];
  uint32_t pa[kGramRows], pb[kGramRows];  // row offsets (a region has fewer than 2^32 words)
#pragma unroll
  for (uint32_t x = 0; x < kGramRows; ++x) {
    const uint32_t r = min(ba * kGramRows + x, n - 1), c = min(bb * kGramRows + x, n - 1);
    pa[x] = (list ? ld_cg(list + path_len + r) : r) * V.Wp;
    pb[x] = (list ? ld_cg(list + path_len + c) : c) * V.Wp;
#pragma unroll
    for (uint32_t y = 0; y < kGramRows; ++y) acc[x][y] = 0;
  }
  for (uint32_t w = w0 + lane; w < w1; w += 32) {
    uint32_t a[kGramRows], b[kGramRows], pre = kFull;
    for (uint32_t t = 0; t < path_len; ++t) pre &= V.Y[(uint64_t)ld_cg(list + t) * V.Wp + w];
#pragma unroll
    for (uint32_t x = 0; x < kGramRows; ++x) {
      a[x] = V.Y[pa[x] + w] & pre;
      b[x] = V.Y[pb[x] + w];
    }
#pragma unroll
    for (uint32_t x = 0; x < kGramRows; ++x)
#pragma unroll
      for (uint32_t y = 0; y < kGramRows; ++y) acc[x][y] += __popc(a[x] & b[y]);
  }
  // the 64 sums over the lanes, two to each lane: at every step a lane keeps one half of its values, sends the other to
  // the lane across and adds what it receives; lane l ends with sums 2 l and 2 l + 1
  uint32_t v[kGramRows * kGramRows];
#pragma unroll
  for (uint32_t x = 0; x < kGramRows * kGramRows; ++x) v[x] = acc[x / kGramRows][x % kGramRows];
#pragma unroll
  for (uint32_t o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (uint32_t i = 0; i < 2 * o; ++i) {
      const uint32_t keep = up ? v[i + 2 * o] : v[i], send = up ? v[i] : v[i + 2 * o];
      v[i] = keep + __shfl_xor_sync(kFull, send, o);
    }
  }
#pragma unroll
  for (uint32_t i = 0; i < 2; ++i) {
    const uint32_t m = ba * kGramRows + lane / 4, e = bb * kGramRows + ((2 * lane + i) & 7u);
    if (m <= e && e < n) {
      uint32_t* g = G + (m < e ? gram_row_off(m, n) + (e - m - 1) : n * (n - 1) / 2 + m);
      if (split) atomicAdd(g, v[i]);
      else *g = v[i];
    }
  }
}

// tile t of the nb (nb + 1) / 2 upper ones -> (ba, bb)
__device__ __forceinline__ void tile_of(uint32_t t, uint32_t& ba, uint32_t& bb) {
  bb = (uint32_t)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
  while (bb * (bb + 1) / 2 > t) --bb;
  while ((bb + 1) * (bb + 2) / 2 <= t) ++bb;
  ba = t - bb * (bb + 1) / 2;
}

// Puts row m' of a region into k_dfs_proj's shared queue.  Without a slot the run is repeated without k_sub.
__device__ __forceinline__ void leave_to_dfs(const SubLaunch& p, uint64_t roff, uint32_t m) {
  const uint32_t slot = atomicAdd(&p.ctrl->dq_tail, 1u);
  if (slot >= p.dq_cap) {
    atomicOr(&p.ctrl->err, DEV_ERR_SUB);
    return;
  }
  atomicAdd(&p.ctrl->proj_pending, 1u);
  p.dq[slot] = make_uint4((uint32_t)roff, (uint32_t)(roff >> 32), m, 1u);
}

// Leaves a frame of the part in S.pool (W words a row) to k_dfs_proj: prefix rows rows_p, prefix ids pid (positions in
// S.ids), two or more survivors rows_s.  Its database part, the survivors' words under the prefix, becomes a region of the
// arena, its extensions items of the shared queue.  False without room in the arena (the run is repeated without k_sub).
__device__ __noinline__ bool leave_subtree(const SubLaunch* pp, SubSmem* Sp, uint32_t rows_p, uint32_t rows_s,
                                           unsigned long long pid, uint32_t W, uint32_t cls) {
  const SubLaunch& p = *pp;
  SubSmem& S = *Sp;
  const uint32_t lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
  const uint32_t ns = __popc(rows_s), plen = __popcll(pid), Ws = W | 1u, Wp = (W + 3) & ~3u;
  const uint64_t rows_off = region_rows_off(plen, ns);
  const unsigned long long size = (rows_off + (unsigned long long)ns * Wp + 31) & ~31ull;
  unsigned long long off = 0;
  if (lane == 0) off = atomicAdd(&p.ctrl->arena_top, size);
  off = __shfl_sync(kFull, off, 0);
  if (off + size > p.arena_words) {
    if (lane == 0) atomicOr(&p.ctrl->err, DEV_ERR_SUB);
    return false;
  }
  uint32_t* const R = p.Y + off;
  if (lane == 0) {
    R[0] = ns;
    R[1] = Wp;
    R[2] = plen;
    R[3] = W;
    R[4] = cls;
    R[5] = kNoGram;
    R[6] = R[7] = 0;
  }
  for (uint32_t q = lane; q < 64; q += 32)
    if ((pid >> q) & 1ull) R[8 + __popcll(pid & ((1ull << q) - 1ull))] = S.ids[q];
  if ((rows_s >> lane) & 1u) R[8 + ((plen + 3) & ~3u) + __popc(rows_s & lt)] = S.ids[S.at[lane]];
  uint32_t* const Y2 = R + rows_off;
  for (uint32_t w = lane; w < Wp; w += 32) {
    uint32_t v = w < W ? kFull : 0u;
    for (uint32_t t = rows_p; t && v; t &= t - 1) v &= S.pool[(__ffs(t) - 1) * Ws + w];
    uint32_t j = 0;
    for (uint32_t t = rows_s; t; t &= t - 1, ++j) Y2[(uint64_t)j * Wp + w] = v ? S.pool[(__ffs(t) - 1) * Ws + w] & v : 0u;
  }
  for (uint32_t t = lane; t + 1 < ns; t += 32) leave_to_dfs(p, off, t);
  return true;
}

constexpr uint32_t kSubStop = DEV_ERR_ABORTED | DEV_ERR_PSTACK | DEV_ERR_TIMEOUT | DEV_ERR_SUB;

// Writes the warp's nrec (1 .. 64) buffered records: one reservation, lane l takes records 2 l and 2 l + 1 (a record's
// items follow those of the record before it).  Returns the items, the longest record and the stop bits of the error
// word.  (Not inlined, and called from several places: k_sub's code would outgrow the instruction cache.)
__device__ __noinline__ uint3 write_records(const SubLaunch* pp, SubSmem* Sp, uint32_t nrec) {
  const SubLaunch& p = *pp;
  SubSmem& S = *Sp;
  const uint32_t lane = threadIdx.x & 31;
  __syncwarp();
  const unsigned long long m0 = 2 * lane < nrec ? S.rec[2 * lane] : 0ull;
  const unsigned long long m1 = 2 * lane + 1 < nrec ? S.rec[2 * lane + 1] : 0ull;
  const uint32_t l0 = __popcll(m0), l1 = __popcll(m1);
  uint32_t x = l0 + l1;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, x, o);
    if (lane >= (uint32_t)o) x += y;
  }
  const uint32_t total = __shfl_sync(kFull, x, 31);
  unsigned long long base = 0;
  uint32_t e = 0;
  if (lane == 0) {
    base = atomicAdd(&p.ctrl->packed, ((unsigned long long)nrec << 32) | total);
    const unsigned long long after = (base >> 32) + nrec;
    e = ld_volatile(&p.ctrl->err);
    if ((p.max_sets && after > p.max_sets) || after > 0xfffffff0ull) {
      atomicOr(&p.ctrl->err, DEV_ERR_ABORTED);
      e |= DEV_ERR_ABORTED;
    }
  }
  base = __shfl_sync(kFull, base, 0);
  e = __shfl_sync(kFull, e, 0);
  uint64_t it = (base & 0xffffffffull) + x - l0 - l1;
  bool over = false;
#pragma unroll 1
  for (uint32_t h = 0; h < 2; ++h) {
    unsigned long long m = h ? m1 : m0;
    const uint64_t rec = (base >> 32) + 2 * lane + h;
    const uint32_t len = h ? l1 : l0;
    if (m) {
      if (rec < p.cap_sets && it + len <= p.cap_items) {
        p.out_off[rec] = it;
        p.out_supp[rec] = S.rsupp[2 * lane + h];
        for (uint32_t* d = p.out_items + it; m; m &= m - 1) *d++ = S.ids[__ffsll(m) - 1];
      } else {
        over = true;
      }
      it += len;
    }
  }
  if (over) atomicOr(&p.ctrl->err, DEV_ERR_OVERFLOW);
  __syncwarp();
  return make_uint3(total, __reduce_max_sync(kFull, max(l0, l1)), e & kSubStop);
}

// dst[j * stride + q] = word q of row lrow[j] (j < n_rows, at most 64) over the transactions that the np_rows rows prow hold
// among words [wb, we) of the region's rows Y (Wp words each); nwords words are written.  256 transactions at a time: their
// positions listed, then for every row the word that holds each position (4 x 8 loads in flight per lane) and a ballot per
// 32 positions.  The order of the transactions is free as long as every row has the same: the lists take one bit of every
// lane that has one left per step, so that no lane lists alone and the 32 positions of a step lie within one line of a row.
__device__ __noinline__ void gather_rows(SubSmem* Sp, const uint32_t* __restrict__ Y, uint32_t Wp, uint32_t np_rows,
                                         uint32_t wb, uint32_t we, uint32_t* dst, uint32_t stride, uint32_t nwords,
                                         uint32_t n_rows) {
  SubSmem& S = *Sp;
  const uint32_t lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
  uint32_t fill = 0, q0 = 0;  // positions listed, first word of the window
  uint32_t nx[4];             // the next 128 words, in flight
  auto fetch = [&](uint32_t w0) {
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      const uint32_t w = w0 + 32 * k + lane;
      nx[k] = w < we ? Y[(uint64_t)S.prow[0] * Wp + w] : 0u;
      for (uint32_t t = 1; t < np_rows; ++t) nx[k] &= w < we ? Y[(uint64_t)S.prow[t] * Wp + w] : 0u;
    }
  };
  __syncwarp();
  fetch(wb);
  for (uint32_t w0 = wb;; w0 += 128) {
    const bool end = w0 >= we;  // (one more round for the last positions)
    uint32_t vs[4];
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) vs[k] = nx[k];
    if (!end) fetch(w0 + 128);
#pragma unroll 1
    for (uint32_t k = 0; k < 4; ++k) {
      uint32_t v = k == 0 ? vs[0] : k == 1 ? vs[1] : k == 2 ? vs[2] : vs[3];
      const uint32_t bit0 = (w0 + 32 * k + lane) * 32 - 1;
      uint32_t more = __ballot_sync(kFull, v != 0u);
      do {
        if (v) S.pos[fill + __popc(more & lt)] = bit0 + __ffs(v);
        v &= v - 1;
        fill += __popc(more);
        more = __ballot_sync(kFull, v != 0u);
        if (fill >= 256 || (end && k == 3 && fill)) {
          __syncwarp();
          uint32_t tid[8];
#pragma unroll
          for (uint32_t r = 0; r < 8; ++r) tid[r] = 32 * r + lane < fill ? S.pos[32 * r + lane] : kFull;
          for (uint32_t j0 = 0; j0 < n_rows; j0 += 4) {
            uint32_t x[4][8];
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
              const uint32_t* rp = Y + (uint64_t)S.lrow[min(j0 + u, n_rows - 1)] * Wp;
#pragma unroll
              for (uint32_t r = 0; r < 8; ++r) x[u][r] = tid[r] != kFull ? rp[tid[r] >> 5] : 0u;
            }
            uint32_t mine = 0;
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u)
#pragma unroll
              for (uint32_t r = 0; r < 8; ++r) {
                const uint32_t y = __ballot_sync(kFull, (x[u][r] >> (tid[r] & 31)) & 1u);
                if (lane == 8 * u + r) mine = y;
              }
            // lane 8 u + r: word r of row j0 + u
            const uint32_t wq = q0 + (lane & 7u);
            if (j0 + (lane >> 3) < n_rows && wq < nwords) dst[(uint64_t)(j0 + (lane >> 3)) * stride + wq] = mine;
          }
          q0 += 8;
          __syncwarp();
          fill = fill > 256 ? fill - 256 : 0;
          if (lane < fill) S.pos[lane] = S.pos[256 + lane];
          __syncwarp();
        }
      } while (more);
    }
    if (end) break;
  }
  __syncwarp();
}

// Count only: adds the pending itemsets to the reservation word, which then feeds nothing but the itemset limit;
// returns the stop bits.
__device__ __noinline__ uint32_t add_counted(const SubLaunch* pp, unsigned long long sets) {
  const SubLaunch& p = *pp;
  uint32_t e = 0;
  if ((threadIdx.x & 31) == 0) {
    e = ld_volatile(&p.ctrl->err);
    if (sets) {
      const unsigned long long after = (atomicAdd(&p.ctrl->packed, sets << 32) >> 32) + sets;
      if ((p.max_sets && after > p.max_sets) || after > 0xfffffff0ull) {
        atomicOr(&p.ctrl->err, DEV_ERR_ABORTED);
        e |= DEV_ERR_ABORTED;
      }
    }
  }
  return __shfl_sync(kFull, e, 0) & kSubStop;
}

__global__ void __launch_bounds__(kSubThreads, kSubCtasPerSm) k_sub(const __grid_constant__ SubLaunch p) {
  extern __shared__ __align__(16) uint8_t smem[];
  const uint32_t lane = threadIdx.x & 31;
  SubSmem& S = reinterpret_cast<SubSmem*>(smem)[threadIdx.x >> 5];
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t nwarps = gridDim.x * kSubWarps;
  __shared__ uint32_t s_done, s_first[2][3];  // of phase_wait; the claims of this round and the next
  unsigned long long st_inter = 0, st_nodes = 0, st_frames = 0, st_bytes = 0, st_sets = 0, st_items = 0;
  uint32_t st_maxlen = 0, st_parts = 0;
  uint32_t nrec = 0;                  // buffered records
  unsigned long long pend_sets = 0;   // count only: itemsets not yet added to the reservation word
  bool stop = false;

  auto flush = [&]() {
    if (nrec == 0) {
      __syncwarp();
      return;
    }
    const uint3 r = write_records(&p, &S, nrec);
    st_sets += nrec;
    st_items += r.x;
    st_maxlen = max(st_maxlen, r.y);
    stop |= r.z != 0;
    nrec = 0;
  };
  // count only: the itemset limit is checked against the running total
  auto flush_count = [&]() {
    stop |= add_counted(&p, pend_sets) != 0;
    pend_sets = 0;
  };

  // A CTA claims the first units, tiles and items of a round, one of each for every warp, before the wait for the round
  // above: no claim is waited for, and no warp gets a second one before each has had one.  The others of a long list are
  // claimed a few at a time.
  const uint32_t wib = threadIdx.x >> 5;
  auto claim_round = [&](uint32_t round) {  // (thread 0)
    SubRound& r = p.state->round[round];
    s_first[round & 1u][0] = round ? atomicAdd(&r.unit_head, kSubWarps) : 0u;
    s_first[round & 1u][1] = atomicAdd(&r.tile_head, kSubWarps);
    s_first[round & 1u][2] = atomicAdd(&r.item_head, kSubWarps);
  };
  // f(t) for the warp's share of 0 .. n - 1; returns how many it took
  auto share = [&](uint32_t first, uint32_t* head, uint32_t n, auto&& f) {
    const uint32_t chunk = max(1u, min(8u, n / (8 * nwarps)));
    uint32_t t0 = first, t1 = t0 + 1, taken = 0, next = 0;
    while (t0 < n) {
      if (lane == 0) next = atomicAdd(head, chunk);
      for (uint32_t t = t0; t < min(t1, n); ++t, ++taken) f(t);
      t0 = __shfl_sync(kFull, next, 0);
      t1 = t0 + chunk;
    }
    return taken;
  };
  auto wait = [&](uint32_t mine, uint32_t* done, uint32_t total, const uint32_t* head, bool claim, uint32_t round) {
    return phase_wait(mine, done, total, head, &p.state->progress, &p.ctrl->err, kSubStop, &s_done, [&] {
      if (claim) claim_round(round + 1);
    });
  };
  if (threadIdx.x == 0) {
    s_done = 0;
    claim_round(0);
  }
  __syncthreads();
  for (uint32_t round = 0;; ++round) {
    // ---------------- pairs ----------------
    const uint32_t par = round & 1u;
    SubRound& now = p.state->round[round];
    SubRound& next_round = p.state->round[round + 1];
    auto within = [](const unsigned long long* n, uint32_t cap) {
      return (uint32_t)min(*(volatile const unsigned long long*)n, (unsigned long long)cap);
    };
    const uint32_t n_tiles = round ? within(&now.tile_n, p.tile_cap) : p.tileoff[p.n1];
    const uint32_t n_items = round ? within(&now.item_n, p.item_cap) : p.ctrl->n_entries_g;
    if (n_items == 0) break;
    // ---------------- rows of the parts that get their own ----------------
    const uint32_t n_units = round ? within(&now.unit_n, p.tile_cap) : 0u;
    const uint32_t my_units = share(s_first[par][0] + wib, &now.unit_head, n_units, [&](uint32_t t) {
      const uint4 d = __ldcg(reinterpret_cast<const uint4*>(p.units + t));
      const uint4 d2 = __ldcg(reinterpret_cast<const uint4*>(p.units + t) + 1);
      if (d.x == kNoop) return;
      const RegionView V = region_view(p.Y + (uint64_t)d.x * 4);
      const uint32_t path_len = d.z & 0xffffu, cnt = d.z >> 16, u = d2.w & 0xffffu;
      __syncwarp();
      for (uint32_t q = lane; q < path_len; q += 32) S.prow[q] = ld_cg(p.lists + d.y + q);
      if (lane < cnt) S.lrow[lane] = ld_cg(p.lists + d.y + path_len + d.w + lane);
      __syncwarp();
      gather_rows(&S, V.Y, V.Wp, path_len, u * kUnitWords, min(V.W, (u + 1) * kUnitWords),
                  p.Y + ((uint64_t)d2.y << 32 | d2.x), d2.z, d2.w >> 16, cnt);
    });
    if (n_units && !wait(my_units, &now.unit_done, n_units, &now.unit_head, false, round)) break;
    const uint32_t my_tiles = share(s_first[par][1] + wib, &now.tile_head, n_tiles, [&](uint32_t t) {
      if (round == 0) {
        uint32_t lo = 0, hi = p.n1;  // the class: the last queue position q with tileoff[q] <= t
        while (hi - lo > 1) {
          const uint32_t mid = (lo + hi) >> 1;
          if (__ldg(p.tileoff + mid) <= t) lo = mid;
          else hi = mid;
        }
        const RegionView V = region_view(p.Y + p.yoff[__ldg(p.row_order + lo)]);
        const uint32_t nb = (V.k + kGramRows - 1) / kGramRows, nt = nb * (nb + 1) / 2;
        const uint32_t local = t - __ldg(p.tileoff + lo), chunk = local / nt;
        uint32_t ba, bb;
        tile_of(local - chunk * nt, ba, bb);
        gram_tile(V, nullptr, 0, V.k, p.G + V.R[5], ba, bb, chunk * kGramWords, min(V.W, (chunk + 1) * kGramWords),
                  V.W > kGramWords);
      } else {
        const uint4 d = __ldcg(reinterpret_cast<const uint4*>(p.tiles + t));
        const uint4 d2 = __ldcg(reinterpret_cast<const uint4*>(p.tiles + t) + 1);
        if (d.x == kNoop) return;
        const RegionView V = region_view(p.Y + (uint64_t)d.x * 4);
        gram_tile(V, d.y == kIdentity ? nullptr : p.lists + d.y, d.z, d.w, p.G + d2.x, d2.y & 0xffffu, d2.y >> 16, d2.z * kGramWords,
                  min(V.W, (d2.z + 1) * kGramWords), V.W > kGramWords);
      }
    });
    if (n_tiles && !wait(my_tiles, &now.tile_done, n_tiles, &now.tile_head, false, round)) break;
    // (the other halves of G, the lists and the items are free: the round before is over)
    const bool last = round + 1 >= p.rounds;
    SubItem* const items = p.items + (uint64_t)par * kSubItemCap;
    SubItem* const next_items = p.items + (uint64_t)(par ^ 1u) * kSubItemCap;
    const uint64_t g_lo = (uint64_t)(par ^ 1u) * (kSubGramCap / 2), l_lo = (uint64_t)(par ^ 1u) * kSubListCap;

    // ---------------- walk ----------------
    uint32_t my_items = 0;
    auto next_item = [&]() {
      uint32_t e = 0;
      if (lane == 0) e = (ld_volatile(&p.ctrl->err) & kSubStop) ? kFull : atomicAdd(&now.item_head, 1u);
      ++my_items;
      return __shfl_sync(kFull, e, 0);
    };
    for (uint32_t e = s_first[par][2] + wib; e < n_items && !stop; e = next_item()) {
      SubItem it;
      if (round) {
        const uint4 d = __ldcg(reinterpret_cast<const uint4*>(items + e));
        const uint4 d2 = __ldcg(reinterpret_cast<const uint4*>(items + e) + 1);
        it = SubItem{d.x, d.y, d.z, d.w, d2.x, d2.y, {0, 0}};
        if (it.roff4 == kNoop) continue;
      } else {
        const uint2 en = p.entries_g[e];
        it = SubItem{(uint32_t)(p.yoff[en.x] / 4), 0, 0, 0, 0, en.y, {0, 0}};
      }
      const RegionView V = region_view(p.Y + (uint64_t)it.roff4 * 4);
      const uint32_t* const list = round && it.list != kIdentity ? p.lists + it.list : nullptr;
      if (!round) {
        it.n = V.k;
        it.goff = V.R[5];
      }
      auto row_of = [&](uint32_t j) { return list ? ld_cg(list + it.path_len + j) : j; };
      const uint32_t cls = V.cls;
      unsigned long long cls_sets = 0, cls_work = 0;
      const bool task = it.m == kSubTask;
      uint32_t n = 0;                       // rows of the part
      const uint32_t np_rows = it.path_len + (task ? 0u : 1u), xlen = V.xlen + np_rows;  // prefix rows, prefix ids
      uint32_t supp = 0;                    // support of the prefix
      __syncwarp();
      for (uint32_t q = lane; q < it.path_len; q += 32) S.prow[q] = ld_cg(list + q);
      if (!task && lane == 0) S.prow[it.path_len] = row_of(it.m);
      // word w of the prefix's bitmap (four at 4-word boundaries)
      auto pre4 = [&](uint32_t w) {
        uint4 v = *reinterpret_cast<const uint4*>(V.Y + (uint64_t)S.prow[0] * V.Wp + w);
        for (uint32_t t = 1; t < np_rows; ++t) {
          const uint4 u = *reinterpret_cast<const uint4*>(V.Y + (uint64_t)S.prow[t] * V.Wp + w);
          v = make_uint4(v.x & u.x, v.y & u.y, v.z & u.z, v.w & u.w);
        }
        return v;
      };
      const uint32_t nc = task ? 0u : it.n - it.m - 1;
      const uint32_t* const g = p.G + it.goff + (task ? 0u : gram_row_off(it.m, it.n));
      if (task) {
        n = it.n;
        for (uint32_t q = lane; q < n; q += 32) S.lrow[q] = row_of(q);
        __syncwarp();
        for (uint32_t w = 4 * lane; w < V.Wp; w += 128) {
          const uint4 v = pre4(w);
          supp += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
        }
        supp = __reduce_add_sync(kFull, supp);
      } else {
        for (uint32_t j0 = 0; j0 < nc; j0 += 32) {
          const uint32_t c = j0 + lane < nc ? ld_cg(g + j0 + lane) : 0u;
          const bool f = c >= p.minsup;  // (minsup >= 1)
          const uint32_t bal = __ballot_sync(kFull, f), at = n + __popc(bal & lt);
          if (f && at < 64) {
            S.lrow[at] = row_of(it.m + 1 + j0 + lane);
            S.lsup[at] = c;
          }
          n += __popc(bal);
        }
        supp = ld_cg(p.G + it.goff + it.n * (it.n - 1) / 2 + it.m);
        __syncwarp();
      }
      uint32_t W = words_of(supp), Ws = W | 1u;
      bool walk = n >= 2;
      const bool small = n + xlen <= 64;
      unsigned long long pre_ids = 0;  // the prefix's positions in ids
      // the ids of the prefix and of the n rows: their ranks, ascending
      if (small && (n || p.leaves)) {
        for (uint32_t q = lane; q < xlen + n; q += 32)
          S.pos[q] = q < V.xlen ? V.R[8 + q] : V.rids[q < xlen ? S.prow[q - V.xlen] : S.lrow[q - xlen]];
        __syncwarp();
        unsigned long long mine = 0;
        for (uint32_t q = lane; q < xlen + n; q += 32) {
          const uint32_t v = S.pos[q];
          uint32_t r = 0;
          for (uint32_t t = 0; t < xlen + n; ++t) r += S.pos[t] < v;
          S.ids[r] = v;
          if (q >= xlen) S.at[q - xlen] = (uint8_t)r;
          else mine |= 1ull << r;
        }
        pre_ids = __reduce_or_sync(kFull, (uint32_t)mine) |
                  (unsigned long long)__reduce_or_sync(kFull, (uint32_t)(mine >> 32)) << 32;
        __syncwarp();
      }
      auto write_prefix = [&](uint32_t* R) {  // the prefix ids, ascending, into a region's header
        auto id_of = [&](uint32_t t) { return t < V.xlen ? V.R[8 + t] : V.rids[S.prow[t - V.xlen]]; };
        for (uint32_t q = lane; q < xlen; q += 32) {
          const uint32_t v = id_of(q);
          uint32_t r = 0;
          for (uint32_t t = 0; t < xlen; ++t) r += id_of(t) < v;
          R[8 + r] = v;
        }
      };
      const bool all = small && n <= kSubAll && !(task && p.leaves);  // (a task's rows come without their supports)
      if (walk && !task && !all && !sub_fits(n, xlen, W)) {
        // not a part for one warp: the next round's (its candidates, their pairs to count, and its extensions)
        uint32_t ok = 0, lo = 0, go = 0;
        unsigned long long ti = 0, ii = 0, ui = 0;
        const uint32_t nb = (n + kGramRows - 1) / kGramRows, nt = nb * (nb + 1) / 2;
        // When X's transactions are few among the region's, the part gets rows of its own over them, built by units of
        // kUnitWords words x 32 rows (every unit's transactions start at a whole word); else it is the region's rows, masked.
        const uint32_t n_units = (V.W + kUnitWords - 1) / kUnitWords, nj = (n + 31) / 32;
        uint32_t unit_words = 0, my_words = 0, my_off = 0;  // lane u: words of unit u, words before it
        const bool own = n_units <= 32 && 2 * W + 2 * n_units <= V.W;
        if (own) {
          for (uint32_t u = 0; u < n_units; ++u) {
            uint32_t c = 0;
            for (uint32_t w = u * kUnitWords + lane; w < min(V.W, (u + 1) * kUnitWords); w += 32) {
              uint32_t v = V.Y[(uint64_t)S.prow[0] * V.Wp + w];
              for (uint32_t t = 1; t < np_rows; ++t) v &= V.Y[(uint64_t)S.prow[t] * V.Wp + w];
              c += __popc(v);
            }
            const uint32_t words = words_of(__reduce_add_sync(kFull, c));
            if (lane == u) {
              my_words = words;
              my_off = unit_words;
            }
            unit_words += words;
          }
        }
        const uint32_t Wn = own ? unit_words : V.W, Wpn = (Wn + 3) & ~3u;
        const uint32_t chunks = (Wn + kGramWords - 1) / kGramWords;
        const unsigned long long n_part_tiles = (unsigned long long)nt * chunks;
        const uint64_t rows_off = region_rows_off(xlen, n);
        unsigned long long dst = 0;
        if (!last && n <= 0xffffu && np_rows < 60) {
          if (lane == 0) {
            const unsigned long long gw = (unsigned long long)n * (n + 1) / 2;
            const unsigned long long size = own ? (rows_off + (unsigned long long)n * Wpn + 31) & ~31ull : 0ull;
            const unsigned long long l = atomicAdd(&next_round.l_top, (unsigned long long)(np_rows + n));
            const unsigned long long gq = atomicAdd(&next_round.g_top, gw);
            ti = atomicAdd(&next_round.tile_n, n_part_tiles);
            ii = atomicAdd(&next_round.item_n, (unsigned long long)(n - 1));
            if (own) {
              ui = atomicAdd(&next_round.unit_n, (unsigned long long)n_units * nj);
              dst = atomicAdd(&p.ctrl->arena_top, size);
            }
            ok = l + np_rows + n <= p.list_cap && gq + gw <= p.g_half && ti + n_part_tiles <= p.tile_cap &&
                 ii + n - 1 <= p.item_cap && (!own || (ui + n_units * nj <= p.tile_cap && dst + size <= p.arena_words));
            lo = (uint32_t)(l_lo + l);
            go = (uint32_t)(g_lo + gq);
          }
          ok = __shfl_sync(kFull, ok, 0);
          lo = __shfl_sync(kFull, lo, 0);
          go = __shfl_sync(kFull, go, 0);
          ti = __shfl_sync(kFull, ti, 0);
          ii = __shfl_sync(kFull, ii, 0);
          ui = __shfl_sync(kFull, ui, 0);
          dst = __shfl_sync(kFull, dst, 0);
          // (reserved slots below the capacities are filled in any case)
          const uint32_t r4 = !ok ? kNoop : own ? (uint32_t)(dst / 4) : it.roff4, plen = own ? 0u : np_rows;
          const uint32_t lrows = lo + np_rows - plen;  // (own rows: the list, which names rows of the region, is not used)
          for (uint32_t t = lane; t < n_part_tiles && ti + t < p.tile_cap; t += 32) {
            uint32_t ba, bb;
            tile_of(t % nt, ba, bb);
            p.tiles[ti + t] = SubTile{r4, own ? kIdentity : lrows, plen, n, go, ba | bb << 16, t / nt, 0};
          }
          for (uint32_t t = lane; t < n - 1 && ii + t < p.item_cap; t += 32)
            next_items[ii + t] = SubItem{r4, own ? kIdentity : lrows, plen, n, go, t, {0, 0}};
          if (own)
            for (uint32_t u = 0; u < n_units; ++u) {
              const uint32_t words = __shfl_sync(kFull, my_words, u), off = __shfl_sync(kFull, my_off, u);
              for (uint32_t j = lane; j < nj; j += 32) {
                const unsigned long long slot = ui + u * nj + j;
                const unsigned long long d = dst + rows_off + (unsigned long long)(32 * j) * Wpn + off;
                if (slot < p.tile_cap)
                  p.units[slot] = SubUnit{ok && words ? it.roff4 : kNoop, lo, np_rows | min(32u, n - 32 * j) << 16, 32 * j,
                                          (uint32_t)d, (uint32_t)(d >> 32), Wpn, u | words << 16};
              }
            }
        }
        if (ok) {
          for (uint32_t q = lane; q < np_rows; q += 32) p.lists[lo + q] = S.prow[q];
          uint32_t* const R = p.Y + dst;
          uint32_t at0 = 0;
          for (uint32_t j0 = 0; j0 < nc; j0 += 32) {
            const bool f = j0 + lane < nc && ld_cg(g + j0 + lane) >= p.minsup;
            const uint32_t bal = __ballot_sync(kFull, f), at = at0 + __popc(bal & lt);
            if (f) {
              const uint32_t r = row_of(it.m + 1 + j0 + lane);
              p.lists[lo + np_rows + at] = r;
              if (own) R[8 + ((xlen + 3) & ~3u) + at] = V.rids[r];
            }
            at0 += __popc(bal);
          }
          if (own) {
            if (lane == 0) {
              R[0] = n;
              R[1] = Wpn;
              R[2] = xlen;
              R[3] = Wn;
              R[4] = cls;
              R[5] = kNoGram;
              R[6] = R[7] = 0;
            }
            write_prefix(R);
            for (uint32_t j = lane; j < n; j += 32)
              for (uint32_t w = Wn; w < Wpn; ++w) R[rows_off + (uint64_t)j * Wpn + w] = 0u;
            st_bytes += 4ull * n * supp + 4ull * n * Wn;
          }
          if (chunks > 1)
            for (uint32_t t = lane; t < n * (n + 1) / 2; t += 32) p.G[go + t] = 0;
          ++st_parts;
        } else if (!round) {  // (k_dfs_proj counts the node again and writes its records)
          if (lane == 0) leave_to_dfs(p, (uint64_t)it.roff4 * 4, it.m);
          continue;
        } else {
          // k_dfs_proj needs the part as a region: built in the arena by this warp, its extensions queued
          const unsigned long long size = (region_rows_off(xlen, n) + (unsigned long long)n * padded_words(supp) + n + 31) & ~31ull;
          unsigned long long off = 0;
          if (lane == 0) off = atomicAdd(&p.ctrl->arena_top, size);
          off = __shfl_sync(kFull, off, 0);
          if (off + size > p.arena_words) {
            if (lane == 0) atomicOr(&p.ctrl->err, DEV_ERR_SUB);
            stop = true;
            continue;
          }
          uint32_t* const R = p.Y + off;
          const uint32_t Wp = padded_words(supp);
          uint32_t* const Y2 = R + region_rows_off(xlen, n);
          uint32_t* const rows = Y2 + (uint64_t)n * Wp;  // rows of V
          uint32_t at0 = 0;
          for (uint32_t j0 = 0; j0 < nc; j0 += 32) {
            const bool f = j0 + lane < nc && ld_cg(g + j0 + lane) >= p.minsup;
            const uint32_t bal = __ballot_sync(kFull, f), at = at0 + __popc(bal & lt);
            if (f) {
              rows[at] = row_of(it.m + 1 + j0 + lane);
              R[8 + ((xlen + 3) & ~3u) + at] = V.rids[rows[at]];
            }
            at0 += __popc(bal);
          }
          if (lane == 0) {
            R[0] = n;
            R[1] = Wp;
            R[2] = xlen;
            R[3] = W;
            R[4] = cls;
            R[5] = kNoGram;
            R[6] = R[7] = 0;
          }
          write_prefix(R);
          __syncwarp();
          for (uint32_t j0 = 0; j0 < n; j0 += 32) {
            __syncwarp();
            if (j0 + lane < n) S.lrow[lane] = rows[j0 + lane];
            if (lane == 0) atomicAdd(&p.state->progress, 1u);
            gather_rows(&S, V.Y, V.Wp, np_rows, 0, V.W, Y2 + (uint64_t)j0 * Wp, Wp, Wp, min(32u, n - j0));
          }
          st_bytes += 4ull * n * supp + 4ull * n * Wp;
          for (uint32_t j = 0; j < n; ++j)  // (words past the last position)
            if (lane < Wp - W) Y2[(uint64_t)j * Wp + W + lane] = 0u;
          __threadfence();
          __syncwarp();
          for (uint32_t t = lane; t + 1 < n; t += 32) leave_to_dfs(p, off, t);
          // (this node's own records are written below, its extensions by k_dfs_proj)
        }
        walk = false;
      }
      if (!task) {
        st_inter += nc;
        cls_work += nc;
        ++st_nodes;
        st_bytes += 4ull * (nc + 1) * V.W;
        if (n >= 2) ++st_frames;
        // the node's records: prefix u {survivor}, or the leaf
        if (n == 0 && !p.leaves) {
          // no record
        } else if (!p.out_off || !small) {
          const uint32_t n_rec = p.leaves ? 1u : n, len = n ? xlen + 1 : xlen;
          cls_sets += n_rec;
          st_sets += n_rec;
          st_items += (unsigned long long)n_rec * len;
          st_maxlen = max(st_maxlen, len);
          if (!p.out_off) {
            pend_sets += n_rec;
          } else {
            // more ids than a record mask holds: written from the pair supports, a lane per record
            unsigned long long base = 0;
            if (lane == 0) {
              base = atomicAdd(&p.ctrl->packed, ((unsigned long long)n_rec << 32) | (unsigned long long)n_rec * len);
              const unsigned long long after = (base >> 32) + n_rec;
              if ((p.max_sets && after > p.max_sets) || after > 0xfffffff0ull) atomicOr(&p.ctrl->err, DEV_ERR_ABORTED);
            }
            base = __shfl_sync(kFull, base, 0);
            uint32_t cnt = 0;
            const uint32_t n_out = n ? nc : 1u;
            for (uint32_t j0 = 0; j0 < n_out; j0 += 32) {
              const uint32_t c = n == 0 ? supp : j0 + lane < nc ? ld_cg(g + j0 + lane) : 0u;
              const bool f = n == 0 ? lane == 0 : c >= p.minsup;
              const uint32_t bal = __ballot_sync(kFull, f), at = cnt + __popc(bal & lt);
              cnt += __popc(bal);
              if (f && (!p.leaves || n == 0 || at + 1 == n)) {  // (leaves: the last survivor's)
                const uint32_t o = p.leaves ? 0u : at;
                const uint64_t rec = (base >> 32) + o, i0 = (base & 0xffffffffull) + (uint64_t)o * len;
                if (rec < p.cap_sets && i0 + len <= p.cap_items) {
                  auto id_of = [&](uint32_t t) {
                    return t < V.xlen ? V.R[8 + t]
                                      : V.rids[t < xlen ? S.prow[t - V.xlen] : row_of(it.m + 1 + j0 + lane)];
                  };
                  for (uint32_t t = 0; t < len; ++t) {
                    const uint32_t v = id_of(t);
                    uint32_t r = 0;
                    for (uint32_t u = 0; u < len; ++u) r += id_of(u) < v;
                    p.out_items[i0 + r] = v;
                  }
                  p.out_off[rec] = i0;
                  p.out_supp[rec] = c;
                } else {
                  atomicOr(&p.ctrl->err, DEV_ERR_OVERFLOW);
                }
              }
            }
          }
        } else if (p.leaves) {
          if (lane == 0) {
            S.rec[0] = n ? pre_ids | 1ull << S.at[n - 1] : pre_ids;
            S.rsupp[0] = n ? S.lsup[n - 1] : supp;
          }
          nrec = 1;
          ++cls_sets;
        } else {
          for (uint32_t q = lane; q < n; q += 32) {
            S.rec[q] = pre_ids | 1ull << S.at[q];
            S.rsupp[q] = S.lsup[q];
          }
          nrec = n;
          cls_sets += n;
        }
        if (!walk || nrec > 32) flush();
      }
      // A part of n = N rows (at most kSubAll), straight from the region's rows: the supports of all subsets of the rows are
      // counted in one pass over the words (lanes over words), then lane M stands for subset M: its record, and its
      // share of the nodes and intersections of the walk (frame M has the survivors e > max(M) with M u {e} frequent).
      auto walk_all = [&](auto tag) {
        constexpr uint32_t N = decltype(tag)::value;
        uint32_t cnt[1u << N];
#pragma unroll
        for (uint32_t m = 0; m < 1u << N; ++m) cnt[m] = 0;
        uint32_t off[N + 2];  // the rows, then the last two of the prefix
#pragma unroll
        for (uint32_t j = 0; j < N; ++j) off[j] = S.lrow[j] * V.Wp;
        off[N] = S.prow[np_rows - 1] * V.Wp;
        off[N + 1] = S.prow[np_rows > 1 ? np_rows - 2 : 0] * V.Wp;
        uint32_t nx[N + 2];  // the next words, in flight while this round's are counted
        auto fetch = [&](uint32_t w) {
#pragma unroll
          for (uint32_t j = 0; j < N + 2; ++j) nx[j] = w < V.W ? V.Y[off[j] + w] : 0u;
        };
        fetch(lane);
        for (uint32_t w = lane; w - lane < V.W; w += 32) {
          uint32_t v[1u << N], y[N];
          v[0] = nx[N] & nx[N + 1];
#pragma unroll
          for (uint32_t j = 0; j < N; ++j) y[j] = nx[j];
          fetch(w + 32);
          for (uint32_t t = 2; t < np_rows; ++t) v[0] &= w < V.W ? V.Y[(uint64_t)S.prow[t - 2] * V.Wp + w] : 0u;
#pragma unroll
          for (uint32_t m = 1; m < 1u << N; ++m) {
            const uint32_t j = 31 - __builtin_clz(m);
            v[m] = v[m ^ (1u << j)] & y[j];
            if (m & (m - 1)) cnt[m] += __popc(v[m]);
          }
        }
        uint32_t c = lane != 0 && (lane & (lane - 1)) == 0 && __ffs(lane) - 1 < (int)n && !task ? S.lsup[__ffs(lane) - 1] : 0u;
#pragma unroll
        for (uint32_t m = 3; m < 1u << N; ++m) {
          if (!(m & (m - 1))) continue;
          const uint32_t t = __reduce_add_sync(kFull, cnt[m]);
          if (lane == m) c = t;
        }
        // F: the frequent subsets (the empty one, the part itself, among them)
        const uint32_t size = __popc(lane), top = lane ? 32 - __clz(lane) : 0;  // elements above max(M): bits top ..
        const bool single = size == 1 && top <= n;
        const uint32_t F = __ballot_sync(kFull, lane == 0 || single || (size >= 2 && c >= p.minsup));
        const bool mine_f = (F >> lane) & 1u;
        uint32_t ns = 0, last_e = 0;  // survivors of frame M, the last of them
        for (uint32_t e = top; e < n; ++e)
          if (mine_f && ((F >> (lane | 1u << e)) & 1u)) {
            ++ns;
            last_e = e;
          }
        const bool frame = ns >= 2;
        const uint32_t n_frames = __popc(__ballot_sync(kFull, frame && (lane != 0 || task)));
        const uint32_t n_nodes = __reduce_add_sync(kFull, frame ? ns - 1 : 0u);
        const uint32_t n_inter = __reduce_add_sync(kFull, frame ? ns * (ns - 1) / 2 : 0u);
        st_frames += n_frames;
        st_nodes += n_nodes;
        st_inter += n_inter;
        cls_work += n_inter;
        st_bytes += 4ull * V.W * (np_rows + n);
        bool rec = mine_f && size >= 2;
        uint32_t set = lane, sp = c;
        if (p.leaves) {
          // node M: frequent, and a later survivor in its parent's frame; its leaf M u {last survivor}, or M alone
          const uint32_t parent = lane ? lane ^ (1u << (top - 1)) : 0u;
          bool node = mine_f && size >= 1;
          bool later = false;
          for (uint32_t e = top; e < n; ++e) later |= (F >> (parent | 1u << e)) & 1u;
          node = node && later;
          const uint32_t up = lane | (ns ? 1u << last_e : 0u);
          sp = __shfl_sync(kFull, c, up);
          set = up;
          rec = node;
        }
        const uint32_t bal = __ballot_sync(kFull, rec), found = __popc(bal);
        if (found) {
          cls_sets += found;
          if (p.out_off) {
            if (nrec + found > 64) flush();
            if (rec) {
              unsigned long long ids = pre_ids;
              for (uint32_t t = set; t; t &= t - 1) ids |= 1ull << S.at[__ffs(t) - 1];
              const uint32_t q = nrec + __popc(bal & lt);
              S.rec[q] = ids;
              S.rsupp[q] = sp;
            }
            nrec += found;
          } else {
            pend_sets += found;
            st_sets += found;
            st_items += __reduce_add_sync(kFull, rec ? xlen + __popc(set) : 0u);
            st_maxlen = max(st_maxlen, __reduce_max_sync(kFull, rec ? xlen + __popc(set) : 0u));
          }
        }
      };
      // The subtree of the part in S.pool, a frame at a time (M: sets of the part's rows).
      auto walk_part = [&]() {
        using M = uint32_t;
        auto popm = [](M x) -> uint32_t { return __popc(x); };
        auto low = [](M x) -> uint32_t { return __ffs(x) - 1; };
        const M one = 1;
        uint32_t* const Y = S.pool;
        uint32_t* const P = S.pool + n * Ws;
        M* const cm0 = P + W;
        M* const todo = reinterpret_cast<M*>(S.pos);  // per depth: children to expand,
        M* const surv = todo + 32;                    // survivors
        M path = 0, cur = n == 32 ? kFull : (one << n) - 1;
        unsigned long long pid = pre_ids;  // the frame's prefix as positions in ids
        uint32_t plen = xlen, cm_top = 0;
        const long long t_start = clock64();
        int32_t depth = -1;
        // one record per lane with f: rec and its support
        auto put = [&](bool f, unsigned long long rec, uint32_t supp_rec) {
          const uint32_t bal = __ballot_sync(kFull, f), cnt = __popc(bal);
          if (cnt == 0) return;
          if (nrec + cnt > 64) flush();
          if (f) {
            const uint32_t q = nrec + __popc(bal & lt);
            S.rec[q] = rec;
            S.rsupp[q] = supp_rec;
          }
          nrec += cnt;
        };
        for (;;) {
          // ---- a frame: prefix rows `path`, survivors `cur` (two or more) ----
          const uint32_t nf = popm(cur), np = nf * (nf - 1) / 2;
          M* const cm = cm0 + cm_top;
          __syncwarp();
          if ((cur >> lane) & 1u) S.idx[popm(cur & lt)] = (uint8_t)lane;
          if (lane < nf) cm[lane] = 0;
          if (path)
            for (uint32_t w = lane; w < W; w += 32) {
              uint32_t v = kFull;
              for (M t = path; t; t &= t - 1) v &= Y[low(t) * Ws + w];
              P[w] = v;
            }
          __syncwarp();
          ++depth;
          if (depth || task) ++st_frames;  // (the first frame of an extension: counted with its node)
          uint32_t found = 0, found2 = 0;
          // 2^s lanes per pair
          {
            const uint32_t s = np > 16 ? 0u : np > 8 ? 1u : np > 4 ? 2u : np > 2 ? 3u : np > 1 ? 4u : 5u;
            const uint32_t sub = lane & ((1u << s) - 1u), step = 1u << s;
            for (uint32_t p0 = 0; p0 < np; p0 += 32u >> s) {
              const uint32_t pr = p0 + (lane >> s);
              const bool valid = pr < np;
              uint32_t b = (uint32_t)((sqrtf(8.f * pr + 1.f) + 1.f) * 0.5f);  // (a, b), a < b, pr = b (b - 1) / 2 + a
              if (b * (b - 1) / 2 > pr) --b;
              if (b * (b + 1) / 2 <= pr) ++b;
              const uint32_t a = pr - b * (b - 1) / 2;
              const uint32_t ra = valid ? S.idx[a] : 0u, rb = valid ? S.idx[b] : 0u;
              const uint32_t *ya = Y + ra * Ws, *yb = Y + rb * Ws;
              uint32_t acc = 0;
              if (path) {
#pragma unroll 4
                for (uint32_t w = sub; w < W; w += step) acc += __popc(ya[w] & yb[w] & P[w]);
              } else {
#pragma unroll 4
                for (uint32_t w = sub; w < W; w += step) acc += __popc(ya[w] & yb[w]);
              }
              for (uint32_t o = step >> 1; o; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
              const bool f = valid && acc >= p.minsup && sub == 0;
              if (f) atomicOr(cm + a, one << rb);
              if (!p.leaves && p.out_off) {
                put(f, pid | 1ull << S.at[ra] | 1ull << S.at[rb], acc);
                cls_sets += __popc(__ballot_sync(kFull, f));
              } else if (!p.leaves) {
                found += __popc(__ballot_sync(kFull, f));
              }
            }
          }
          __syncwarp();
          // children: with two survivors (counted here), with more (expanded)
          const uint32_t pc = lane < nf ? popm(cm[lane]) : 0u;
          const uint32_t t2 = __ballot_sync(kFull, pc == 2), n_two = __popc(t2);
          if (pc == 2) S.two[__popc(t2 & lt)] = (uint8_t)lane;
          const M open = __reduce_or_sync(kFull, pc > 2 ? one << S.idx[lane] : 0u);
          __syncwarp();
          if (p.leaves) {
            // the leaf of every node prefix u {a}: with its last survivor, or alone
            {
              const uint32_t a = lane;
              const bool in = a + 1 < nf;
              const uint32_t ra = in ? S.idx[a] : 0u;
              const M ch = in ? cm[a] : (M)0;
              const uint32_t rl = ch ? 31 - __clz(ch) : ra;
              uint32_t acc = 0;
              if (p.out_off) {
#pragma unroll 4
                for (uint32_t w = 0; w < W; ++w) acc += __popc(Y[ra * Ws + w] & Y[rl * Ws + w] & (path ? P[w] : kFull));
                put(in, pid | 1ull << S.at[ra] | 1ull << S.at[rl], acc);
              }
              const uint32_t len = in ? plen + 1 + (ch != 0) : 0u;
              if (!p.out_off) {
                st_items += __reduce_add_sync(kFull, len);
                st_maxlen = max(st_maxlen, __reduce_max_sync(kFull, len));
              }
            }
            cls_sets += nf - 1;
            found = nf - 1;
          }
          if (n_two) {
            const uint32_t s = n_two > 16 ? 0u : n_two > 8 ? 1u : n_two > 4 ? 2u : n_two > 2 ? 3u : n_two > 1 ? 4u : 5u;
            const uint32_t sub = lane & ((1u << s) - 1u), step = 1u << s;
            for (uint32_t q0 = 0; q0 < n_two; q0 += 32u >> s) {
              const uint32_t q = q0 + (lane >> s);
              const bool valid = q < n_two;
              const uint32_t a = S.two[valid ? q : 0];
              const M ch = cm[a];
              const uint32_t ra = S.idx[a], re = low(ch), rf = 31 - __clz(ch);
              const uint32_t *ya = Y + ra * Ws, *ye = Y + re * Ws, *yf = Y + rf * Ws;
              uint32_t acc = 0, acc2 = 0;  // prefix u {a, e, f}, and (for a leaf) prefix u {a, e}
#pragma unroll 4
              for (uint32_t w = sub; w < W; w += step) {
                const uint32_t x = ya[w] & ye[w] & (path ? P[w] : kFull);
                acc += __popc(x & yf[w]);
                if (p.leaves) acc2 += __popc(x);
              }
              for (uint32_t o = step >> 1; o; o >>= 1) {
                acc += __shfl_xor_sync(kFull, acc, o);
                acc2 += __shfl_xor_sync(kFull, acc2, o);
              }
              const bool lead = valid && sub == 0, f = lead && acc >= p.minsup;
              const unsigned long long ae = pid | 1ull << S.at[ra] | 1ull << S.at[re];
              if (p.leaves) {
                const uint32_t c3 = __popc(__ballot_sync(kFull, f)), call = __popc(__ballot_sync(kFull, lead));
                cls_sets += call;
                if (p.out_off) {
                  put(lead, f ? ae | 1ull << S.at[rf] : ae, f ? acc : acc2);
                } else {
                  found2 += call;
                  st_items += (unsigned long long)call * (plen + 2) + c3;
                  st_maxlen = max(st_maxlen, plen + 2 + (c3 != 0));
                }
              } else if (p.out_off) {
                put(f, ae | 1ull << S.at[rf], acc);
                cls_sets += __popc(__ballot_sync(kFull, f));
              } else {
                found2 += __popc(__ballot_sync(kFull, f));
              }
            }
            st_frames += n_two;
          }
          st_nodes += nf - 1 + n_two;
          st_inter += np + n_two;
          cls_work += np + n_two;
          st_bytes += 4ull * W * (np + nf - 1 + 2 * n_two);
          if (!p.out_off) {  // (with records: counted when they are written)
            pend_sets += found + found2;
            st_sets += found + found2;
            if (!p.leaves) {
              cls_sets += found + found2;
              st_items += (unsigned long long)found * (plen + 2) + (unsigned long long)found2 * (plen + 3);
              if (found) st_maxlen = max(st_maxlen, plen + 2 + (found2 != 0));
            }
            if (pend_sets >= 256) flush_count();
          }
          if (stop) break;
          if (lane == 0) {
            todo[depth] = open;
            surv[depth] = cur;
            S.path[depth] = path;
            S.pids[depth] = pid;
          }
          cm_top += nf;
          __syncwarp();
          if (clock64() - t_start > p.cycles) {
            // what is left goes to the next round: every open child of every open frame, with its rows; without room there,
            // and in the last round, to k_dfs_proj, whose warps share large frames.  (A warp that walked on alone kept the
            // others waiting, past the end of their patience: 27 items in every transaction, queues of one entry: a timeout
            // after 4.4 s, now 0.8 s; 24 items 2.5 s, now 1.35.)
            uint32_t cnt = 0, words = 0, base = cm_top;
            for (int32_t d = depth; d >= 0; --d) {
              const M sd = surv[d];
              base -= popm(sd);
              const uint32_t pl = np_rows + popm((M)S.path[d]) + 1;
              for (M t = todo[d]; t; t &= t - 1, ++cnt) words += pl + popm(cm0[base + popm(sd & ((one << low(t)) - 1))]);
            }
            unsigned long long slot = p.item_cap;
            uint32_t at = 0, ok = 0;
            if (cnt && !last && lane == 0) {
              const unsigned long long l = atomicAdd(&next_round.l_top, (unsigned long long)words);
              slot = atomicAdd(&next_round.item_n, (unsigned long long)cnt);
              ok = l + words <= p.list_cap && slot + cnt <= p.item_cap;
              at = (uint32_t)(l_lo + l);
            }
            ok = __shfl_sync(kFull, ok, 0);
            at = __shfl_sync(kFull, at, 0);
            slot = __shfl_sync(kFull, slot, 0);
            base = cm_top;
            for (int32_t d = depth; d >= 0; --d) {
              const M sd = surv[d], pd = (M)S.path[d];
              base -= popm(sd);
              for (M t = todo[d]; t; t &= t - 1, ++slot) {
                const uint32_t r = low(t);
                const M rows_p = pd | one << r, rows_s = cm0[base + popm(sd & ((one << r) - 1))];
                const uint32_t pl = np_rows + popm(rows_p), ns = popm(rows_s);
                if (ok) {
                  for (uint32_t q = lane; q < np_rows; q += 32) p.lists[at + q] = S.prow[q];
                  if ((rows_p >> lane) & 1u) p.lists[at + np_rows + popm(rows_p & lt)] = S.lrow[lane];
                  if ((rows_s >> lane) & 1u) p.lists[at + pl + popm(rows_s & lt)] = S.lrow[lane];
                } else {
                  ++st_frames;
                  st_bytes += 4ull * W * (popm(rows_p) + 2 * ns);
                  stop |= !leave_subtree(&p, &S, rows_p, rows_s, S.pids[d] | 1ull << S.at[r], W, cls);
                }
                if (lane == 0 && slot < p.item_cap)
                  next_items[slot] = SubItem{ok ? it.roff4 : kNoop, at, pl, ns, 0, kSubTask, {0, 0}};
                at += pl + ns;
              }
            }
            break;
          }
          // ---- the next child: of the deepest frame that has one ----
          M t = todo[depth];
          while (t == 0) {
            cm_top -= popm(surv[depth]);
            if (--depth < 0) break;
            t = todo[depth];
          }
          if (depth < 0) break;
          const uint32_t r = low(t);
          const M sd = surv[depth];
          path = (M)S.path[depth] | one << r;
          pid = S.pids[depth] | 1ull << S.at[r];
          plen = xlen + popm(path);
          cur = cm0[cm_top - popm(sd) + popm(sd & ((one << r) - 1))];
          __syncwarp();
          if (lane == 0) todo[depth] = t & (t - 1);
          __syncwarp();
        }
      };
      if (walk && !stop && all) {
        __syncwarp();
        if (n == 2) walk_all(std::integral_constant<uint32_t, 2>{});
        else if (n == 3) walk_all(std::integral_constant<uint32_t, 3>{});
        else if (n == 4) walk_all(std::integral_constant<uint32_t, 4>{});
        else walk_all(std::integral_constant<uint32_t, 5>{});
      } else if (walk && !stop) {
        __syncwarp();
        gather_rows(&S, V.Y, V.Wp, np_rows, 0, V.W, S.pool, Ws, W, n);
        st_bytes += 4ull * n * supp + 4ull * n * W;
        __syncwarp();
        walk_part();
      }
      flush();
      if (!p.out_off && pend_sets >= 64) flush_count();
      if (lane == 0) {
        if (p.class_sets && cls_sets) atomicAdd(&p.class_sets[cls], cls_sets);
        if (p.class_work && cls_work) atomicAdd(&p.class_work[cls], cls_work);
      }
    }
    if (!wait(my_items, &now.item_done, n_items, &now.item_head, round + 1 < p.rounds, round)) break;
    if (round + 1 >= p.rounds) break;
  }
  if (!p.out_off && pend_sets) flush_count();
  if (lane == 0 && st_nodes) {
    atomicAdd(&p.ctrl->n_intersections, st_inter);
    atomicAdd(&p.ctrl->n_nodes, st_nodes);
    atomicAdd(&p.ctrl->n_frames, st_frames);
    atomicAdd(&p.ctrl->proj_bytes, st_bytes);
    if (st_parts) atomicAdd(&p.ctrl->proj_splits, st_parts);
    if (st_sets) {
      atomicAdd(&p.ctrl->sets_total, st_sets);
      atomicAdd(&p.ctrl->items_total, st_items);
      atomicMax(&p.ctrl->max_len, st_maxlen);
    }
  }
}

// dynamic shared memory and CTAs of k_sub (as many as run at once), asked once per device
cudaError_t sub_ctas(int num_sms, uint32_t* out) {
  static std::mutex mu;
  static std::map<int, uint32_t> known;
  const size_t smem = kSubWarps * sizeof(SubSmem);
  cudaError_t e = kernel_smem_limit(reinterpret_cast<const void*>(k_sub), (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, occ = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  auto it = known.find(dev);
  if (it == known.end()) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_sub, (int)kSubThreads, smem);
    if (e != cudaSuccess) return e;
    it = known.emplace(dev, (uint32_t)num_sms * std::min<uint32_t>(kSubCtasPerSm, (uint32_t)std::max(occ, 0))).first;
  }
  *out = it->second;
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_sub(const SubLaunch& p, int num_sms, cudaStream_t st) {
  uint32_t ctas = 0;
  cudaError_t e = sub_ctas(num_sms, &ctas);
  if (e != cudaSuccess) return e;
  if (ctas == 0) return cudaErrorInvalidConfiguration;
  k_sub<<<ctas, kSubThreads, kSubWarps * sizeof(SubSmem), st>>>(p);
  note_launch();
  return cudaGetLastError();
}

}  // namespace fim
