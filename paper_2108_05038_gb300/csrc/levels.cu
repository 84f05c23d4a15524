// K4 for mines of few rows: the whole search below the level-2 counts, a level at a time.
//
// With few frequent rows the search is short and bound by its chain of dependent steps, not by its work: dense_deep has
// 3,578 itemsets of up to 6 items over 41 rows, and the frame passes (k_dfs_frames: one class per CTA, ten CTA-wide
// barriers per frame) take 95 us for it, after 11 us for the level-2 lists and queue.  Here every itemset of a level
// that can be extended is expanded at the same time, by as many warps as its candidates and words take, so that the
// chain is one step per level:
//
//   frame   a prefix X with its survivors S (rows s_0 < s_1 < .. with X u {s} frequent), two or more.  Its nodes are
//           X u {s_m}, m < |S| - 1, with the candidates s_{m+1} .. (Eclat-DFS-Computation, App. B.3.2).
//   unit    up to 8 candidates of a node over 512 words a warp: one to eight warps of a CTA, by the length of the rows, AND
//           the node's rows word by word (four words per lane and load), count the candidates under them and add their
//           counts in shared memory.  (Added in global memory, a node of four warps paid four more L2 round trips a level:
//           a replayed mine of dense_deep's database took 146 us against 131.)
//   finish  the warp that has a node's last supports writes its records behind one
//           reservation, and makes the child's frame and units for the next level; or, with two to five survivors and
//           short rows, counts all their subsets in one pass, which ends the subtree there.
//
// The groups of warps claim the units of a level one after the other, and a CTA goes on to the next level when all are
// finished (phase_wait).  Level 2 enters the same way: a warp per row reads its pair counts.  Lists, supports and
// units of two levels live in fixed arenas; a search that outgrows them is repeated by the frame passes (DEV_ERR_SUB).
// The nodes, candidates and records are those of the other traversals.
//
// Measured (level-2 lists, queue and search): dense_deep 107 -> 74 us, tiny 65 -> 48 us, its 738-row sample 70 -> 45 us.  What
// bounds a level (about 8 us) is its chain of about six dependent L2 round trips: unit, rows, words, reservation, and the
// next launch or wait.
#include <algorithm>
#include <map>
#include <mutex>
#include <type_traits>

#include "proj_device.cuh"

namespace fim {
namespace {

constexpr uint32_t kLevWarps = kLevThreads / 32;
constexpr uint32_t kLevCtasPerSm = 2;
constexpr uint32_t kLevCand = 8;      // candidates of a unit
constexpr uint32_t kLevSeg4 = 128;    // 16-byte words of a unit for one warp (512 words; 64 or 256: 10% and 1% slower)
constexpr uint32_t kLevPath = 62;     // longest prefix (rows)
constexpr uint32_t kLevSingles = 3;   // levels launched by themselves
constexpr uint32_t kLevFew = 5;       // at most so many survivors: all their subsets counted at once
// Longest rows for that with two survivors, with three to five: one warp goes through the words, so that long rows take longer
// than the levels they save.  Searches of 2,800 to 3,500 itemsets (75 dense items, 300 of patterns) without the pass, with it
// for two, with it for up to five survivors, us: rows of 384 words 62, 56, 52 and 56, 56, 54; 512 words 64, 58, 58 and 56,
// 56, 58; 640 words 62, 56, 60 and 56, 54, 62; 800 words 64, 64, 66 and 58, 60, 70; 1,184 words 72, 74, 80 and 62, 66, 88.
constexpr uint32_t kLevPairWords = 800, kLevFewWords = 400;

__device__ __forceinline__ uint32_t tri_off(uint32_t m, uint32_t n) { return m * n - m * (m + 1) / 2; }  // of (m, m + 1)
// units of the nodes before node m of a frame of n survivors, for one segment: sum over nodes of ceil(candidates / 8)
__device__ __forceinline__ uint32_t units_before(uint32_t m, uint32_t n) {
  // node q has n - 1 - q candidates: the sum of ceil(c / 8) over c = n - m .. n - 1
  auto upto = [](uint32_t c) {  // sum of ceil(k / 8) for k = 1 .. c
    const uint32_t f = c / kLevCand, r = c % kLevCand;
    return kLevCand * f * (f + 1) / 2 + r * (f + 1);
  };
  return upto(n - 1) - upto(n - 1 - m);
}

// first: the level to begin with (0: level 2 from the pair counts); single: that level alone, its units dealt out in order,
// else until one is empty, the units claimed
__global__ void __launch_bounds__(kLevThreads, kLevCtasPerSm) k_levels(const __grid_constant__ LevLaunch p, const uint32_t first,
                                                                       const bool single) {
  if (p.cta_time && threadIdx.x == 0) p.cta_time[2 * blockIdx.x] = global_ns();
  __shared__ uint32_t s_rows[kLevWarps][64], s_ids[kLevWarps][64], s_few[kLevWarps][4 * kLevFew];
  __shared__ uint32_t s_part[2][kLevWarps][kLevCand], s_next[2][kLevWarps];
  __shared__ uint32_t s_run, s_first, s_done;
  const uint32_t lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
  uint32_t* const prow = s_rows[threadIdx.x >> 5];  // the node's rows
  uint32_t* const xs = s_ids[threadIdx.x >> 5];     // their ids, ascending
  uint32_t* const few = s_few[threadIdx.x >> 5];    // the first survivors: rows, supports; ids ascending, whose they are
  const uint32_t nwarps = gridDim.x * kLevWarps;
  // A unit is taken by a group of `group` warps of one CTA, a power of two: with rows of up to 512 words a warp, so that
  // the supports of rows of up to 4,096 words are added in shared memory.
  const uint32_t stride4 = p.stride / 4, group = p.group, sub = (threadIdx.x >> 5) & (group - 1);
  const uint32_t segs = (stride4 + group * kLevSeg4 - 1) / (group * kLevSeg4);
  unsigned long long st_inter = 0, st_nodes = 0, st_frames = 0, st_sets = 0, st_items = 0, st_entries = 0;
  uint32_t st_maxlen = 0;
  constexpr uint32_t kStop = DEV_ERR_ABORTED | DEV_ERR_TIMEOUT | DEV_ERR_SUB;

  // The ids of the rows prow[0 .. plen), ascending, to xs.
  auto sort_ids = [&](uint32_t plen) {
    __syncwarp();
    for (uint32_t q = lane; q < plen; q += 32) {
      const uint32_t v = __ldg(p.ids + prow[q]);
      uint32_t r = 0;
      for (uint32_t t = 0; t < plen; ++t) r += __ldg(p.ids + prow[t]) < v;
      xs[r] = v;
    }
    __syncwarp();
  };

  // The whole subtree of a node with N survivors (few), counted in one pass over the words: lane M stands for the
  // subset M of the survivors, its record and its share of the nodes and intersections of the walk (frame M has the
  // survivors e > max(M) with M u {e} frequent).  One reservation for all records.
  auto few_survivors = [&](auto tag, uint32_t n, uint32_t plen, uint32_t own) {
    constexpr uint32_t N = decltype(tag)::value;  // (n <= N: the rows past n hold nothing)
    uint32_t cnt[1u << N];
#pragma unroll
    for (uint32_t m = 0; m < 1u << N; ++m) cnt[m] = 0;
#pragma unroll 1
    for (uint32_t v = lane; v < stride4; v += 32) {
      uint4 a = __ldg(p.rows4 + (uint64_t)prow[0] * stride4 + v);
      uint4 y[N];
#pragma unroll
      for (uint32_t j = 0; j < N; ++j)
        y[j] = j < n ? __ldg(p.rows4 + (uint64_t)few[j] * stride4 + v) : make_uint4(0u, 0u, 0u, 0u);
      for (uint32_t q = 1; q < plen; ++q) {
        const uint4 x = __ldg(p.rows4 + (uint64_t)prow[q] * stride4 + v);
        a = make_uint4(a.x & x.x, a.y & x.y, a.z & x.z, a.w & x.w);
      }
#pragma unroll
      for (uint32_t w = 0; w < 4; ++w) {
        uint32_t z[1u << N];
        z[0] = w == 0 ? a.x : w == 1 ? a.y : w == 2 ? a.z : a.w;
#pragma unroll
        for (uint32_t m = 1; m < 1u << N; ++m) {
          const uint32_t j = 31 - __builtin_clz(m);
          z[m] = z[m ^ (1u << j)] & (w == 0 ? y[j].x : w == 1 ? y[j].y : w == 2 ? y[j].z : y[j].w);
          if (m & (m - 1)) cnt[m] += __popc(z[m]);
        }
      }
    }
    const uint32_t size = __popc(lane), top = lane ? 32 - __clz(lane) : 0;  // elements above max(M): bits top ..
    uint32_t c = size == 1 && top <= n ? few[kLevFew + top - 1] : lane == 0 ? own : 0u;
#pragma unroll
    for (uint32_t m = 3; m < 1u << N; ++m) {
      if (!(m & (m - 1))) continue;
      const uint32_t t = __reduce_add_sync(kFull, cnt[m]);
      if (lane == m) c = t;
    }
    const uint32_t F = __ballot_sync(kFull, lane == 0 || (size == 1 && top <= n) || (size >= 2 && c >= p.minsup));
    const bool mine_f = (F >> lane) & 1u;
    uint32_t ns = 0;  // survivors of frame M
#pragma unroll
    for (uint32_t e = 0; e < N; ++e) ns += e >= top && mine_f && ((F >> (lane | 1u << e)) & 1u);
    const bool frame = ns >= 2;
    st_frames += __popc(__ballot_sync(kFull, frame && (lane != 0 || !own)));
    st_nodes += __reduce_add_sync(kFull, frame ? ns - 1 : 0u);
    const uint32_t inter = __reduce_add_sync(kFull, frame ? ns * (ns - 1) / 2 : 0u);
    st_inter += inter;
    // records: the subsets found (lane 0: a one-item class's own), in lane order
    const bool rec_f = mine_f && (lane != 0 || own);
    const uint32_t bal = __ballot_sync(kFull, rec_f), sets = __popc(bal);
    const uint32_t len = rec_f ? plen + size : 0u;
    uint32_t x = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    const uint32_t items = __shfl_sync(kFull, x, 31);
    unsigned long long base = 0;
    if (lane == 0) {
      base = atomicAdd(&p.ctrl->packed, ((unsigned long long)sets << 32) | (p.out_off ? items : 0u));
      const unsigned long long after = (base >> 32) + sets;
      if ((p.max_sets && after > p.max_sets) || after > 0xfffffff0ull) atomicOr(&p.ctrl->err, DEV_ERR_ABORTED);
      if (p.class_sets) atomicAdd(&p.class_sets[prow[0]], (unsigned long long)sets);
      if (p.class_work && inter) atomicAdd(&p.class_work[prow[0]], (unsigned long long)inter);
    }
    st_sets += sets;
    st_items += items;
    st_maxlen = max(st_maxlen, __reduce_max_sync(kFull, len));
    if (own) st_entries += n - 1;
    if (!p.out_off) return;
    // the survivors by ascending id: their ids, and which survivor each is
    const uint32_t id = lane < n ? __ldg(p.ids + few[lane]) : kFull;
    uint32_t r = 0;
#pragma unroll
    for (uint32_t j = 0; j < N; ++j) r += __shfl_sync(kFull, id, j) < id;
    if (lane < n) {
      few[2 * kLevFew + r] = id;
      few[3 * kLevFew + r] = lane;
    }
    sort_ids(plen);
    base = __shfl_sync(kFull, base, 0);
    if (rec_f) {
      const uint64_t rec = (base >> 32) + __popc(bal & lt), it = (base & 0xffffffffull) + x - len;
      if (rec < p.cap_sets && it + len <= p.cap_items) {
        uint32_t* d = p.out_items + it;
        uint32_t q = 0;
#pragma unroll
        for (uint32_t j = 0; j < N; ++j)
          if (j < n && (lane >> few[3 * kLevFew + j]) & 1u) {
            const uint32_t v = few[2 * kLevFew + j];
            for (; q < plen && xs[q] < v; ++q) *d++ = xs[q];
            *d++ = v;
          }
        for (; q < plen; ++q) *d++ = xs[q];
        p.out_off[rec] = it;
        p.out_supp[rec] = c;
      } else {
        atomicOr(&p.ctrl->err, DEV_ERR_OVERFLOW);
      }
    }
  };

  // A node whose rows are prow[0 .. plen) and whose nc candidates have the supports sups[0 .. nc) (lane l has the l-th already,
  // s0) and are the rows list[0 .. nc), or row0 .. when list is NULL: its records (and, for a one-item class, its own: support
  // own), and its frame for level `next`.  (One call: the kernel's code has to stay within the instruction cache.)
  auto finish = [&](uint32_t plen, uint32_t nc, uint32_t s0, const uint32_t* sups, const uint32_t* rows_of, uint32_t row0,
                    uint32_t own, uint32_t next) {
    auto sup = [&](uint32_t j) { return __ldcg(sups + j); };
    auto row = [&](uint32_t j) { return rows_of ? __ldcg(rows_of + j) : row0 + j; };
    const uint32_t par = next & 1u, cls = prow[0];
    uint32_t n = 0;
    auto count = [&](uint32_t j, uint32_t c) {
      const uint32_t bal = __ballot_sync(kFull, c >= p.minsup), at = n + __popc(bal & lt);
      if (c >= p.minsup && at < kLevFew) {
        few[at] = row(j);
        few[kLevFew + at] = c;
      }
      n += __popc(bal);
    };
    count(lane, s0);
    for (uint32_t j0 = 32; j0 < nc; j0 += 128) {
      uint32_t c[4];
#pragma unroll
      for (uint32_t u = 0; u < 4; ++u) c[u] = j0 + 32 * u + lane < nc ? sup(j0 + 32 * u + lane) : 0u;
#pragma unroll
      for (uint32_t u = 0; u < 4; ++u) count(j0 + 32 * u + lane, c[u]);
    }
    __syncwarp();
    if (n == 2 && p.stride <= kLevPairWords) {
      few_survivors(std::integral_constant<uint32_t, 2>{}, n, plen, own);
      return;
    }
    if (n >= 3 && n <= kLevFew && p.stride <= kLevFewWords) {
      few_survivors(std::integral_constant<uint32_t, kLevFew>{}, n, plen, own);
      return;
    }
    const uint32_t singles = own ? 1u : 0u, sets = n + singles, items = n * (plen + 1) + singles;
    if (lane == 0 && p.class_sets && sets) atomicAdd(&p.class_sets[cls], (unsigned long long)sets);
    st_sets += sets;
    st_items += items;
    if (sets) st_maxlen = max(st_maxlen, n ? plen + 1 : plen);
    if (own) st_entries += n ? n - 1 : 0u;
    else if (n >= 2) ++st_frames;
    if (sets == 0) return;
    // one lane each reserves records, the frame, its lists, supports, nodes and units
    const bool frame = n >= 2;
    const uint32_t n_units = frame ? units_before(n - 1, n) * segs : 0u;
    LevCount* const c = p.state->level + next;
    unsigned long long got = 0;
    if (lane == 0) got = atomicAdd(&p.ctrl->packed, ((unsigned long long)sets << 32) | (p.out_off ? items : 0u));
    if (frame) {
      if (lane == 2) got = atomicAdd(&c->list, plen + n);
      if (lane == 3) got = atomicAdd(&c->sup, n * (n - 1) / 2);
      if (lane == 4) got = atomicAdd(&c->nodes, n - 1);
      if (lane == 5) got = atomicAdd(&c->units, n_units);
    }
    const unsigned long long base = __shfl_sync(kFull, got, 0);
    const uint32_t g32 = (uint32_t)got;
    const uint32_t li = __shfl_sync(kFull, g32, 2), si = __shfl_sync(kFull, g32, 3);
    const uint32_t ni = __shfl_sync(kFull, g32, 4), ui = __shfl_sync(kFull, g32, 5);
    const unsigned long long after = (base >> 32) + sets;
    if (lane == 0 && ((p.max_sets && after > p.max_sets) || after > 0xfffffff0ull)) atomicOr(&p.ctrl->err, DEV_ERR_ABORTED);
    const bool fits = frame && (uint64_t)li + plen + n <= p.list_cap &&
                      (uint64_t)si + n * (n - 1) / 2 <= p.sup_cap && (uint64_t)ni + n - 1 <= p.node_cap &&
                      (uint64_t)ui + n_units <= p.unit_cap && plen + 1 < kLevPath && next + 1 < kLevMax;
    if (frame && !fits && lane == 0) atomicOr(&p.ctrl->err, DEV_ERR_SUB);
    uint32_t* const list = p.lists + (uint64_t)par * kLevListWords + li;
    uint32_t* const nsup = p.sups + (uint64_t)par * kLevSupWords + si;
    if (p.out_off) sort_ids(plen);
    if (fits)
      for (uint32_t q = lane; q < plen; q += 32) list[q] = prow[q];
    uint32_t at0 = 0;
    for (uint32_t j0 = 0; j0 < nc; j0 += 32) {
      const uint32_t s = j0 == 0 ? s0 : j0 + lane < nc ? sup(j0 + lane) : 0u;
      const bool f = s >= p.minsup;
      const uint32_t bal = __ballot_sync(kFull, f), at = at0 + __popc(bal & lt);
      at0 += __popc(bal);
      if (f) {
        const uint32_t r = row(j0 + lane);
        if (fits) list[plen + at] = r;
        if (p.out_off) {
          const uint64_t rec = (base >> 32) + singles + at;
          const uint64_t it = (base & 0xffffffffull) + singles + (uint64_t)at * (plen + 1);
          if (rec < p.cap_sets && it + plen + 1 <= p.cap_items) {
            const uint32_t v = __ldg(p.ids + r);
            uint32_t* d = p.out_items + it;
            uint32_t q = 0;
            for (; q < plen && xs[q] < v; ++q) *d++ = xs[q];
            *d++ = v;
            for (; q < plen; ++q) *d++ = xs[q];
            p.out_off[rec] = it;
            p.out_supp[rec] = s;
          } else {
            atomicOr(&p.ctrl->err, DEV_ERR_OVERFLOW);
          }
        }
      }
    }
    if (own && p.out_off && lane == 0) {
      const uint64_t rec = base >> 32, it = base & 0xffffffffull;
      if (rec < p.cap_sets && it < p.cap_items) {
        p.out_off[rec] = it;
        p.out_items[it] = xs[0];
        p.out_supp[rec] = own;
      } else {
        atomicOr(&p.ctrl->err, DEV_ERR_OVERFLOW);
      }
    }
    if (!fits) return;
    for (uint32_t t = lane; t < n * (n - 1) / 2; t += 32) nsup[t] = 0;
    uint32_t* const left = p.nodes + (uint64_t)par * kLevNodes + ni;
    LevUnit* const U = p.units + (uint64_t)par * kLevUnits + ui;
    for (uint32_t m = lane; m + 1 < n; m += 32) {
      const uint32_t blocks = (n - 1 - m + kLevCand - 1) / kLevCand;
      left[m] = blocks * segs;
      LevUnit* u = U + units_before(m, n) * segs;
      for (uint32_t b = 0; b < blocks; ++b)
        for (uint32_t g = 0; g < segs; ++g) *u++ = LevUnit{li, plen, n, si, m, b, g, ni + m};
    }
  };

  // A CTA claims the first units of a level, one for each of its groups, before the wait for the level above, and a group's
  // first warp the next one while a unit is counted: no claim is waited for, and no group gets a second unit before each has
  // had one.  (A claim per group for the first ones too: 2,432 additions to one word, a step of tiny 250 us against 245.)
  const uint32_t wib = threadIdx.x >> 5;
  uint32_t round = 0, claim = 0;  // (claim: thread 0)
  auto claim_of = [&](uint32_t level) {
    if (!single) claim = atomicAdd(&p.state->level[level].head, kLevWarps / group);
  };
  if (threadIdx.x == 0) {
    s_done = 0;
    claim_of(first);
  }
  for (uint32_t level = first;; ++level) {
    const uint32_t par = level & 1u;
    if (threadIdx.x == 0) {
      // After an error no unit is touched: a frame that found no room leaves its reserved units unwritten, and its error was
      // set before the level above was finished.
      const uint32_t err = ld_volatile(&p.ctrl->err);
      const uint32_t n = level ? min(ld_volatile(&p.state->level[level].units), p.unit_cap) : p.n1;
      s_run = (level ? err & kStop : err & DEV_ERR_TIMEOUT) ? 0u : n;  // (a timeout: pair counts left incomplete)
      s_first = single ? blockIdx.x * (level ? kLevWarps / group : kLevWarps) : claim;
    }
    __syncthreads();
    const uint32_t n_run = s_run;  // (one value for the CTA: a group's warps go through the units together)
    if (n_run == 0) break;
    const LevUnit* const units = p.units + (uint64_t)par * kLevUnits;
    const uint32_t step = level ? nwarps / group : nwarps;
    uint32_t finished = 0, next = 0;  // units of this group; its next one (group 1: in lane 0)
    for (uint32_t t = s_first + (level ? wib / group : wib); t < n_run;
         t = single ? t + step : __shfl_sync(kFull, next, 0)) {
      if (sub == 0) ++finished;
      if (!single && sub == 0 && lane == 0) next = atomicAdd(&p.state->level[level].head, 1u);
      uint32_t plen, nc, s0, own = 0, row0 = 0;
      const uint32_t *sups, *rows_of = nullptr;
      __syncwarp();
      if (level == 0) {
        own = __ldg(p.row_supp + t);
        if (own < p.minsup) continue;  // (a sample's row)
        if (lane == 0) prow[0] = t;
        plen = 1;
        nc = p.n1 - t - 1;
        row0 = t + 1;
        sups = p.C2 + (uint64_t)t * p.n1 + t + 1;
        s0 = lane < nc ? __ldcg(sups + lane) : 0u;
        __syncwarp();
      } else {
        const uint4 f4 = __ldcg(reinterpret_cast<const uint4*>(units + t));
        const uint4 u4 = __ldcg(reinterpret_cast<const uint4*>(units + t) + 1);
        const uint32_t* const list = p.lists + (uint64_t)par * kLevListWords + f4.x;
        const uint32_t n = f4.z, m = u4.x, c0 = u4.y * kLevCand;
        plen = f4.y + 1;
        nc = n - 1 - m;
        rows_of = list + plen + m;
        uint32_t* const sup = p.sups + (uint64_t)par * kLevSupWords + f4.w + tri_off(m, n);
        sups = sup;
        for (uint32_t q = lane; q < plen; q += 32) prow[q] = __ldcg(list + (q + 1 < plen ? q : plen - 1 + m));
        const uint32_t cnt = min(kLevCand, nc - c0);
        const uint32_t myrow = lane < cnt ? __ldcg(rows_of + c0 + lane) : 0u;
        __syncwarp();
        const uint4* rows4[kLevCand];
#pragma unroll
        for (uint32_t g = 0; g < kLevCand; ++g)
          rows4[g] = p.rows4 + (uint64_t)__shfl_sync(kFull, myrow, min(g, cnt - 1)) * stride4;
        uint32_t acc[kLevCand];
#pragma unroll
        for (uint32_t g = 0; g < kLevCand; ++g) acc[g] = 0;
        const uint32_t v0 = u4.z * group * kLevSeg4, v1 = min(stride4, v0 + group * kLevSeg4);
#pragma unroll 1
        for (uint32_t v = v0 + sub * 32 + lane; v < v1; v += 32 * group) {
          uint4 a = __ldg(p.rows4 + (uint64_t)prow[0] * stride4 + v);
          for (uint32_t q = 1; q < plen; ++q) {
            const uint4 x = __ldg(p.rows4 + (uint64_t)prow[q] * stride4 + v);
            a = make_uint4(a.x & x.x, a.y & x.y, a.z & x.z, a.w & x.w);
          }
#pragma unroll
          for (uint32_t g = 0; g < kLevCand; ++g) {
            const uint4 x = __ldg(rows4[g] + v);
            acc[g] += __popc(a.x & x.x) + __popc(a.y & x.y) + __popc(a.z & x.z) + __popc(a.w & x.w);
          }
        }
        s0 = 0;
#pragma unroll
        for (uint32_t g = 0; g < kLevCand; ++g) {
          const uint32_t s = __reduce_add_sync(kFull, acc[g]);
          if (lane == g && g < cnt) s0 = s;
        }
        if (group > 1) {  // (two buffers: a third round's supports are written after the second's barrier)
          const uint32_t buf = round++ & 1u;
          uint32_t(*const part)[kLevCand] = s_part[buf] + (wib - sub);
          uint32_t* const nx = s_next[buf] + (wib - sub);
          if (sub && lane < kLevCand) part[sub][lane] = s0;
          if (sub == 0 && lane == 0) *nx = next;
          __syncwarp();
          asm volatile("bar.sync %0, %1;" ::"r"(1 + wib / group), "r"(group * 32) : "memory");
          if (sub) next = *nx;
          if (sub) continue;
          if (lane < cnt)
            for (uint32_t g = 1; g < group; ++g) s0 += part[g][lane];
        }
        if (nc > kLevCand || segs > 1) {  // (else: the node's only unit, its supports in the lanes)
          if (s0) atomicAdd(sup + c0 + lane, s0);
          __threadfence();
          __syncwarp();
          uint32_t left = 0;
          if (lane == 0) left = atomicSub(p.nodes + (uint64_t)par * kLevNodes + u4.w, 1u);
          if (__shfl_sync(kFull, left, 0) != 1u) continue;
          __threadfence();  // the node's last unit
          s0 = lane < nc ? __ldcg(sup + lane) : 0u;
        }
        st_inter += nc;
        ++st_nodes;
        if (lane == 0 && p.class_work) atomicAdd(&p.class_work[prow[0]], (unsigned long long)nc);
      }
      finish(plen, nc, s0, sups, rows_of, row0, own, level + 1);
    }
    if (single) break;
    LevCount* const c = p.state->level + level;
    if (!phase_wait(finished, &c->done, n_run, &c->head, &c->head, &p.ctrl->err, kStop, &s_done, [&] { claim_of(level + 1); }))
      break;
  }
  if (lane == 0 && st_sets) {
    atomicAdd(&p.ctrl->sets_total, st_sets);
    atomicAdd(&p.ctrl->items_total, st_items);
    atomicMax(&p.ctrl->max_len, st_maxlen);
  }
  if (lane == 0 && st_nodes) {
    atomicAdd(&p.ctrl->n_intersections, st_inter);
    atomicAdd(&p.ctrl->n_nodes, st_nodes);
    atomicAdd(&p.ctrl->n_frames, st_frames);
  }
  if (lane == 0 && st_entries) atomicAdd(&p.ctrl->n_entries, (uint32_t)st_entries);
  if (p.cta_time) {
    __syncthreads();
    if (threadIdx.x == 0) p.cta_time[2 * blockIdx.x + 1] = global_ns();
  }
}

}  // namespace

// CTAs of the launch (as many as run at once), asked once per device
cudaError_t levels_ctas(int num_sms, uint32_t* out) {
  static std::mutex mu;
  static std::map<int, uint32_t> known;
  int dev = 0, occ = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  auto it = known.find(dev);
  if (it == known.end()) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_levels, (int)kLevThreads, 0);
    if (e != cudaSuccess) return e;
    it = known.emplace(dev, (uint32_t)num_sms * std::min<uint32_t>(kLevCtasPerSm, (uint32_t)std::max(occ, 0))).first;
  }
  *out = it->second;
  return *out ? cudaSuccess : cudaErrorInvalidConfiguration;
}

cudaError_t launch_levels(const LevLaunch& p, uint32_t ctas, cudaStream_t st) {
  // The first levels, which nearly every search has, as launches of their own, the others until one is empty.  (With two,
  // three, four of their own: a step of tiny 255, 259, 269 us, of dense_deep's database 328, 328, 333, its replayed mine
  // 120.7, 119.8, 118.4.)
  LevLaunch q = p;
  q.cta_time = nullptr;
  for (q.group = 1; q.group < kLevWarps && q.group * kLevSeg4 * 4 < p.stride; q.group *= 2) {}
  for (uint32_t level = 0; level < kLevSingles; ++level) {
    k_levels<<<ctas, kLevThreads, 0, st>>>(q, level, true);
    note_launch();
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  q.cta_time = p.cta_time;
  k_levels<<<ctas, kLevThreads, 0, st>>>(q, kLevSingles, false);
  note_launch();
  return cudaGetLastError();
}

}  // namespace fim
