// Greedy max-coverage (Alg. 4 / Alg. 7) by peaks: every pick that can be known at once.
//
// The greedy's key is (marginal gain, smaller id first).  An element is a peak when its key is
// the largest among the elements that share an uncovered walk with it.  A peak is a pick with
// its present gain, whatever else is picked before it: its gain changes only when an element
// that shares a walk with it is picked, those have smaller keys, and keys only fall, so the
// greedy comes to the peak first.  And the greedy's picks come in key order.  So each round
// takes all peaks, covers their walks, takes the counts down and looks again, and the picks
// are sorted at the end; it stops once k picks are above everything that is left.  Rounds
// follow the longest chain of picks that touch each other, not k: 1-5 for 300-1,000 picks of
// R-MAT edges over 7 K-55 K walks, 6-35 for 100 picks where a few nodes hold most walks.
//
// A phase looks at the candidates whose count reaches a floor, found from a histogram of the
// counts: those below it have smaller keys, so they make no difference until the rest has
// fallen below the floor, which ends the phase.
//
// The greedy with one pick per barrier (cover.cu) is bound by latency, 3.4-8 us a pick.  Per
// greedy against it: k = 1000 edges, 150 K R-MAT 22 walks, 5.1 -> 0.25 ms; k = 300 edges,
// 7 K-222 K R-MAT 18 walks, 1.1-2.0 -> 0.10-0.14 ms; k = 100 nodes of 8 K with random coins,
// 5.3 K walks, 0.59 -> 0.27 ms (33 rounds).  Taking one gain level a round instead (the picks of
// a level are an independent set) needed 9-104 rounds there and measured 0.15-1.1 ms.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <utility>

#include "solver.cuh"

namespace hsaw {

namespace cg = cooperative_groups;

namespace {

constexpr uint32_t COUNT_BINS = 4096;  // counts from COUNT_BINS - 1 up share the last bin
constexpr uint32_t SORT_MAX = 4096;    // picks ranked against each other from shared memory

// ctl words of a run; the list's length (high half) and its pairs (low half) grow together in
// one 64-bit word
enum { PC_PICKS = 0, PC_FLOOR = 1, PC_GAIN = 2, PC_ROUNDS = 3, PC_STUCK = 4, PC_TOTAL = 5, PC_LIST = 6 /* 64 bits */,
       PC_OWNED = 8 /* counts were not taken down */, PC_LEFT = 9 /* it takes too long this way */,
       PC_KEEP = 10 /* pairs that may lie outside the CTAs */, PC_WORDS = 16 };

// A walk of a listed element: {walk, element, index in the list, 1 for the element's first}.
using Pair = uint4;

struct PeakParams {
  const Pair* pairs;
  uint32_t* failed;            // per listed element: the last round in which it was no peak
  uint2* seen;                 // and the last round that looked at it, with its count then
  uint32_t* cnt;               // running counts
  const uint32_t* walk_eoff;   // per walk: its entries, from the range's first
  const uint32_t* entry;       // element of each entry; the range's first is entry[*from - from_sub] (from NULL: 0)
  const int64_t* from;
  int64_t from_sub;
  uint32_t list_cap, pair_cap;
  uint32_t* stamp;             // per walk: 0, or the round that covered it
  unsigned long long* top[2];  // per walk, by the round's parity: the largest key signed on it
  uint32_t* out_u;
  uint32_t* out_gain;
  uint32_t* ctl;
  uint32_t k;
  uint32_t round0;             // rounds of earlier phases
  uint32_t max_rounds;
  uint32_t room;               // pairs that the CTAs hold
};

__device__ __forceinline__ unsigned long long peak_key(uint32_t count, uint32_t u) {
  return ((unsigned long long)count << 32) | (0xFFFFFFFFu - u);
}

// The counts of the entries [range.x, range.y) of the walks of the lanes in `mine` go down by
// one, the whole warp on each.  Four walks' entries are in flight at a time.
__device__ __forceinline__ void take_down(const PeakParams& P, const uint32_t* __restrict__ entry, unsigned mine,
                                          uint2 range, int lane) {
  while (mine) {
    uint32_t b[4], e[4], x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int src = mine ? __ffs(mine) - 1 : 0;
      b[j] = __shfl_sync(0xffffffffu, range.x, src) + lane;
      e[j] = mine ? __shfl_sync(0xffffffffu, range.y, src) : 0u;
      mine &= mine - 1;
      x[j] = b[j] < e[j] ? __ldg(&entry[b[j]]) : 0u;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (b[j] < e[j]) atomicSub(&P.cnt[x[j]], 1u);
      for (uint32_t p = b[j] + 32; p < e[j]; p += 32) atomicSub(&P.cnt[__ldg(&entry[p])], 1u);
    }
  }
}

// A CTA's own part of the list: whole elements, their pairs in registers, their counts in shared
// memory.
constexpr int OWN_PAIRS = 16;            // pairs a thread
constexpr uint32_t OWN_ELEMENTS = 3072;  // elements a CTA (16 bits each in registers)

struct OwnPart {
  uint32_t count[OWN_ELEMENTS];   // uncovered walks of the element
  uint32_t id[OWN_ELEMENTS];
  uint32_t failed[OWN_ELEMENTS];  // the last round in which it was no peak
  uint32_t first[2];              // the CTA's first pair, and the next CTA's
  uint32_t none[16];              // per CTA: 1 if its part has no room
};

// This CTA's part, [first[0], first[1]): an even share of the pairs, moved up to where an element
// begins.  True if each CTA of the cluster has room for its own.
__device__ __forceinline__ bool own_part(const PeakParams& P, uint32_t n, OwnPart& O, cg::cluster_group& cluster) {
  constexpr uint32_t NONE = 0xffffffffu;
  const uint32_t rank = cluster.block_rank(), C = cluster.num_blocks();
  const uint32_t from[2] = {(uint32_t)((uint64_t)n * rank / C), (uint32_t)((uint64_t)n * (rank + 1) / C)};
  cg::cluster_group::arrival_token started = cluster.barrier_arrive();
  if (threadIdx.x < 2) O.first[threadIdx.x] = NONE;
  __syncthreads();
  for (uint32_t j = 0; j < OWN_PAIRS; ++j) {  // an element longer than that has no room in a CTA
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const uint32_t i = from[q] + j * blockDim.x + threadIdx.x;
      if (i >= n) atomicMin(&O.first[q], n);
      else if (__ldg(&P.pairs[i].w)) atomicMin(&O.first[q], i);
    }
    __syncthreads();
    const bool found = O.first[0] != NONE && O.first[1] != NONE;
    __syncthreads();
    if (found) break;
  }
  const uint32_t b = O.first[0], e = O.first[1];
  bool room = b != NONE && e != NONE && e - b <= OWN_PAIRS * blockDim.x;
  if (room && e > b) room = __ldg(&P.pairs[e - 1].z) - __ldg(&P.pairs[b].z) < OWN_ELEMENTS;
  cluster.barrier_wait(std::move(started));  // the peers run: their shared memory can be written
  if (threadIdx.x < C) *cluster.map_shared_rank(&O.none[rank], threadIdx.x) = room ? 0u : 1u;
  cluster.sync();
  return !__any_sync(0xffffffffu, (threadIdx.x & 31) < C && O.none[threadIdx.x & 31]);
}

}  // namespace

// One cluster, a thread per (element, walk) pair of the list; stamps and keys in global memory
// (L2).  Bound by latency: the barriers of a round and the dependent L2 reads before each.
//
// Where whole elements of the list fit the CTAs (OwnPart: 16 pairs a thread, 2^18 on 16 CTAs of 1,024
// threads and 2^17 of 512, less what the division at elements costs; 3,072 elements a CTA), an element's walks are looked at by one CTA alone: its count is
// that of its pairs whose walk has no stamp, so no pick takes counts down walk entry by walk
// entry (k_take_down does that for all of a phase's walks if another phase follows), and whether
// it is a peak is settled within the CTA, which leaves two cluster barriers a round of three.
// Against counts in global memory, 1,024 threads a CTA: the greedy of 5.3 K node walks and k = 100 (33 rounds)
// 360 -> 298 us, of 7-222 K edge walks and k = 300 110-220 -> 94-137 us.
// Longer lists, or an element in more walks than a CTA has room for, keep counts in global memory:
// about 0.15-0.25 ns a pair and round, against 5 us a pick and an index of the walks (65 us a million
// elements) for the greedy that takes one pick at a time.  Which is the faster then depends on the
// rounds, which nothing tells beforehand: peak_pairs draws the line.
__global__ void __launch_bounds__(1024, 1) k_greedy_peaks(const __grid_constant__ PeakParams P) {
  __shared__ uint32_t s_red[32];
  __shared__ uint32_t slot[2][16];  // by round parity, per CTA: its largest count
  const unsigned FULL = 0xffffffffu;
  cg::cluster_group cluster = cg::this_cluster();
  const uint32_t rank = cluster.block_rank(), C = cluster.num_blocks();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t gtid = rank * blockDim.x + threadIdx.x, threads = C * blockDim.x;
  const uint32_t gwarp = gtid >> 5, warps = threads >> 5;
  const uint32_t n = __ldcg(&P.ctl[PC_LIST]);
  // the host makes room and comes back, or leaves it
  if (n > min(P.pair_cap, max(__ldcg(&P.ctl[PC_KEEP]), P.room)) || __ldcg(&P.ctl[PC_LIST + 1]) > P.list_cap) return;
  const uint32_t* __restrict__ entry = P.entry + (P.from ? *P.from - P.from_sub : 0);
  const uint32_t stripe = (n + 31) / 32;
  const uint32_t floor_gain = __ldcg(&P.ctl[PC_FLOOR]);
  __shared__ OwnPart O;
  __shared__ uint32_t s_picks;  // of earlier phases
  if (threadIdx.x == 0) s_picks = __ldcg(&P.ctl[PC_PICKS]);
  if (threadIdx.x < 32) s_red[threadIdx.x] = 0u;  // a block may have fewer than 32 warps
  const bool owned = own_part(P, n, O, cluster);
  uint32_t walk[OWN_PAIRS], el2[OWN_PAIRS / 2] = {}, alive = 0;  // this thread's pairs; elements in 16 bits
  auto el = [&](int j) { return el2[j / 2] >> 16 * (j & 1) & 0xFFFFu; };
  const uint32_t own_first = owned ? O.first[0] : 0u, own_n = owned ? O.first[1] - own_first : 0u;
  const uint32_t el_first = own_n ? __ldg(&P.pairs[own_first].z) : 0u;
  const uint32_t own_elements = own_n ? __ldg(&P.pairs[own_first + own_n - 1].z) - el_first + 1 : 0u;
  if (owned) {
    for (uint32_t e = threadIdx.x; e < own_elements; e += blockDim.x) O.count[e] = O.failed[e] = 0u;
#pragma unroll
    for (int j = 0; j < OWN_PAIRS; ++j) {
      const uint32_t i = j * blockDim.x + threadIdx.x;
      walk[j] = 0u;
      if (i < own_n) {
        const Pair x = __ldg(&P.pairs[own_first + i]);
        walk[j] = x.x;
        const uint32_t e = x.z - el_first;
        el2[j / 2] |= e << 16 * (j & 1);
        alive |= 1u << j;
        if (x.w) O.id[e] = x.y;
      }
    }
    __syncthreads();
    // walks that earlier phases cover are no longer counted
#pragma unroll
    for (int j = 0; j < OWN_PAIRS; ++j) {
      if (!(alive >> j & 1u)) continue;
      if (__ldcg(&P.stamp[walk[j]])) alive &= ~(1u << j);
      else atomicAdd(&O.count[el(j)], 1u);
    }
    __syncthreads();
  }
  uint32_t picks = 0, g = 0, r = P.round0;
  bool stuck = false, left = false;
  for (;;) {
    ++r;
    picks = __ldcg(&P.ctl[PC_PICKS]);
    if (!owned) {
      const uint64_t keep = __ldcg(&P.ctl[PC_KEEP]);
      left = n > keep || (uint64_t)n * (r - P.round0) > 16 * keep + (picks - s_picks) * PEAK_PICK;
      if (left) break;  // the same decision in every CTA
    }
    // 1. elements at or above the floor sign their keys on their uncovered walks; the largest
    // count
    unsigned long long* const top = P.top[r & 1];
    uint32_t m = 0;
    if (owned) {
      if (r > P.round0 + 1) {  // the last round's walks leave the counts
        uint32_t gone = 0;
#pragma unroll
        for (int j = 0; j < OWN_PAIRS; ++j)
          if (alive >> j & 1u) gone |= (__ldcg(&P.stamp[walk[j]]) ? 1u : 0u) << j;
#pragma unroll
        for (int j = 0; j < OWN_PAIRS; ++j)
          if (gone >> j & 1u) atomicSub(&O.count[el(j)], 1u);
        alive &= ~gone;
        __syncthreads();
      }
#pragma unroll
      for (int j = 0; j < OWN_PAIRS; ++j) {
        if (!(alive >> j & 1u)) continue;
        const uint32_t c = O.count[el(j)];
        if (c < floor_gain) continue;
        m = max(m, c);
        atomicMax(&top[walk[j]], peak_key(c, O.id[el(j)]));
      }
    }
#pragma unroll 4
    for (uint32_t i = owned ? n : gtid; i < n; i += threads) {
      const Pair x = __ldg(&P.pairs[i]);
      const uint32_t c = __ldcg(&P.cnt[x.y]), st = __ldcg(&P.stamp[x.x]);
      if (c >= floor_gain) {
        m = max(m, c);
        if (st == 0u) atomicMax(&top[x.x], peak_key(c, x.y));
      }
    }
    m = __reduce_max_sync(FULL, m);
    if (lane == 0) s_red[w] = m;
    __syncthreads();
    if (w == 0) {
      const uint32_t bm = __reduce_max_sync(FULL, s_red[lane]);
      if (lane < (int)C) *cluster.map_shared_rank(&slot[r & 1][rank], lane) = bm;
    }
    cluster.sync();
    g = __reduce_max_sync(FULL, lane < (int)C ? slot[r & 1][lane] : 0u);
    if (g < floor_gain || g == 0) break;  // the same decision in every warp
    if (picks >= P.k) {                   // k picks above everything left?
      uint32_t above = 0;
      for (uint32_t i = threadIdx.x; i < picks; i += blockDim.x) above += __ldcg(&P.out_gain[i]) > g ? 1u : 0u;
      above = __reduce_add_sync(FULL, above);
      if (lane == 0) s_red[w] = above;
      __syncthreads();
      above = __reduce_add_sync(FULL, s_red[lane]);
      __syncthreads();  // s_red is written again in the next round
      if (above >= P.k) break;
    }
    if (r - P.round0 > P.max_rounds) {
      stuck = true;
      break;
    }
    // 2. an element whose key is not the largest on one of its uncovered walks is no peak.  The
    // other parity's words are cleared for the next round on the way: a walk that no element
    // at or above the floor reaches any more is not looked at again.
    unsigned long long* const other = P.top[(r + 1) & 1];
    if (owned) {
      unsigned long long t[4];
#pragma unroll
      for (int j0 = 0; j0 < OWN_PAIRS; j0 += 4) {
#pragma unroll
        for (int j = j0; j < j0 + 4; ++j) t[j - j0] = alive >> j & 1u ? __ldcg(&top[walk[j]]) : 0ull;
#pragma unroll
        for (int j = j0; j < j0 + 4; ++j) {
          const uint32_t c = alive >> j & 1u ? O.count[el(j)] : 0u;
          if (c < floor_gain) continue;
          if (t[j - j0] != peak_key(c, O.id[el(j)])) O.failed[el(j)] = r;
          other[walk[j]] = 0ull;
        }
      }
      __syncthreads();
      // 3. peaks are picks, their walks are stamped
      for (uint32_t e = threadIdx.x; e < own_elements; e += blockDim.x) {
        const uint32_t c = O.count[e];
        if (c < floor_gain || O.failed[e] == r) continue;
        const uint32_t pos = atomicAdd(&P.ctl[PC_PICKS], 1u);
        P.out_u[pos] = O.id[e];
        P.out_gain[pos] = c;
      }
#pragma unroll
      for (int j = 0; j < OWN_PAIRS; ++j)
        if ((alive >> j & 1u) && O.count[el(j)] >= floor_gain && O.failed[el(j)] != r) P.stamp[walk[j]] = r;
      cluster.sync();
      continue;
    }
#pragma unroll 4
    for (uint32_t i = gtid; i < n; i += threads) {
      const Pair x = __ldg(&P.pairs[i]);
      const uint32_t c = __ldcg(&P.cnt[x.y]), st = __ldcg(&P.stamp[x.x]);
      const unsigned long long t = __ldcg(&top[x.x]);
      if (c >= floor_gain) {
        if (st == 0u) {
          if (t != peak_key(c, x.y)) P.failed[x.z] = r;
          other[x.x] = 0ull;
        }
        if (x.w) P.seen[x.z] = make_uint2(r, c);
      }
    }
    cluster.sync();
    // 3. peaks are picks: their uncovered walks are stamped and the elements of those lose one
    // each (peaks by what step 2 noted: the counts fall from here on).  A warp's lanes take
    // pairs from 32 stripes, so that a peak's walks spread over the warps.
    for (uint32_t i0 = gwarp; i0 < stripe; i0 += warps) {
      const uint32_t i = lane * stripe + i0;
      uint2 range = make_uint2(0u, 0u);
      bool fresh = false;
      if (i < n) {
        const Pair x = __ldg(&P.pairs[i]);
        const uint2 seen = __ldcg(&P.seen[x.z]);
        if (seen.x == r && __ldcg(&P.failed[x.z]) != r) {
          fresh = __ldcg(&P.stamp[x.x]) == 0u;
          range = make_uint2(__ldg(&P.walk_eoff[x.x]), __ldg(&P.walk_eoff[x.x + 1]));
          if (fresh) P.stamp[x.x] = r;
          if (x.w) {
            const uint32_t pos = atomicAdd(&P.ctl[PC_PICKS], 1u);
            P.out_u[pos] = x.y;
            P.out_gain[pos] = seen.y;
          }
        }
      }
      take_down(P, entry, __ballot_sync(FULL, fresh), range, lane);
    }
    cluster.sync();
  }
  cluster.sync();  // no CTA leaves while a peer may still write its shared memory
  if (gtid == 0) {
    P.ctl[PC_GAIN] = g;
    P.ctl[PC_ROUNDS] = r;
    P.ctl[PC_STUCK] = stuck ? 1u : 0u;
    P.ctl[PC_OWNED] = owned ? 1u : 0u;
    P.ctl[PC_LEFT] = left ? 1u : 0u;
  }
}

// Counts without the walks stamped after round `round0`: a warp looks at 32 stamps and reads those
// walks' entries one walk at a time.
__global__ void __launch_bounds__(256) k_take_down(const __grid_constant__ PeakParams P, uint32_t walks, uint32_t round0) {
  const uint32_t* __restrict__ entry = P.entry + (P.from ? *P.from - P.from_sub : 0);
  const int lane = threadIdx.x & 31;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t j0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; (uint64_t)j0 * 32 < walks; j0 += warps) {
    const uint32_t j = j0 * 32 + lane;
    const bool mine = j < walks && P.stamp[j] > round0;
    const uint2 range = mine ? make_uint2(__ldg(&P.walk_eoff[j]), __ldg(&P.walk_eoff[j + 1])) : make_uint2(0u, 0u);
    take_down(P, entry, __ballot_sync(0xffffffffu, mine), range, lane);
  }
}

// Counts of the elements of walks [first, first + count), by element id.
__global__ void __launch_bounds__(256) k_count_elements(const int64_t* __restrict__ node_off, int64_t first,
                                                        int64_t count, int edge_mode, const int32_t* __restrict__ el,
                                                        uint32_t* __restrict__ cnt) {
  const int64_t b = node_off[first] - (edge_mode ? first : 0);
  const int64_t e = node_off[first + count] - (edge_mode ? first + count : 0);
  for (int64_t p = b + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < e; p += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&cnt[el[p]], 1u);
}

// Histogram of the counts of the candidates (counts from 1 up).  Most R-MAT walk elements occur
// once or twice: those two bins are kept in registers, not counted by atomics on one word.
// uid: element id of each count, NULL if counts are by id.
__global__ void __launch_bounds__(512) k_peak_hist(const uint32_t* __restrict__ cnt, const int32_t* __restrict__ uid,
                                                   const uint8_t* __restrict__ cand, uint32_t U,
                                                   uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[COUNT_BINS];
  for (uint32_t i = threadIdx.x; i < COUNT_BINS; i += blockDim.x) h[i] = 0;
  __syncthreads();
  uint32_t one = 0, two = 0;
  auto add = [&](uint32_t u, uint32_t v) {
    if (v == 0 || (cand && !cand[uid ? uid[u] : u])) return;
    if (v == 1) ++one;
    else if (v == 2) ++two;
    else atomicAdd(&h[min(v, COUNT_BINS - 1)], 1u);
  };
  const uint4* cnt4 = reinterpret_cast<const uint4*>(cnt);  // a buffer of its own: 16-byte aligned
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < U / 4; q += gridDim.x * blockDim.x) {
    const uint4 v = cnt4[q];
    if (v.x | v.y | v.z | v.w) {
      add(4 * q, v.x);
      add(4 * q + 1, v.y);
      add(4 * q + 2, v.z);
      add(4 * q + 3, v.w);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x < U % 4) add(U / 4 * 4 + threadIdx.x, cnt[U / 4 * 4 + threadIdx.x]);
  one = __reduce_add_sync(0xffffffffu, one);
  two = __reduce_add_sync(0xffffffffu, two);
  if ((threadIdx.x & 31) == 0) {
    if (one) atomicAdd(&h[1], one);
    if (two) atomicAdd(&h[2], two);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < COUNT_BINS; i += blockDim.x)
    if (h[i]) atomicAdd(&hist[i], h[i]);
}

// The phase's floor and the list of candidates that reach it, {element, its first entry of
// inv_walk, its first pair, 0}, in no order.  Every listed element may be picked and covered, and
// is read in each round, so the list holds half as many again as the k picks wanted (1,000
// R-MAT edge picks came from the first 1,100-1,500) and a few, and more while it is short.
__global__ void __launch_bounds__(512) k_peak_list(const uint32_t* __restrict__ hist, uint32_t k, uint32_t keep,
                                                   uint32_t sparse, uint64_t elements,
                                                   const uint32_t* __restrict__ cnt, const int32_t* __restrict__ uid,
                                                   const uint8_t* __restrict__ cand,
                                                   const uint32_t* __restrict__ inv_off, uint32_t U, uint32_t list_cap,
                                                   uint4* __restrict__ list, uint32_t* __restrict__ failed,
                                                   uint2* __restrict__ seen, uint32_t* __restrict__ index,
                                                   uint32_t* __restrict__ ctl) {
  constexpr uint32_t PER = COUNT_BINS / 512;
  constexpr unsigned long long FEW_WALKS = 1ull << 15;
  __shared__ uint32_t n_warp[16], s_few, s_want;
  __shared__ unsigned long long w_warp[16];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_few = s_want = COUNT_BINS;
  // thread t holds PER bins from COUNT_BINS - 1 - t PER downwards, so an inclusive scan over the
  // threads gives the candidates at or above a bin and their walks
  const uint32_t hi = COUNT_BINS - 1 - threadIdx.x * PER;
  uint32_t own[PER], n = 0;
  unsigned long long walks = 0;
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    own[i] = hi - i ? hist[hi - i] : 0u;
    n += own[i];
    walks += (unsigned long long)own[i] * (hi - i);
  }
  uint32_t n_inc = n;
  unsigned long long w_inc = walks;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, n_inc, o);
    const unsigned long long z = __shfl_up_sync(0xffffffffu, w_inc, o);
    if (lane >= o) {
      n_inc += y;
      w_inc += z;
    }
  }
  if (lane == 31) {
    n_warp[w] = n_inc;
    w_warp[w] = w_inc;
  }
  __syncthreads();
  uint32_t above = n_inc - n, total = 0;
  unsigned long long walks_above = w_inc - walks;
  for (int i = 0; i < 16; ++i) {
    total += n_warp[i];
    if (i < w) {
      above += n_warp[i];
      walks_above += w_warp[i];
    }
  }
  const uint32_t want = (uint32_t)min((uint64_t)total, peak_list_goal(k));
  const unsigned long long few = max(16ull * k, 1024ull);
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    const uint32_t bin = hi - i, before = above;  // before: the candidates above this bin
    above += own[i];
    walks_above += (unsigned long long)own[i] * bin;
    if (bin == 0) continue;
    if (above <= few && walks_above <= FEW_WALKS) atomicMin(&s_few, bin);
    // the bin that brings the list to `want`; with too many ties, the bin above it
    if (above >= want && before < want) s_want = above <= few || before == 0 ? bin : bin + 1;
  }
  __syncthreads();
  const uint32_t floor_gain = total ? min(s_few, s_want) : 1u;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ctl[PC_FLOOR] = floor_gain;
    ctl[PC_TOTAL] = total;
    ctl[PC_KEEP] = keep + (elements < (uint64_t)total * PEAK_SPARSE ? sparse : 0u);
  }
  // 128 counts a warp at a time: few reach the floor, so most are looked at once, four a lane
  const uint4* cnt4 = reinterpret_cast<const uint4*>(cnt);
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t g0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; (uint64_t)g0 * 128 < U; g0 += warps) {
    const uint32_t at4 = g0 * 32 + lane;  // the lane's four counts
    uint4 q = make_uint4(0u, 0u, 0u, 0u);
    if (at4 < U / 4) {
      q = cnt4[at4];
    } else if (at4 == U / 4) {
      const uint32_t left = U % 4;
      q.x = left > 0 ? cnt[4 * at4] : 0u;
      q.y = left > 1 ? cnt[4 * at4 + 1] : 0u;
      q.z = left > 2 ? cnt[4 * at4 + 2] : 0u;
    }
    if (!__any_sync(0xffffffffu, max(max(q.x, q.y), max(q.z, q.w)) >= floor_gain)) continue;
#pragma unroll
    for (int part = 0; part < 4; ++part) {
      const uint32_t u = 4 * at4 + part;
      const uint32_t v = part == 0 ? q.x : part == 1 ? q.y : part == 2 ? q.z : q.w;
      const bool in = v >= floor_gain && (!cand || cand[uid ? uid[u] : u]);
      const unsigned b = __ballot_sync(0xffffffffu, in);
      if (!b) continue;
      const uint32_t q0 = in && inv_off ? inv_off[u] : 0u, len = !in ? 0u : inv_off ? inv_off[u + 1] - q0 : v;
      unsigned long long inc = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      unsigned long long at = 0;
      if (lane == 31) at = atomicAdd(reinterpret_cast<unsigned long long*>(&ctl[PC_LIST]),
                                     ((unsigned long long)__popc(b) << 32) | inc);
      at = __shfl_sync(0xffffffffu, at, 31);
      const uint32_t i = (uint32_t)(at >> 32) + __popc(b & ((1u << lane) - 1u));
      if (in && i < list_cap) {
        list[i] = make_uint4(u, q0, (uint32_t)at + (uint32_t)(inc - len), 0u);
        failed[i] = 0u;
        seen[i] = make_uint2(0u, 0u);
        if (index) index[u] = i;
      }
    }
  }
}

// The list's (element, walk) pairs, element by element, from the inverted index.
__global__ void __launch_bounds__(256) k_peak_pairs(const uint4* __restrict__ list, const uint32_t* __restrict__ inv_walk,
                                                    const uint32_t* __restrict__ ctl, uint32_t list_cap,
                                                    uint32_t pair_cap, Pair* __restrict__ pairs) {
  const uint32_t n = ctl[PC_LIST], elements = ctl[PC_LIST + 1];
  if (n > pair_cap || elements > list_cap) return;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = elements;  // the last element whose first pair is at or before i
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (list[mid].z <= i) lo = mid; else hi = mid;
    }
    const uint4 x = list[lo];
    pairs[i] = make_uint4(inv_walk[x.y + ((uint32_t)i - x.z)], x.x, lo, x.z == i ? 1u : 0u);
  }
}

// The same pairs from the walks themselves, where counts are by element id and no inverted index
// was made: LANES lanes read a walk that no pick covers yet, and each entry whose count reaches
// the floor takes the next pair of its element.  Reads every entry once, with its count.
template <int LANES>
__global__ void __launch_bounds__(256) k_walk_pairs(const __grid_constant__ PeakParams P, uint32_t walks,
                                                    const uint8_t* __restrict__ cand,
                                                    const uint32_t* __restrict__ index, uint4* __restrict__ list,
                                                    Pair* __restrict__ pairs) {
  if (P.ctl[PC_LIST] > min(P.pair_cap, max(P.ctl[PC_KEEP], P.room)) || P.ctl[PC_LIST + 1] > P.list_cap) return;
  const uint32_t floor_gain = P.ctl[PC_FLOOR];
  const uint32_t* __restrict__ entry = P.entry + (*P.from - P.from_sub);
  const uint32_t lane = threadIdx.x % LANES;
  const uint32_t groups = gridDim.x * blockDim.x / LANES;
  for (uint32_t j = (blockIdx.x * blockDim.x + threadIdx.x) / LANES; j < walks; j += groups) {
    const uint32_t b = P.walk_eoff[j], e = P.walk_eoff[j + 1];
    if (P.stamp[j] != 0u) continue;
    for (uint32_t p = b + lane; p < e; p += LANES) {
      const uint32_t x = __ldg(&entry[p]);
      if (__ldg(&P.cnt[x]) < floor_gain || (cand && !cand[x])) continue;
      const uint32_t i = index[x];
      const uint32_t at = atomicAdd(&list[i].w, 1u);
      pairs[list[i].z + at] = make_uint4(j, x, i, at == 0 ? 1u : 0u);
    }
  }
}

// Picks in the greedy's order: gain down, element up; the first k of them as ids and gains.
// Eight lanes rank a pick against all of them from shared memory.  More than SORT_MAX picks are
// left to the radix sort.
constexpr int RANK_LANES = 8, RANK_THREADS = 128;
__global__ void __launch_bounds__(RANK_THREADS) k_peak_order(const uint32_t* __restrict__ out_u,
                                                             const uint32_t* __restrict__ out_gain,
                                                             const uint32_t* __restrict__ ctl,
                                                             const int32_t* __restrict__ uid, uint32_t k,
                                                             int64_t* __restrict__ ids,
                                                             uint32_t* __restrict__ gains) {
  constexpr uint32_t PICKS = RANK_THREADS / RANK_LANES;
  __shared__ unsigned long long key[SORT_MAX];
  const uint32_t n = ctl[PC_PICKS];
  if (n > SORT_MAX || blockIdx.x * PICKS >= n) return;
  for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) key[i] = peak_key(out_gain[i], out_u[i]);
  __syncthreads();
  const uint32_t i = blockIdx.x * PICKS + threadIdx.x / RANK_LANES;
  const unsigned long long mine = i < n ? key[i] : 0ull;
  uint32_t rank = 0;
#pragma unroll 4
  for (uint32_t j = threadIdx.x % RANK_LANES; j < n; j += RANK_LANES) rank += key[j] > mine ? 1u : 0u;
#pragma unroll
  for (int o = RANK_LANES / 2; o; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
  if (i < n && threadIdx.x % RANK_LANES == 0 && rank < k) {
    const uint32_t u = 0xFFFFFFFFu - (uint32_t)mine;
    ids[rank] = uid ? uid[u] : (int64_t)u;
    gains[rank] = (uint32_t)(mine >> 32);
  }
}

__global__ void k_flip(uint32_t* __restrict__ x, uint32_t n) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) x[i] = ~x[i];
}

__global__ void k_peak_emit(const uint32_t* __restrict__ u, const uint32_t* __restrict__ flipped_gain, uint32_t n,
                             const int32_t* __restrict__ uid, int64_t* __restrict__ ids,
                             uint32_t* __restrict__ gains) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    ids[i] = uid ? uid[u[i]] : (int64_t)u[i];
    gains[i] = ~flipped_gain[i];
  }
}

// The largest cluster (16 CTAs, else 8) that k_greedy_peaks can run on; 0: none.
int peak_cluster() {
  static const int cached = [] {
    const int want[2] = {16, 8};
    for (int c : want) {
      if (c > 8 &&
          cudaFuncSetAttribute(k_greedy_peaks, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        continue;
      }
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = c;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.gridDim = dim3(c);
      cfg.blockDim = dim3(1024);
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int clusters = 0;
      if (cudaOccupancyMaxActiveClusters(&clusters, k_greedy_peaks, &cfg) == cudaSuccess && clusters > 0) return c;
      cudaGetLastError();
    }
    return 0;
  }();
  return cached;
}

// Threads of a CTA.  Fewer warps meet at a barrier sooner, and have half the loads in flight and half
// the room for whole elements: 512 threads against 1,024 on 5.3 K walks 266 against 298 us (stopping
// rule query 677 against 730 us), 7-28 K walks of a pool 91-102 against 94-106, 55-222 K walks
// 107-143 against 103-137; 32 instances of 20 K walks at once 7.47 against 7.08 ms.  The line lies
// below those instances: side by side they share the SMs, and there the fewer warps cost more than the
// barriers gain, while 20-28 K walks alone gain at most a few us.
static unsigned peak_threads(int64_t walks) { return walks <= (1 << 14) ? 512 : 1024; }
uint64_t peak_room(int64_t walks) { return (uint64_t)peak_cluster() * peak_threads(walks) * OWN_PAIRS; }

// Counts by element id and walk offsets of walks [first, first + count), with no read back: the
// rest of the greedy takes sizes from the device.  M elements.
hsaw_status count_by_id(const Stream& st, bool edges, int64_t first, int64_t count, int64_t M, Cover& cv,
                        cudaStream_t s) {
  HSAW_TRY(cv.walk_eoff.ensure((size_t)count + 1, s));
  HSAW_TRY(cv.keys.ensure((size_t)M, s));
  HSAW_CK(cudaMemsetAsync(cv.keys.p, 0, (size_t)M * 4, s));
  const int32_t* el = edges ? st.edges.p : st.nodes.p;
  count_launch();
  k_count_elements<<<8 * sm_count(), 256, 0, s>>>(st.node_off.p, first, count, edges ? 1 : 0, el, cv.keys.p);
  HSAW_CK(cudaGetLastError());
  HSAW_TRY(walk_offsets(st, edges, first, count, cv, s));
  cv.by_id = true;
  cv.el = el;
  cv.from = st.node_off.p + first;
  cv.from_sub = edges ? first : 0;
  cv.elements = M;
  return HSAW_OK;
}

hsaw_status peak_greedy(Cover& cv, const uint8_t* cand, int32_t k, const PickBlock& out, uint32_t* host,
                        int32_t* rounds, bool* done, bool* copied, cudaStream_t s) {
  *done = *copied = false;
  int64_t* const ids = out.ids;
  uint32_t *const gains = out.gains, *const ctl = out.ctl, *const hist = out.work;
  static_assert(PC_WORDS == PickBlock::CTL && COUNT_BINS == PickBlock::WORK, "layout of the picks' block");
  // always the largest cluster: greedy and coverage on streams of 150-1,000 walks take 0.26-0.29
  // ms on 1 to 16 CTAs alike, on 2,500 walks 0.57, 0.41 and 0.35 ms on 1, 4 and 16, and more
  // beyond
  const int csize = peak_cluster();
  if (!csize) return HSAW_OK;
  const bool by_id = cv.by_id;
  const uint32_t U = (uint32_t)(by_id ? cv.elements : cv.unique), W = (uint32_t)cv.walks;
  const uint32_t most = std::min(U, W);  // a pick covers a walk of its own
  // room for the list and its pairs; a phase that needs more says so and is run again
  uint32_t list_cap = (uint32_t)std::min<uint64_t>(std::max<uint64_t>(16ull * k, 1ull << 15), 1ull << 20);
  uint32_t pair_cap = (uint32_t)std::min<uint64_t>(std::max<uint64_t>(256ull * k, 1ull << 18), 1ull << 22);
  uint32_t* const cnt = by_id ? cv.keys.p : cv.cnt.p;
  const int32_t* const uid = by_id ? nullptr : cv.uid.p;
  if (by_id) HSAW_TRY(cv.vals.ensure(U, s));  // list index of each listed element
  HSAW_TRY(cv.covered.ensure(W, s));
  HSAW_TRY(cv.partial.ensure(2 * (size_t)W, s));
  HSAW_TRY(cv.g_cnt.ensure((size_t)4 * most, s));  // picks, and room to sort them
  uint32_t* out_u = cv.g_cnt.p;
  uint32_t* out_gain = out_u + most;
  HSAW_CK(cudaMemsetAsync(cv.covered.p, 0, (size_t)W * 4, s));
  HSAW_CK(cudaMemsetAsync(ctl, 0, (PC_WORDS + COUNT_BINS) * 4, s));
  const bool log = getenv("HSAW_LOG_LAUNCHES") != nullptr;  // measurement aid
  cudaEvent_t ev[2] = {nullptr, nullptr};
  if (log) {
    cudaEventCreate(&ev[0]);
    cudaEventCreate(&ev[1]);
    cudaEventRecord(ev[0], s);
  }
  uint32_t h[PC_WORDS] = {0}, phases = 0, owned_phases = 0, unique = 0;
  PeakParams P = {};
  const uint64_t about = by_id ? cv.about : cv.entries;
  const uint32_t room = (uint32_t)peak_room(W), keep = (uint32_t)std::min<uint64_t>(peak_pairs(W, about, k), 0xF0000000u);
  bool again = false;  // the phase did not fit its list or pairs
  bool left = false;   // to the greedy that takes one pick at a time
  do {
    if (!again) {
      if (phases++) {  // the candidates below the last floor
        HSAW_CK(cudaMemsetAsync(hist, 0, COUNT_BINS * 4, s));
        if (h[PC_OWNED]) {
          count_launch();
          k_take_down<<<grid_for(W, 256, 8 * sm_count()), 256, 0, s>>>(P, W, P.round0);
          HSAW_CK(cudaGetLastError());
        }
      }
      count_launch();
      k_peak_hist<<<grid_for((U + 3) / 4, 512, 4 * sm_count()), 512, 0, s>>>(cnt, uid, cand, U, hist);
      HSAW_CK(cudaGetLastError());
      HSAW_CK(cudaMemsetAsync(cv.partial.p, 0, (size_t)W * 16, s));
    }
    if (again || phases > 1) HSAW_CK(cudaMemsetAsync(ctl + PC_LIST, 0, 2 * 4, s));
    HSAW_TRY(cv.peak_list.ensure(list_cap, s));
    HSAW_TRY(cv.g_list.ensure(list_cap, s));
    HSAW_TRY(cv.g_rng.ensure(list_cap, s));
    HSAW_TRY(cv.inv_ent.ensure(pair_cap, s));
    count_launch();
    k_peak_list<<<grid_for((U + 3) / 4, 512, 4 * sm_count()), 512, 0, s>>>(
        hist, (uint32_t)k, keep, peak_sparse_pairs(k), about, cnt, uid, cand, by_id ? nullptr : cv.inv_off.p, U, list_cap, cv.peak_list.p, cv.g_list.p,
        cv.g_rng.p, by_id ? cv.vals.p : nullptr, ctl);
    HSAW_CK(cudaGetLastError());
    P.pairs = cv.inv_ent.p;
    P.failed = cv.g_list.p;
    P.seen = cv.g_rng.p;
    P.cnt = cnt;
    P.walk_eoff = cv.walk_eoff.p;
    P.entry = by_id ? reinterpret_cast<const uint32_t*>(cv.el) : cv.entry_uidx.p;
    P.from = by_id ? cv.from : nullptr;
    P.from_sub = cv.from_sub;
    P.list_cap = list_cap;
    P.pair_cap = pair_cap;
    P.stamp = cv.covered.p;
    P.top[0] = cv.partial.p;
    P.top[1] = cv.partial.p + W;
    P.out_u = out_u;
    P.out_gain = out_gain;
    P.ctl = ctl;
    P.k = (uint32_t)k;
    P.round0 = h[PC_ROUNDS];
    P.max_rounds = most;  // a round makes a pick
    P.room = room;
    count_launch();
    if (!by_id)
      k_peak_pairs<<<4 * sm_count(), 256, 0, s>>>(cv.peak_list.p, cv.inv_walk.p, ctl, list_cap, pair_cap, cv.inv_ent.p);
    else if (cv.short_walks)
      k_walk_pairs<8><<<grid_for((size_t)W * 8, 256, 8 * sm_count()), 256, 0, s>>>(P, W, cand, cv.vals.p,
                                                                                  cv.peak_list.p, cv.inv_ent.p);
    else
      k_walk_pairs<32><<<grid_for((size_t)W * 32, 256, 8 * sm_count()), 256, 0, s>>>(P, W, cand, cv.vals.p,
                                                                                    cv.peak_list.p, cv.inv_ent.p);
    HSAW_CK(cudaGetLastError());
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = csize;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(csize);
    cfg.blockDim = dim3(peak_threads(W));
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    count_launch();
    HSAW_CK(cudaLaunchKernelEx(&cfg, k_greedy_peaks, P));
    count_launch();
    k_peak_order<<<SORT_MAX * RANK_LANES / RANK_THREADS, RANK_THREADS, 0, s>>>(out_u, out_gain, ctl, uid, (uint32_t)k, ids, gains);
    HSAW_CK(cudaGetLastError());
    // picks and control words come back in one copy
    HSAW_CK(cudaMemcpyAsync(host, out.ids, PickBlock::copied_words(k) * 4, cudaMemcpyDeviceToHost, s));
    HSAW_CK(cudaStreamSynchronize(s));
    std::memcpy(h, host + (out.ctl - reinterpret_cast<uint32_t*>(out.ids)), sizeof(h));
    if (h[PC_STUCK]) return fail(HSAW_E_DEVICE, "greedy: a round made no pick");
    if (phases == 1) unique = h[PC_TOTAL];
    again = h[PC_LIST] > pair_cap || h[PC_LIST + 1] > list_cap;
    left = h[PC_LIST] > std::max(h[PC_KEEP], room) || (!again && h[PC_LEFT]);
    if (left) break;
    if (again) {
      pair_cap = std::max(pair_cap, h[PC_LIST]);
      list_cap = std::max(list_cap, h[PC_LIST + 1]);
    } else {
      owned_phases += h[PC_OWNED];
    }
  } while (again || (h[PC_PICKS] < (uint32_t)k && h[PC_FLOOR] > 1));
  if (left) {
    if (log) {
      fprintf(stderr, "hsaw: k_greedy_peaks left rounds=%u phases=%u pairs=%u picks=%u walks=%lld\n", h[PC_ROUNDS], phases,
              h[PC_LIST], h[PC_PICKS], (long long)cv.walks);
      cudaEventDestroy(ev[0]);
      cudaEventDestroy(ev[1]);
    }
    return HSAW_OK;
  }
  const uint32_t made = h[PC_PICKS], kept = std::min<uint32_t>(made, (uint32_t)k);
  if (made > SORT_MAX) {  // by element, then (stable) by gain downwards
    uint32_t *k1 = out_u, *v1 = out_gain, *k2 = out_u + 2 * (size_t)most, *v2 = k2 + most;
    bool alt = false;
    HSAW_TRY(radix_sort_pairs(k1, v1, k2, v2, made, bit_width(U - 1), s, &alt));
    uint32_t *key = alt ? v2 : v1, *val = alt ? k2 : k1, *key2 = alt ? v1 : v2, *val2 = alt ? k1 : k2;
    count_launch();
    k_flip<<<grid_for(made, 256, 4096), 256, 0, s>>>(key, made);
    HSAW_CK(cudaGetLastError());
    HSAW_TRY(radix_sort_pairs(key, val, key2, val2, made, 32, s, &alt));
    count_launch();
    k_peak_emit<<<grid_for(kept, 256, 1024), 256, 0, s>>>(alt ? val2 : val, alt ? key2 : key, kept, uid, ids, gains);
    HSAW_CK(cudaGetLastError());
  }
  if (log) {
    // the kernel and what is its own, then the fields that the one-pick greedies' records have too
    uint32_t entries = 0;
    cudaMemcpyAsync(&entries, cv.walk_eoff.p + W, 4, cudaMemcpyDeviceToHost, s);
    cudaEventRecord(ev[1], s);
    cudaEventSynchronize(ev[1]);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ev[0], ev[1]);
    fprintf(stderr,
            "hsaw: k_greedy_peaks rounds=%u phases=%u owned=%u pairs=%u made=%u by_id=%d ms=%.3f, as k_greedy_cluster "
            "walks=%lld entries=%u unique=%u cluster=%d gshift=0 k=%d picks=%u spread=0\n",
            h[PC_ROUNDS], phases, owned_phases, h[PC_LIST], made, by_id ? 1 : 0, ms, (long long)cv.walks, entries, unique,
            csize, k, kept);
    cudaEventDestroy(ev[0]);
    cudaEventDestroy(ev[1]);
  }
  *rounds = (int32_t)kept;
  *done = true;
  *copied = made <= SORT_MAX;
  return HSAW_OK;
}

}  // namespace hsaw
