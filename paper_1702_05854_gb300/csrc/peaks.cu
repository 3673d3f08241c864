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
// 7 K-222 K R-MAT 18 walks, 1.1-2.0 -> 0.11-0.18 ms; k = 100 nodes of 8 K with random coins,
// 5.3 K walks, 0.59 -> 0.35 ms (33 rounds).  Taking one gain level a round instead (the picks of
// a level are an independent set) needed 9-104 rounds there and measured 0.15-1.1 ms.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

#include "solver.cuh"

namespace hsaw {

namespace cg = cooperative_groups;

namespace {

constexpr uint32_t NOT_CANDIDATE = 0x80000000u;  // bit 31 of a running count
constexpr uint32_t COUNT_BINS = 4096;            // counts from COUNT_BINS - 1 up share the last bin
constexpr uint32_t SORT_MAX = 4096;              // picks ordered by one block

// ctl words of a run; the list's length (high half) and its pairs (low half) grow together in
// one 64-bit word
enum { PC_PICKS = 0, PC_FLOOR = 1, PC_GAIN = 2, PC_ROUNDS = 3, PC_STUCK = 4, PC_LIST = 6 /* 64 bits */, PC_WORDS = 16 };

// A walk of a listed element: {walk, element, index in the list, 1 for the element's first}.
using Pair = uint4;

struct PeakParams {
  const Pair* pairs;
  uint32_t* failed;            // per listed element: the last round in which it was no peak
  uint2* seen;                 // and the last round that looked at it, with its count then
  uint32_t* cnt;               // running counts | NOT_CANDIDATE
  const uint32_t* walk_eoff;   // per walk: its entries of entry_uidx
  const uint32_t* entry_uidx;
  uint32_t* stamp;             // per walk: 0, or the round that covered it
  unsigned long long* top[2];  // per walk, by the round's parity: the largest key signed on it
  uint32_t* out_u;
  uint32_t* out_gain;
  uint32_t* ctl;
  uint32_t k;
  uint32_t round0;             // rounds of earlier phases
  uint32_t max_rounds;
};

__device__ __forceinline__ unsigned long long peak_key(uint32_t count, uint32_t u) {
  return ((unsigned long long)count << 32) | (0xFFFFFFFFu - u);
}

// The counts of the entries [range.x, range.y) of the walks of the lanes in `mine` go down by
// one, the whole warp on each.  Four walks' entries are in flight at a time.
__device__ __forceinline__ void take_down(const PeakParams& P, unsigned mine, uint2 range, int lane) {
  while (mine) {
    uint32_t b[4], e[4], x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int src = mine ? __ffs(mine) - 1 : 0;
      b[j] = __shfl_sync(0xffffffffu, range.x, src) + lane;
      e[j] = mine ? __shfl_sync(0xffffffffu, range.y, src) : 0u;
      mine &= mine - 1;
      x[j] = b[j] < e[j] ? __ldg(&P.entry_uidx[b[j]]) : 0u;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (b[j] < e[j]) atomicSub(&P.cnt[x[j]], 1u);
      for (uint32_t p = b[j] + 32; p < e[j]; p += 32) atomicSub(&P.cnt[__ldg(&P.entry_uidx[p])], 1u);
    }
  }
}

}  // namespace

// One cluster, a thread per (element, walk) pair of the list; counts, stamps and
// keys in global memory (L2).  Bound by latency: three barriers a round, two or three
// dependent L2 reads before each.
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
  const uint32_t stripe = (n + 31) / 32;
  const uint32_t floor_gain = __ldcg(&P.ctl[PC_FLOOR]);
  uint32_t picks = 0, g = 0, r = P.round0;
  bool stuck = false;
  for (;;) {
    ++r;
    picks = __ldcg(&P.ctl[PC_PICKS]);
    // 1. elements at or above the floor sign their keys on their uncovered walks; the largest
    // count
    unsigned long long* const top = P.top[r & 1];
    uint32_t m = 0;
#pragma unroll 4
    for (uint32_t i = gtid; i < n; i += threads) {
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
      take_down(P, __ballot_sync(FULL, fresh), range, lane);
    }
    cluster.sync();
  }
  cluster.sync();  // no CTA leaves while a peer may still write its shared memory
  if (gtid == 0) {
    P.ctl[PC_GAIN] = g;
    P.ctl[PC_ROUNDS] = r;
    P.ctl[PC_STUCK] = stuck ? 1u : 0u;
  }
}

// Histogram of the running counts of the candidates (counts from 1 up).  first: the counts
// are taken from cnt and the candidate mask first.  Most R-MAT walk elements occur once or
// twice: those two bins are counted by ballot, not by atomics on one word.
__global__ void __launch_bounds__(512) k_peak_hist(bool first, const int32_t* __restrict__ uid,
                                                    const uint32_t* __restrict__ cnt, const uint8_t* __restrict__ cand,
                                                    uint32_t U, uint32_t* __restrict__ work,
                                                    uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[COUNT_BINS];
  for (uint32_t i = threadIdx.x; i < COUNT_BINS; i += blockDim.x) h[i] = 0;
  __syncthreads();
  uint32_t one = 0, two = 0;
  for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < U; u += gridDim.x * blockDim.x) {
    uint32_t v;
    if (first) {
      v = cnt[u] | ((cand && !cand[uid[u]]) ? NOT_CANDIDATE : 0u);
      work[u] = v;
    } else {
      v = work[u];
    }
    if (v & NOT_CANDIDATE) continue;
    if (v == 1) ++one;
    else if (v == 2) ++two;
    else if (v) atomicAdd(&h[min(v, COUNT_BINS - 1)], 1u);
  }
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
// inv_walk, its first pair}, in no order.  Every listed element may be picked and covered, and
// is read in each round, so the list holds half as many again as the k picks wanted (1,000
// R-MAT edge picks came from the first 1,100-1,500) and a few, and more while it is short.
__global__ void __launch_bounds__(512) k_peak_list(const uint32_t* __restrict__ hist, uint32_t k,
                                                   const uint32_t* __restrict__ work,
                                                   const uint32_t* __restrict__ inv_off, uint32_t U,
                                                   uint4* __restrict__ list, uint32_t* __restrict__ failed,
                                                   uint2* __restrict__ seen, uint32_t* __restrict__ ctl) {
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
  const uint32_t want = (uint32_t)min((unsigned long long)total, (unsigned long long)k + k / 2 + 64);
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
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl[PC_FLOOR] = floor_gain;
  for (uint32_t u0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; u0 < U; u0 += gridDim.x * blockDim.x) {
    const uint32_t u = u0 + lane;
    const uint32_t v = u < U ? work[u] : 0u;
    const bool in = !(v & NOT_CANDIDATE) && v >= floor_gain;
    const unsigned b = __ballot_sync(0xffffffffu, in);
    if (!b) continue;
    const uint32_t q0 = in ? inv_off[u] : 0u, len = in ? inv_off[u + 1] - q0 : 0u;
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
    if (in) {
      const uint32_t i = (uint32_t)(at >> 32) + __popc(b & ((1u << lane) - 1u));
      list[i] = make_uint4(u, q0, (uint32_t)at + (uint32_t)(inc - len), 0u);
      failed[i] = 0u;
      seen[i] = make_uint2(0u, 0u);
    }
  }
}

// The list's (element, walk) pairs, element by element.
__global__ void __launch_bounds__(256) k_peak_pairs(const uint4* __restrict__ list, const uint32_t* __restrict__ inv_walk,
                                                    const uint32_t* __restrict__ ctl, Pair* __restrict__ pairs) {
  const uint32_t n = ctl[PC_LIST], elements = ctl[PC_LIST + 1];
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

// Picks in the greedy's order: gain down, element up (bitonic sort in one block); the first k
// of them as ids and gains.  More than SORT_MAX picks are left to the radix sort.
__global__ void __launch_bounds__(1024) k_peak_order(const uint32_t* __restrict__ out_u,
                                                      const uint32_t* __restrict__ out_gain,
                                                      const uint32_t* __restrict__ ctl,
                                                      const int32_t* __restrict__ uid, uint32_t k,
                                                      int64_t* __restrict__ ids, uint32_t* __restrict__ gains) {
  __shared__ unsigned long long key[SORT_MAX];
  const uint32_t n = ctl[PC_PICKS];
  if (n > SORT_MAX) return;
  uint32_t size = 32;
  while (size < n) size *= 2;
  for (uint32_t i = threadIdx.x; i < size; i += blockDim.x)
    key[i] = i < n ? ((unsigned long long)(~out_gain[i]) << 32) | out_u[i] : ~0ull;
  for (uint32_t span = 2; span <= size; span *= 2)
    for (uint32_t step = span / 2; step; step /= 2) {
      __syncthreads();
      for (uint32_t t = threadIdx.x; t < size / 2; t += blockDim.x) {
        const uint32_t i = 2 * t - (t & (step - 1)), j = i + step;
        const unsigned long long a = key[i], b = key[j];
        if ((a > b) == ((i & span) == 0)) {
          key[i] = b;
          key[j] = a;
        }
      }
    }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < min(n, k); i += blockDim.x) {
    ids[i] = uid[(uint32_t)key[i]];
    gains[i] = ~(uint32_t)(key[i] >> 32);
  }
}

__global__ void k_flip(uint32_t* __restrict__ x, uint32_t n) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) x[i] = ~x[i];
}

__global__ void k_peak_emit(const uint32_t* __restrict__ u, const uint32_t* __restrict__ flipped_gain, uint32_t n,
                             const int32_t* __restrict__ uid, int64_t* __restrict__ ids,
                             uint32_t* __restrict__ gains) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    ids[i] = uid[u[i]];
    gains[i] = ~flipped_gain[i];
  }
}

// The largest cluster (16 CTAs, else 8) that k_greedy_peaks can run on; 0: none.
static int peak_cluster() {
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

hsaw_status peak_greedy(Cover& cv, const uint8_t* cand, int32_t k, int64_t* ids, uint32_t* gains, int32_t* rounds,
                        bool* done, cudaStream_t s) {
  *done = false;
  const int largest = peak_cluster();
  if (!largest) return HSAW_OK;
  const uint32_t U = (uint32_t)cv.unique, W = (uint32_t)cv.walks;
  const uint32_t most = std::min(U, W);  // a pick covers a walk of its own
  // always the largest cluster: greedy and coverage on streams of 150-1,000 walks take 0.26-0.29
  // ms on 1 to 16 CTAs alike, on 2,500 walks 0.57, 0.41 and 0.35 ms on 1, 4 and 16, and more
  // beyond
  const uint32_t csize = (uint32_t)largest;
  HSAW_TRY(cv.cnt_work.ensure(U, s));
  HSAW_TRY(cv.peak_list.ensure(U, s));
  HSAW_TRY(cv.inv_ent.ensure((size_t)cv.entries, s));  // pairs
  HSAW_TRY(cv.g_list.ensure(U, s));
  HSAW_TRY(cv.g_rng.ensure(U, s));
  HSAW_TRY(cv.covered.ensure(W, s));
  HSAW_TRY(cv.partial.ensure(2 * (size_t)W, s));
  HSAW_TRY(cv.g_cnt.ensure((size_t)4 * most + COUNT_BINS + PC_WORDS + 2, s));  // picks (and room to sort), bins, ctl
  uint32_t* out_u = cv.g_cnt.p;
  uint32_t* out_gain = out_u + most;
  uint32_t* hist = out_u + ((4 * (size_t)most + 1) & ~(size_t)1);  // ctl holds a 64-bit word
  uint32_t* ctl = hist + COUNT_BINS;
  HSAW_CK(cudaMemsetAsync(cv.covered.p, 0, (size_t)W * 4, s));
  HSAW_CK(cudaMemsetAsync(hist, 0, (COUNT_BINS + PC_WORDS) * 4, s));
  const bool log = getenv("HSAW_LOG_LAUNCHES") != nullptr;  // measurement aid
  cudaEvent_t ev[2] = {nullptr, nullptr};
  if (log) {
    cudaEventCreate(&ev[0]);
    cudaEventCreate(&ev[1]);
    cudaEventRecord(ev[0], s);
  }
  uint32_t h[PC_WORDS] = {0}, phases = 0;
  do {
    if (phases++) {  // every pick down to the floor is made: the candidates below it
      HSAW_CK(cudaMemsetAsync(hist, 0, COUNT_BINS * 4, s));
      HSAW_CK(cudaMemsetAsync(ctl + PC_LIST, 0, 2 * 4, s));
    }
    HSAW_CK(cudaMemsetAsync(cv.partial.p, 0, (size_t)W * 16, s));
    count_launch();
    k_peak_hist<<<grid_for(U, 512, 4 * sm_count()), 512, 0, s>>>(phases == 1, cv.uid.p, cv.cnt.p, cand, U, cv.cnt_work.p,
                                                                hist);
    HSAW_CK(cudaGetLastError());
    count_launch();
    k_peak_list<<<grid_for(U, 512, 4 * sm_count()), 512, 0, s>>>(hist, (uint32_t)k, cv.cnt_work.p, cv.inv_off.p, U,
                                                                cv.peak_list.p, cv.g_list.p, cv.g_rng.p, ctl);
    HSAW_CK(cudaGetLastError());
    count_launch();
    k_peak_pairs<<<4 * sm_count(), 256, 0, s>>>(cv.peak_list.p, cv.inv_walk.p, ctl, cv.inv_ent.p);
    HSAW_CK(cudaGetLastError());
    PeakParams P;
    P.pairs = cv.inv_ent.p;
    P.failed = cv.g_list.p;
    P.seen = cv.g_rng.p;
    P.cnt = cv.cnt_work.p;
    P.walk_eoff = cv.walk_eoff.p;
    P.entry_uidx = cv.entry_uidx.p;
    P.stamp = cv.covered.p;
    P.top[0] = cv.partial.p;
    P.top[1] = cv.partial.p + W;
    P.out_u = out_u;
    P.out_gain = out_gain;
    P.ctl = ctl;
    P.k = (uint32_t)k;
    P.round0 = h[PC_ROUNDS];
    P.max_rounds = most;  // a round makes a pick
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = csize;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(csize);
    cfg.blockDim = dim3(1024);
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    count_launch();
    HSAW_CK(cudaLaunchKernelEx(&cfg, k_greedy_peaks, P));
    count_launch();
    k_peak_order<<<1, 1024, 0, s>>>(out_u, out_gain, ctl, cv.uid.p, (uint32_t)k, ids, gains);
    HSAW_CK(cudaGetLastError());
    HSAW_CK(cudaMemcpyAsync(h, ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
    HSAW_CK(cudaStreamSynchronize(s));
    if (h[PC_STUCK]) return fail(HSAW_E_DEVICE, "greedy: a round made no pick");
  } while (h[PC_PICKS] < (uint32_t)k && h[PC_FLOOR] > 1);
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
    k_peak_emit<<<grid_for(kept, 256, 1024), 256, 0, s>>>(alt ? val2 : val, alt ? key2 : key, kept, cv.uid.p, ids, gains);
    HSAW_CK(cudaGetLastError());
  }
  if (log) {
    // a greedy on one cluster with counts in global memory, like k_greedy_cluster, whose record
    // this is
    cudaEventRecord(ev[1], s);
    cudaEventSynchronize(ev[1]);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ev[0], ev[1]);
    fprintf(stderr,
            "hsaw: k_greedy_cluster walks=%lld entries=%lld unique=%u cluster=%u gshift=0 k=%d picks=%u spread=0 "
            "rounds=%u phases=%u pairs=%u made=%u ms=%.3f\n",
            (long long)cv.walks, (long long)cv.entries, U, csize, k, kept, h[PC_ROUNDS], phases, h[PC_LIST], made, ms);
    cudaEventDestroy(ev[0]);
    cudaEventDestroy(ev[1]);
  }
  *rounds = (int32_t)kept;
  *done = true;
  return HSAW_OK;
}

}  // namespace hsaw
