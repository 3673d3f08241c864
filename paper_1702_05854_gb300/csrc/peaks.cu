// Greedy max-coverage (Alg. 4 / Alg. 7) one gain level at a time.
//
// While the largest marginal gain is g, the greedy takes the elements of gain g in increasing
// id, each unless a pick before it covered one of its walks: counts only fall, so nothing
// joins the level while it lasts, and what a pick touches leaves it.  The picks of a level
// are therefore the lexicographically first maximal independent set of its elements, two of
// them adjacent when an uncovered walk holds both.  That set is found in rounds: an element
// that is the smallest candidate on each of its uncovered walks is a pick whatever the others
// do, so all such elements are taken at once, their walks covered and their elements' counts
// taken down, and the next round looks at what is left of the level.  Most levels take one
// round, and k picks fall on few levels: 1,000 picks on 3-104 levels over 7 K-450 K R-MAT
// walks (100 picks on 43-94 levels where a few nodes hold most walks).
//
// The greedy with one pick per barrier (cover.cu) is bound by latency, 3.4-8 us a pick.  Whole
// calls against it: greedy and coverage on 150 K R-MAT 22 walks, k = 1000, 6.99 -> 2.03 ms; a
// pooled stopping-rule query on R-MAT 18, k = 300, six greedies, 15.5 -> 8.0 ms.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

#include "solver.cuh"

namespace hsaw {

namespace cg = cooperative_groups;

namespace {

constexpr uint32_t NOT_CANDIDATE = 0x80000000u;  // bit 31 of a running count
constexpr uint32_t LEVEL_BINS = 4096;            // counts from LEVEL_BINS - 1 up share the last bin
constexpr uint32_t SORT_MAX = 4096;              // picks ordered by one block
constexpr uint32_t LANE_GAIN = 8;                // up to this gain a lane walks a candidate's list by itself

// ctl words of a run
enum { LC_PICKS = 0, LC_QUEUE = 1 /* two words */, LC_LIST = 3, LC_FLOOR = 4, LC_GAIN = 5, LC_ROUNDS = 6, LC_LEVELS = 7,
       LC_SINGLE = 8, LC_STUCK = 9, LC_WORDS = 16 };

struct LevelParams {
  const uint32_t* list;        // the phase's elements: every candidate with a count of at least ctl[LC_FLOOR]
  uint32_t* cnt;               // running counts | NOT_CANDIDATE
  const uint32_t* inv_off;     // per element: its entries of inv_walk
  const uint32_t* inv_walk;
  const uint32_t* walk_eoff;   // per walk: its entries of entry_uidx
  const uint32_t* entry_uidx;
  uint32_t* stamp;             // per walk: 0, or the round that covered it
  unsigned long long* owner;   // per walk: (~round << 32) | smallest candidate of that round
  uint2* queue;                // walks to cover this round, as entry ranges
  uint32_t* out_u;
  uint32_t* out_gain;
  uint32_t* ctl;
  uint32_t k;
  uint32_t round0;             // rounds of earlier phases
  uint32_t max_rounds;
};

// The counts of the entries [e0, e1) of each of the warp's n <= 32 walks (lane i holds walk
// i's range) go down by one.  Four walks' entries are in flight at a time.
__device__ __forceinline__ void take_down(const LevelParams& P, uint2 range, uint32_t n, int lane) {
  for (uint32_t i = 0; i < n; i += 4) {
    uint32_t b[4], e[4], x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int src = (int)min(i + j, 31u);
      b[j] = __shfl_sync(0xffffffffu, range.x, src) + lane;
      e[j] = __shfl_sync(0xffffffffu, range.y, src);
      if (i + j >= n) e[j] = 0;
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

// One cluster; counts, stamps and owners in global memory (L2).  Bound by latency: a round
// with one candidate is two barriers, any other four, each with two to four dependent L2
// reads before it.
__global__ void __launch_bounds__(1024, 1) k_greedy_levels(const __grid_constant__ LevelParams P) {
  __shared__ uint32_t s_max[32], s_cnt[32], s_u[32];
  __shared__ uint4 slot[2][16];  // by round parity, per CTA: largest count, elements that have it, the smallest of them
  const unsigned FULL = 0xffffffffu;
  cg::cluster_group cluster = cg::this_cluster();
  const uint32_t rank = cluster.block_rank(), C = cluster.num_blocks();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t gtid = rank * blockDim.x + threadIdx.x, threads = C * blockDim.x;
  const uint32_t gwarp = gtid >> 5, warps = threads >> 5;
  auto barrier = [&] {
    if (C == 1) __syncthreads();
    else cluster.sync();
  };
  const uint32_t n = __ldcg(&P.ctl[LC_LIST]), floor_gain = __ldcg(&P.ctl[LC_FLOOR]);
  uint32_t picks = __ldcg(&P.ctl[LC_PICKS]);
  uint32_t last = 0xFFFFFFFFu, g = 0, levels = 0, single = 0, shared = 0, r = P.round0;
  bool stuck = false;
  for (;;) {
    ++r;
    // 1. the largest count and how many elements have it
    uint32_t m = 0, c = 0, mu = 0xFFFFFFFFu;
    for (uint32_t i = gtid; i < n; i += threads) {
      const uint32_t u = __ldg(&P.list[i]), v = __ldcg(&P.cnt[u]);
      if (v > m) {
        m = v;
        c = 0;
        mu = 0xFFFFFFFFu;
      }
      if (v == m) {
        ++c;
        mu = min(mu, u);
      }
    }
    {
      const uint32_t wm = __reduce_max_sync(FULL, m);
      const uint32_t wc = __reduce_add_sync(FULL, m == wm ? c : 0u);
      const uint32_t wu = __reduce_min_sync(FULL, m == wm ? mu : 0xFFFFFFFFu);
      if (lane == 0) {
        s_max[w] = wm;
        s_cnt[w] = wc;
        s_u[w] = wu;
      }
    }
    __syncthreads();
    if (w == 0) {
      const uint32_t bm = __reduce_max_sync(FULL, s_max[lane]);
      const uint32_t bc = __reduce_add_sync(FULL, s_max[lane] == bm ? s_cnt[lane] : 0u);
      const uint32_t bu = __reduce_min_sync(FULL, s_max[lane] == bm ? s_u[lane] : 0xFFFFFFFFu);
      if (lane < (int)C) *cluster.map_shared_rank(&slot[r & 1][rank], lane) = make_uint4(bm, bc, bu, 0u);
    }
    barrier();
    uint32_t total, u1;
    {
      const uint4 s = lane < (int)C ? slot[r & 1][lane] : make_uint4(0u, 0u, 0xFFFFFFFFu, 0u);
      g = __reduce_max_sync(FULL, s.x);
      total = __reduce_add_sync(FULL, s.x == g ? s.y : 0u);
      u1 = __reduce_min_sync(FULL, s.x == g ? s.z : 0xFFFFFFFFu);
    }
    // the same decision in every warp: nothing left to gain, the phase's elements do not hold
    // the whole level, or enough picks and the last level complete
    if (g == 0 || g < floor_gain || (picks >= P.k && g < last)) break;
    if (r - P.round0 > P.max_rounds) {
      stuck = true;
      break;
    }
    if (g != last) ++levels;
    last = g;
    if (total == 1) {
      // 2a. the only candidate: the whole cluster covers its walks
      ++single;
      const uint32_t q0 = __ldg(&P.inv_off[u1]), q1 = __ldg(&P.inv_off[u1 + 1]);
      const uint32_t per = min(32u, (q1 - q0 + warps - 1) / warps);
      for (uint32_t q = q0 + gwarp * per; q < q1; q += warps * per) {
        const uint32_t have = min(per, q1 - q);
        uint2 range = make_uint2(0u, 0u);
        if (lane < (int)have) {
          const uint32_t j = __ldg(&P.inv_walk[q + lane]);
          const uint2 e = make_uint2(__ldg(&P.walk_eoff[j]), __ldg(&P.walk_eoff[j + 1]));
          if (__ldcg(&P.stamp[j]) == 0u) {
            P.stamp[j] = r;
            range = e;
          }
        }
        take_down(P, range, have, lane);
      }
      if (gtid == 0) {
        P.out_u[picks] = u1;
        P.out_gain[picks] = g;
        P.ctl[LC_PICKS] = picks + 1;
      }
      ++picks;
      barrier();
      continue;
    }
    // 2b. every candidate signs its uncovered walks; the smallest candidate owns the walk
    const unsigned long long tag = (unsigned long long)(~r) << 32;
    auto sign = [&](uint32_t e, uint32_t at, uint32_t step) {
      const uint32_t q1 = __ldg(&P.inv_off[e + 1]);
      for (uint32_t q = __ldg(&P.inv_off[e]) + at; q < q1; q += step) {
        const uint32_t j = __ldg(&P.inv_walk[q]);
        if (__ldcg(&P.stamp[j]) == 0u) atomicMin(&P.owner[j], tag | e);
      }
    };
    // owns every uncovered walk of its list (walks covered earlier in this round count: the
    // pick that covered one of them owns it)
    auto owns = [&](uint32_t e, uint32_t at, uint32_t step) {
      const uint32_t q1 = __ldg(&P.inv_off[e + 1]);
      bool ok = true;
      for (uint32_t q = __ldg(&P.inv_off[e]) + at; ok && q < q1; q += step) {
        const uint32_t j = __ldg(&P.inv_walk[q]);
        const uint32_t st = __ldcg(&P.stamp[j]);
        if (st == 0u || st == r) ok = (uint32_t)__ldcg(&P.owner[j]) == e;
      }
      return ok;
    };
    auto each = [&](auto&& body) {  // body(element, is a candidate): per lane, in step
      for (uint32_t i0 = gwarp * 32; i0 < n; i0 += threads) {
        const uint32_t i = i0 + lane;
        const uint32_t u = i < n ? __ldg(&P.list[i]) : 0u;
        body(u, i < n && __ldcg(&P.cnt[u]) == g);
      }
    };
    if (g <= LANE_GAIN) {
      each([&](uint32_t u, bool is) {
        if (is) sign(u, 0, 1);
      });
    } else {
      each([&](uint32_t u, bool is) {
        for (unsigned todo = __ballot_sync(FULL, is); todo; todo &= todo - 1)
          sign(__shfl_sync(FULL, u, __ffs(todo) - 1), lane, 32);
      });
    }
    barrier();
    // 3. candidates that own all their uncovered walks are picks; those walks (g each) are
    // stamped and queued
    uint32_t* const queued = &P.ctl[LC_QUEUE + (shared & 1)];  // by turns; the other one is cleared below
    ++shared;
    if (g <= LANE_GAIN) {
      each([&](uint32_t u, bool is) {
        if (!is || !owns(u, 0, 1)) return;
        const uint32_t pos = atomicAdd(&P.ctl[LC_PICKS], 1u);
        P.out_u[pos] = u;
        P.out_gain[pos] = g;
        uint32_t at = atomicAdd(queued, g);
        const uint32_t q1 = __ldg(&P.inv_off[u + 1]);
        for (uint32_t q = __ldg(&P.inv_off[u]); q < q1; ++q) {
          const uint32_t j = __ldg(&P.inv_walk[q]);
          if (__ldcg(&P.stamp[j]) != 0u) continue;
          P.stamp[j] = r;
          P.queue[at++] = make_uint2(__ldg(&P.walk_eoff[j]), __ldg(&P.walk_eoff[j + 1]));
        }
      });
    } else {
      each([&](uint32_t u, bool is) {
        for (unsigned todo = __ballot_sync(FULL, is); todo; todo &= todo - 1) {
          const uint32_t e = __shfl_sync(FULL, u, __ffs(todo) - 1);
          if (!__all_sync(FULL, owns(e, lane, 32))) continue;
          uint32_t at = 0;
          if (lane == 0) {
            const uint32_t pos = atomicAdd(&P.ctl[LC_PICKS], 1u);
            P.out_u[pos] = e;
            P.out_gain[pos] = g;
            at = atomicAdd(queued, g);
          }
          at = __shfl_sync(FULL, at, 0);
          const uint32_t q1 = __ldg(&P.inv_off[e + 1]);
          for (uint32_t q = __ldg(&P.inv_off[e]); q < q1; q += 32) {
            bool fresh = false;
            uint32_t j = 0;
            if (q + lane < q1) {
              j = __ldg(&P.inv_walk[q + lane]);
              fresh = __ldcg(&P.stamp[j]) == 0u;
            }
            const unsigned b = __ballot_sync(FULL, fresh);
            if (fresh) {
              P.stamp[j] = r;
              P.queue[at + __popc(b & ((1u << lane) - 1u))] = make_uint2(__ldg(&P.walk_eoff[j]),
                                                                         __ldg(&P.walk_eoff[j + 1]));
            }
            at += __popc(b);
          }
        }
      });
    }
    barrier();
    // 4. the queued walks' elements lose one each
    picks = __ldcg(&P.ctl[LC_PICKS]);
    const uint32_t nq = __ldcg(queued);
    if (gtid == 0) P.ctl[LC_QUEUE + (shared & 1)] = 0u;
    const uint32_t per = min(32u, (nq + warps - 1) / warps);
    for (uint32_t q = gwarp * per; q < nq; q += warps * per) {
      const uint32_t have = min(per, nq - q);
      const uint2 range = lane < (int)have ? __ldcg(&P.queue[q + lane]) : make_uint2(0u, 0u);
      take_down(P, range, have, lane);
    }
    barrier();
  }
  if (C > 1) cluster.sync();  // no CTA leaves while a peer may still read or write its shared memory
  if (gtid == 0) {
    P.ctl[LC_GAIN] = g;
    P.ctl[LC_ROUNDS] = r;
    P.ctl[LC_LEVELS] += levels;
    P.ctl[LC_SINGLE] += single;
    P.ctl[LC_STUCK] = stuck ? 1u : 0u;
    P.ctl[LC_QUEUE] = P.ctl[LC_QUEUE + 1] = 0u;
  }
}

// Histogram of the running counts of the candidates (counts from 1 up).  first: the counts
// are taken from cnt and the candidate mask first.  Most R-MAT walk elements occur once or
// twice: those two bins are counted by ballot, not by atomics on one word.
__global__ void __launch_bounds__(512) k_level_hist(bool first, const int32_t* __restrict__ uid,
                                                    const uint32_t* __restrict__ cnt, const uint8_t* __restrict__ cand,
                                                    uint32_t U, uint32_t* __restrict__ work,
                                                    uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[LEVEL_BINS];
  for (uint32_t i = threadIdx.x; i < LEVEL_BINS; i += blockDim.x) h[i] = 0;
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
    else if (v) atomicAdd(&h[min(v, LEVEL_BINS - 1)], 1u);
  }
  one = __reduce_add_sync(0xffffffffu, one);
  two = __reduce_add_sync(0xffffffffu, two);
  if ((threadIdx.x & 31) == 0) {
    if (one) atomicAdd(&h[1], one);
    if (two) atomicAdd(&h[2], two);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < LEVEL_BINS; i += blockDim.x)
    if (h[i]) atomicAdd(&hist[i], h[i]);
}

// The phase's floor: the smallest count that at most `cap` candidates reach, or the largest
// count there is; and the list of the candidates that reach it, in no order.
__global__ void __launch_bounds__(512) k_level_list(const uint32_t* __restrict__ hist, uint32_t cap,
                                                    const uint32_t* __restrict__ work, uint32_t U,
                                                    uint32_t* __restrict__ list, uint32_t* __restrict__ ctl) {
  constexpr uint32_t PER = LEVEL_BINS / 512;
  __shared__ uint32_t sums[16], s_floor, s_top;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    s_floor = LEVEL_BINS;
    s_top = 0;
  }
  // thread t holds the bins (LEVEL_BINS - 1 - t PER) downwards, so an inclusive scan over
  // the threads gives the candidates at or above a bin
  const uint32_t hi = LEVEL_BINS - 1 - threadIdx.x * PER;
  uint32_t own[PER], sum = 0;
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) sum += own[i] = hist[hi - i];
  uint32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) sums[w] = inc;
  __syncthreads();
  uint32_t above = inc - sum;
  for (int i = 0; i < w; ++i) above += sums[i];
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    const uint32_t bin = hi - i;
    above += own[i];
    if (bin >= 1) {
      if (above <= cap) atomicMin(&s_floor, bin);
      if (own[i]) atomicMax(&s_top, bin);
    }
  }
  __syncthreads();
  const uint32_t floor_gain = max(1u, min(s_floor, s_top));
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl[LC_FLOOR] = floor_gain;
  for (uint32_t u0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; u0 < U; u0 += gridDim.x * blockDim.x) {
    const uint32_t u = u0 + lane;
    const uint32_t v = u < U ? work[u] : 0u;
    const bool in = !(v & NOT_CANDIDATE) && v >= floor_gain;
    const unsigned b = __ballot_sync(0xffffffffu, in);
    if (!b) continue;
    uint32_t at = 0;
    if (lane == 0) at = atomicAdd(&ctl[LC_LIST], (uint32_t)__popc(b));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (in) list[at + __popc(b & ((1u << lane) - 1u))] = u;
  }
}

// Picks in the greedy's order: gain down, element up (bitonic sort in one block); the first k
// of them as ids and gains.  More than SORT_MAX picks are left to the radix sort.
__global__ void __launch_bounds__(1024) k_level_order(const uint32_t* __restrict__ out_u,
                                                      const uint32_t* __restrict__ out_gain,
                                                      const uint32_t* __restrict__ ctl,
                                                      const int32_t* __restrict__ uid, uint32_t k,
                                                      int64_t* __restrict__ ids, uint32_t* __restrict__ gains) {
  __shared__ unsigned long long key[SORT_MAX];
  const uint32_t n = ctl[LC_PICKS];
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

__global__ void k_level_emit(const uint32_t* __restrict__ u, const uint32_t* __restrict__ flipped_gain, uint32_t n,
                             const int32_t* __restrict__ uid, int64_t* __restrict__ ids,
                             uint32_t* __restrict__ gains) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    ids[i] = uid[u[i]];
    gains[i] = ~flipped_gain[i];
  }
}

// The largest cluster (16 CTAs, else 8) that k_greedy_levels can run on; 0: none.
static int level_cluster() {
  static const int cached = [] {
    const int want[2] = {16, 8};
    for (int c : want) {
      if (c > 8 &&
          cudaFuncSetAttribute(k_greedy_levels, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
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
      if (cudaOccupancyMaxActiveClusters(&clusters, k_greedy_levels, &cfg) == cudaSuccess && clusters > 0) return c;
      cudaGetLastError();
    }
    return 0;
  }();
  return cached;
}

hsaw_status level_greedy(Cover& cv, const uint8_t* cand, int32_t k, int64_t* ids, uint32_t* gains, int32_t* rounds,
                         bool* done, cudaStream_t s) {
  *done = false;
  const int largest = level_cluster();
  if (!largest) return HSAW_OK;
  const uint32_t U = (uint32_t)cv.unique, W = (uint32_t)cv.walks;
  const uint32_t most = std::min(U, W);  // a pick covers a walk of its own
  // one CTA for small streams (its barrier is __syncthreads), else the largest cluster: a solve
  // with 38 K walk elements measured 1.35 ms on 1 CTA, 1.41 on 4 to 16; a pooled one whose
  // greedies see 0.26-8.2 M elements 10.3, 8.6, 8.2 and 8.0 ms on 1, 4, 8 and 16
  const uint32_t csize = (uint64_t)cv.entries <= (1ull << 17) ? 1u : (uint32_t)largest;
  // the list: about what k picks need, or as many as the cluster has threads
  const uint32_t cap = (uint32_t)std::min<uint64_t>(U, std::max<uint64_t>(16ull * (uint64_t)k, 1024ull * csize));
  HSAW_TRY(cv.cnt_work.ensure(U, s));
  HSAW_TRY(cv.g_list.ensure(U, s));
  HSAW_TRY(cv.covered.ensure(W, s));
  HSAW_TRY(cv.partial.ensure(W, s));
  HSAW_TRY(cv.g_rng.ensure(W, s));
  HSAW_TRY(cv.g_cnt.ensure((size_t)4 * most + LEVEL_BINS + LC_WORDS, s));  // picks (and room to sort them), bins, ctl
  uint32_t* out_u = cv.g_cnt.p;
  uint32_t* out_gain = out_u + most;
  uint32_t* hist = out_u + 4 * (size_t)most;
  uint32_t* ctl = hist + LEVEL_BINS;
  HSAW_CK(cudaMemsetAsync(cv.covered.p, 0, (size_t)W * 4, s));
  HSAW_CK(cudaMemsetAsync(cv.partial.p, 0xFF, (size_t)W * 8, s));
  HSAW_CK(cudaMemsetAsync(hist, 0, (LEVEL_BINS + LC_WORDS) * 4, s));
  const bool log = getenv("HSAW_LOG_LAUNCHES") != nullptr;  // measurement aid
  cudaEvent_t ev[2] = {nullptr, nullptr};
  if (log) {
    cudaEventCreate(&ev[0]);
    cudaEventCreate(&ev[1]);
    cudaEventRecord(ev[0], s);
  }
  uint32_t h[LC_WORDS] = {0};
  for (bool first = true;; first = false) {
    if (!first) {  // every level down to the floor is done: the rest of the elements
      HSAW_CK(cudaMemsetAsync(hist, 0, LEVEL_BINS * 4, s));
      HSAW_CK(cudaMemsetAsync(ctl + LC_LIST, 0, 4, s));
    }
    count_launch();
    k_level_hist<<<grid_for(U, 512, 4 * sm_count()), 512, 0, s>>>(first, cv.uid.p, cv.cnt.p, cand, U, cv.cnt_work.p, hist);
    HSAW_CK(cudaGetLastError());
    count_launch();
    k_level_list<<<grid_for(U, 512, 4 * sm_count()), 512, 0, s>>>(hist, cap, cv.cnt_work.p, U, cv.g_list.p, ctl);
    HSAW_CK(cudaGetLastError());
    LevelParams P;
    P.list = cv.g_list.p;
    P.cnt = cv.cnt_work.p;
    P.inv_off = cv.inv_off.p;
    P.inv_walk = cv.inv_walk.p;
    P.walk_eoff = cv.walk_eoff.p;
    P.entry_uidx = cv.entry_uidx.p;
    P.stamp = cv.covered.p;
    P.owner = cv.partial.p;
    P.queue = cv.g_rng.p;
    P.out_u = out_u;
    P.out_gain = out_gain;
    P.ctl = ctl;
    P.k = (uint32_t)k;
    P.round0 = h[LC_ROUNDS];
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
    HSAW_CK(cudaLaunchKernelEx(&cfg, k_greedy_levels, P));
    count_launch();
    k_level_order<<<1, 1024, 0, s>>>(out_u, out_gain, ctl, cv.uid.p, (uint32_t)k, ids, gains);
    HSAW_CK(cudaGetLastError());
    HSAW_CK(cudaMemcpyAsync(h, ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
    HSAW_CK(cudaStreamSynchronize(s));
    if (h[LC_STUCK]) return fail(HSAW_E_DEVICE, "greedy: a level made no progress");
    if (h[LC_PICKS] >= (uint32_t)k || h[LC_GAIN] == 0) {
      if (h[LC_FLOOR] <= 1 || h[LC_PICKS] >= (uint32_t)k) break;
    }
  }
  const uint32_t made = h[LC_PICKS], kept = std::min<uint32_t>(made, (uint32_t)k);
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
    k_level_emit<<<grid_for(kept, 256, 1024), 256, 0, s>>>(alt ? val2 : val, alt ? key2 : key, kept, cv.uid.p, ids, gains);
    HSAW_CK(cudaGetLastError());
  }
  if (log) {
    // a greedy on one cluster with counts in global memory, like k_greedy_cluster (whose record
    // this is), made by levels; spread: picks covered by the whole cluster
    cudaEventRecord(ev[1], s);
    cudaEventSynchronize(ev[1]);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ev[0], ev[1]);
    fprintf(stderr,
            "hsaw: k_greedy_cluster walks=%lld entries=%lld unique=%u cluster=%u gshift=0 k=%d picks=%u spread=%u "
            "levels=%u rounds=%u list=%u made=%u ms=%.3f\n",
            (long long)cv.walks, (long long)cv.entries, U, csize, k, kept, std::min(h[LC_SINGLE], kept), h[LC_LEVELS],
            h[LC_ROUNDS], h[LC_LIST], made, ms);
    cudaEventDestroy(ev[0]);
    cudaEventDestroy(ev[1]);
  }
  *rounds = (int32_t)kept;
  *done = true;
  return HSAW_OK;
}

}  // namespace hsaw
