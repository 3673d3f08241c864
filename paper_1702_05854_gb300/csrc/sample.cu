// HSAW sampling (Sec. 4, Alg. 1-3) on sm_103a.
//
// Attempt a is one live-edge world: node v's live in-edge and source coin come from
// Philox(seed; a, v), so a walk is a trajectory of a functional graph and O(1)-space cycle
// detection (the idea of Sec. 4.2.2) is exact: any revisit proves the cycle.  A persistent warp claims
// chunks of consecutive attempts; lanes that finish take the next attempt of the warp's
// chunk cursor at once (no lane waits for the warp's longest walk).  Hits are recorded
// per chunk as (attempt offset, length); the compaction kernel orders each chunk's hits
// by attempt id and places them by an exclusive scan over chunks, so the stream is
// ordered by attempt id regardless of which warp ran what.  Hit walks are then
// re-derived from their attempt id (the paper's <Seed_h, Len_h> path encoding) straight
// into the flat walk buffers.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "solver.cuh"

namespace hsaw {

enum : uint32_t { ST_OVERFLOW = 1u, ST_STEP_CAP = 2u };

// Control words of a sampler launch, before its chunks' hit counts (cleared together, read back
// in one copy): work counter, status bits, hits, live-edge draws and the hits' nodes (64 bits
// each).
enum SampleCtl { SC_NEXT = 0, SC_STATUS = 1, SC_HITS = 2, SC_STEPS = 4, SC_NODES = 6, SC_WORDS = 8 };

struct SampleParams {
  WalkTables T;
  const uint32_t* __restrict__ s_bits;
  const uint32_t* __restrict__ p32;
  const uint32_t* __restrict__ edge_removed;
  const uint32_t* __restrict__ node_removed;
  uint32_t n;
  uint32_t k0, k1;
  uint64_t a0;           // first attempt of this launch
  uint32_t n_attempts;   // attempts in this launch
  uint32_t chunk_shift;  // chunks of 2^chunk_shift attempts
  uint32_t n_chunks;
  uint32_t cap;          // hit records per chunk
  uint32_t step_cap;
  uint32_t* ctl;         // SampleCtl words
  uint32_t* chunk_hits;  // n_chunks
  uint2* recs;           // n_chunks * cap
  uint4* kept;           // 2 per record, or NULL: the checkpoints of the hit's walk, newest first
  PhiloxKeys keys;       // round keys of (k0, k1)
};

__device__ __forceinline__ bool bit_at(const uint32_t* __restrict__ bits, uint32_t x) {
  return (__ldg(&bits[x >> 5]) >> (x & 31)) & 1u;
}

// A warp draws the starts of its attempts 32 at a time, with every lane, into a buffer in
// shared memory, and its lanes take their next attempt from there: the start draw and the
// node record's latency are paid once per 32 attempts instead of in nearly every iteration
// for the few lanes whose walk just ended.  A start at a node without in-weight that is no
// suspect ends there, without a draw, and never takes a lane (half the nodes of an R-MAT
// graph).  The next chunk is claimed one chunk ahead, so no warp waits for the counter.
// Measured with the 16-byte records: 16 K-node Chung-Lu graph (L2-resident, bound by the ALU
// and issue) 8.48 -> 6.50 ms per 200 K-hit solve; R-MAT 20 with unequal weights 281 -> 239 ms
// per 1 M hits.  One loop that drew starts and live edges in the same Philox block instead
// cost 10-23% more than refilling each lane by itself (fewer lanes active per instruction).
constexpr int SAMPLE_WARPS = 8;
constexpr int START_SLOTS = 64;  // at most 31 left when 32 more are drawn

template <bool HAS_P, bool HAS_REM, Layout L>
__global__ void __launch_bounds__(SAMPLE_WARPS * 32, 6) k_sample(const __grid_constant__ SampleParams P) {
  __shared__ uint4 start_rec[SAMPLE_WARPS][START_SLOTS];  // node record of the start
  __shared__ uint2 start_at[SAMPLE_WARPS][START_SLOTS];   // attempt (within the launch), start node
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  uint32_t cur = 0, cur_end = 0;  // warp's attempt cursor within the launch
  uint32_t ahead = 0;             // lane 0: the next chunk
  if (lane == 0) ahead = atomicAdd(P.ctl + SC_NEXT, 1u);
  uint32_t ready = 0;  // starts in the buffer
  bool more = true;
  bool active = false;
  uint32_t off = 0, v = 0, len = 0;
  uint4 rec = make_uint4(0, 0, 0, 0);  // node record of v: first in-edge, in-degree, equal weight, in-sum
  Ckpt ck;
  ck.reset(0);
  uint32_t my_steps = 0, my_nodes = 0;
  for (;;) {
    const unsigned need = __ballot_sync(FULL, !active);
    if (need) {
      const uint32_t want = __popc(need);
      while (ready < want) {
        if (cur >= cur_end) {
          if (!more) break;
          const uint32_t c = __shfl_sync(FULL, ahead, 0);
          more = c < P.n_chunks;
          if (!more) break;
          cur = c << P.chunk_shift;
          cur_end = min(cur + (1u << P.chunk_shift), P.n_attempts);
          if (lane == 0) ahead = atomicAdd(P.ctl + SC_NEXT, 1u);
        }
        const uint32_t i = cur + lane;
        bool walk = false;
        uint32_t sv = 0;
        uint4 srec = make_uint4(0, 0, 0, 0);
        if (i < cur_end) {
          const uint64_t a = P.a0 + i;
          sv = __umulhi(philox4x32_10_rk(make_uint4((uint32_t)a, (uint32_t)(a >> 32), 0u, 1u), P.keys).x, P.n);
          srec = __ldg(&P.T.node[sv]);
          walk = bit_at(P.s_bits, sv) || srec.w != 0;
          if (HAS_REM && P.node_removed && bit_at(P.node_removed, sv)) walk = false;
        }
        const unsigned got = __ballot_sync(FULL, walk);
        if (walk) {
          const uint32_t slot = ready + __popc(got & lt);
          start_at[w][slot] = make_uint2(i, sv);
          start_rec[w][slot] = srec;
        }
        ready += __popc(got);
        cur = min(cur + 32u, cur_end);
      }
      __syncwarp();
      const uint32_t take = min(want, ready);
      if (take == 0 && need == FULL) break;
      const uint32_t rank = __popc(need & lt);
      if (!active && rank < take) {
        const uint32_t slot = ready - 1 - rank;
        const uint2 at = start_at[w][slot];
        rec = start_rec[w][slot];
        off = at.x;
        v = at.y;
        ck.reset(v);
        len = 1;
        active = true;
      }
      ready -= take;
      __syncwarp();  // slots are read before they are filled again
    }
    if (active) {
      // one live-edge draw at node v (Alg. 1 lines 5-13); the tail's record comes with it
      const uint64_t a = P.a0 + off;
      const uint32_t sw = __ldg(&P.s_bits[v >> 5]);
      const uint4 x = philox4x32_10_rk(make_uint4((uint32_t)a, (uint32_t)(a >> 32), v, 0u), P.keys);
      const bool live = x.x < rec.w;
      uint4 next = make_uint4(0, 0, 0, 0);
      uint32_t e = 0, u = 0;
      if (live) e = record_step<L>(P.T, v, rec, x.x, u, next);
      bool gone = false;  // the removal bit is read beside the walk record
      if (HAS_REM && live && P.edge_removed) gone = bit_at(P.edge_removed, e);
      const bool suspect = (sw >> (v & 31)) & 1u;
      int outcome = -1;  // -1 continue, 0 miss, 1 hit
      if (suspect && (!HAS_P || source_coin(x.y, __ldg(&P.p32[v])))) {
        outcome = 1;
      } else {
        ++my_steps;
        if (!live) {
          outcome = 0;  // no live in-edge
        } else if (HAS_REM && (gone || (P.node_removed && bit_at(P.node_removed, u)))) {
          outcome = 0;
        } else if (ck.seen(u)) {
          outcome = 0;  // the walk closed a cycle
        } else {
          ck.keep(u, len);
          v = u;
          rec = next;
          if (++len > P.step_cap) {
            atomicOr(P.ctl + SC_STATUS, ST_STEP_CAP);
            outcome = 0;
          }
        }
      }
      if (outcome >= 0) {
        active = false;
        if (outcome == 1) {
          my_nodes += len;
          const uint32_t ck_i = off >> P.chunk_shift;
          const uint32_t slot = atomicAdd(&P.chunk_hits[ck_i], 1u);
          if (slot < P.cap) {
            const size_t at = (size_t)ck_i * P.cap + slot;
            P.recs[at] = make_uint2(off, len);
            if (P.kept) {
              P.kept[2 * at] = make_uint4(ck.c0, ck.c1, ck.c2, ck.c3);
              P.kept[2 * at + 1] = make_uint4(ck.c4, ck.c5, ck.c6, ck.c7);
            }
          } else atomicOr(P.ctl + SC_STATUS, ST_OVERFLOW);
        }
      }
    }
  }
  // draws and hit nodes of this warp
  unsigned long long warp_steps = my_steps, warp_nodes = my_nodes;
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    warp_steps += __shfl_down_sync(FULL, warp_steps, o);
    warp_nodes += __shfl_down_sync(FULL, warp_nodes, o);
  }
  if (lane == 0 && warp_steps) atomicAdd(reinterpret_cast<unsigned long long*>(P.ctl + SC_STEPS), warp_steps);
  if (lane == 0 && warp_nodes) atomicAdd(reinterpret_cast<unsigned long long*>(P.ctl + SC_NODES), warp_nodes);
}

// Order each chunk's hits by attempt id and write them at the chunk's scanned offset (*total:
// the hits of all chunks).  One warp per chunk; rank = number of the chunk's records with a
// smaller offset.
__global__ void k_compact(const uint32_t* __restrict__ chunk_off, const uint32_t* __restrict__ total,
                          const uint2* __restrict__ recs, uint32_t cap, uint32_t n_chunks, uint64_t a0,
                          const uint4* __restrict__ kept, uint64_t* __restrict__ out_aid,
                          uint32_t* __restrict__ out_len, uint4* __restrict__ out_kept) {
  const int lane = threadIdx.x & 31;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t ck = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; ck < n_chunks; ck += warps) {
    const uint32_t base = chunk_off[ck];
    const uint32_t c = (ck + 1 < n_chunks ? chunk_off[ck + 1] : *total) - base;
    if (c == 0) continue;
    const uint2* r = recs + (size_t)ck * cap;
    for (uint32_t i = lane; i < c; i += 32) {
      const uint2 me = r[i];
      uint32_t rank = 0;
      for (uint32_t j = 0; j < c; ++j) rank += (r[j].x < me.x) ? 1u : 0u;
      out_aid[base + rank] = a0 + me.x;
      out_len[base + rank] = me.y;
      if (kept) {
        out_kept[2 * (size_t)(base + rank)] = kept[2 * ((size_t)ck * cap + i)];
        out_kept[2 * (size_t)(base + rank) + 1] = kept[2 * ((size_t)ck * cap + i) + 1];
      }
    }
  }
}

// node_off[i] = base + len[0] + ... + len[i - 1], i <= n: sums of 4,096-walk tiles, their scan,
// then the tiles' own scans.
constexpr int OFF_THREADS = 512, OFF_TILE = 4096;
__device__ __forceinline__ uint64_t block_scan_u64(uint64_t v, uint64_t* sums, uint64_t* total) {  // exclusive
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint64_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) sums[w] = inc;
  __syncthreads();
  uint64_t before = 0, all = 0;
  for (int i = 0; i < OFF_THREADS / 32; ++i) {
    const uint64_t x = sums[i];
    if (i < w) before += x;
    all += x;
  }
  *total = all;
  return before + inc - v;
}

__global__ void __launch_bounds__(OFF_THREADS) k_len_tiles(const uint32_t* __restrict__ len, int64_t n,
                                                           uint64_t* __restrict__ tile_sum) {
  __shared__ uint64_t sums[OFF_THREADS / 32];
  uint64_t v = 0, total;
  const int64_t base = (int64_t)blockIdx.x * OFF_TILE;
  for (int i = threadIdx.x; i < OFF_TILE; i += OFF_THREADS)
    if (base + i < n) v += len[base + i];
  block_scan_u64(v, sums, &total);
  if (threadIdx.x == 0) tile_sum[blockIdx.x] = total;
}

__global__ void __launch_bounds__(OFF_THREADS) k_len_offsets(const uint32_t* __restrict__ len, int64_t n,
                                                             const uint64_t* __restrict__ tile_off, int64_t base,
                                                             int64_t* __restrict__ node_off) {
  constexpr int PER = OFF_TILE / OFF_THREADS;
  __shared__ uint64_t sums[OFF_THREADS / 32];
  const int64_t i0 = (int64_t)blockIdx.x * OFF_TILE + threadIdx.x * PER;
  uint32_t l[PER];
  uint64_t v = 0, total;
#pragma unroll
  for (int i = 0; i < PER; ++i) v += l[i] = i0 + i < n ? len[i0 + i] : 0u;
  uint64_t run = block_scan_u64(v, sums, &total) + base + (tile_off ? tile_off[blockIdx.x] : 0ull);
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    if (i0 + i <= n) node_off[i0 + i] = (int64_t)run;
    run += l[i];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == OFF_THREADS - 1 && i0 + PER == n) node_off[n] = (int64_t)run;
}

static hsaw_status len_offsets(const uint32_t* len, int64_t n, int64_t base, int64_t* node_off, DBuf<uint64_t>& tmp,
                               cudaStream_t s) {
  const int64_t tiles = (n + OFF_TILE - 1) / OFF_TILE;
  if (tiles > 1) {
    HSAW_TRY(tmp.ensure((size_t)tiles, s));
    count_launch();
    k_len_tiles<<<(unsigned)tiles, OFF_THREADS, 0, s>>>(len, n, tmp.p);
    HSAW_CK(cudaGetLastError());
    HSAW_TRY(exclusive_scan_u64(tmp.p, (size_t)tiles, nullptr, s));
  }
  count_launch();
  k_len_offsets<<<(unsigned)tiles, OFF_THREADS, 0, s>>>(len, n, tiles > 1 ? tmp.p : nullptr, base, node_off);
  HSAW_CK(cudaGetLastError());
  return HSAW_OK;
}

// Re-derive hit walks from their attempt ids (path encoding) into the flat buffers.
template <Layout L>
__global__ void k_rewalk(const WalkTables T, uint32_t n, uint32_t k0, uint32_t k1, const uint64_t* __restrict__ aid,
                         const uint32_t* __restrict__ len, const int64_t* __restrict__ node_off, int64_t h0, int64_t h1,
                         int32_t* __restrict__ nodes, int32_t* __restrict__ edges) {
  for (int64_t h = h0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; h < h1; h += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t a = aid[h];
    const uint32_t l = len[h];
    const int64_t nb = node_off[h], eb = nb - h;
    uint32_t v = start_node(a, n, k0, k1);
    nodes[nb] = (int32_t)v;
    uint4 rec = l > 1 ? __ldg(&T.node[v]) : make_uint4(0, 0, 0, 0);
    for (uint32_t i = 1; i < l; ++i) {
      const uint4 x = node_draw(a, v, k0, k1);
      if (x.x >= rec.w) break;  // a hit's walk has a live in-edge at each of its first l - 1 nodes
      edges[eb + i - 1] = (int32_t)record_step<L>(T, v, rec, x.x, v, rec);
      nodes[nb + i] = (int32_t)v;
    }
  }
}

// The same by segments: the walk's last eight checkpoints (kept, newest first) are known, so its
// parts between them are walked side by side, each a fifth of the walk at most.  A launch takes
// as long as its longest chain of dependent reads: the longest hit of a window is 5-10 times
// the mean.
constexpr int SEGMENTS = 9;
template <Layout L>
__global__ void k_rewalk_segments(const WalkTables T, uint32_t n, uint32_t k0, uint32_t k1,
                                  const uint64_t* __restrict__ aid, const uint32_t* __restrict__ len,
                                  const int64_t* __restrict__ node_off, const uint32_t* __restrict__ kept, int64_t h0,
                                  int64_t h1, int32_t* __restrict__ nodes, int32_t* __restrict__ edges) {
  const int64_t total = (h1 - h0) * SEGMENTS;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t h = h0 + i / SEGMENTS;
    const uint32_t seg = (uint32_t)(i % SEGMENTS);  // from the checkpoint that is seg-th from the end; 8: from the start
    const uint32_t l = len[h];
    // the positions kept before l, newest first: how many, and those this segment lies between
    uint32_t count = 0;
    for (uint32_t p = 1; p < l; p = Ckpt::after(p)) ++count;
    const uint32_t have = min(count, 8u);
    if (seg < 8 && seg >= have) continue;
    const uint32_t from_rank = seg < 8 ? count - seg : 0u;              // rank 0: the start, at position 0
    const uint32_t to_rank = seg < 8 ? from_rank + 1 : count - have + 1;  // rank count + 1: the end
    uint32_t from = 0, to = l - 1, p = 1;
    for (uint32_t rank = 1; rank <= count; ++rank, p = Ckpt::after(p)) {
      if (rank == from_rank) from = p;
      if (rank == to_rank) to = p;
    }
    const uint64_t a = aid[h];
    const int64_t nb = node_off[h], eb = nb - h;
    uint32_t v;
    if (seg < 8) {
      v = kept[8 * (h - h0) + seg];
    } else {
      v = start_node(a, n, k0, k1);
      nodes[nb] = (int32_t)v;
    }
    uint4 rec = to > from ? __ldg(&T.node[v]) : make_uint4(0, 0, 0, 0);
    for (uint32_t q = from; q < to; ++q) {
      const uint4 x = node_draw(a, v, k0, k1);
      if (x.x >= rec.w) break;  // a hit's walk has a live in-edge at each of its first l - 1 nodes
      edges[eb + q] = (int32_t)record_step<L>(T, v, rec, x.x, v, rec);
      nodes[nb + q + 1] = (int32_t)v;
    }
  }
}

// Per-attempt outcome (0 no edge, 1 hit, 2 cycle, 3 removed) and nodes walked.
template <bool HAS_P, bool HAS_REM>
__global__ void k_classify(SampleParams P, uint64_t first, int64_t count, int8_t* __restrict__ outcome,
                           int32_t* __restrict__ length) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t a = first + (uint64_t)i;
    uint32_t v = start_node(a, P.n, P.k0, P.k1), len = 1;
    Ckpt ck;
    ck.reset(v);
    int out = -1;
    if (HAS_REM && P.node_removed && bit_at(P.node_removed, v)) out = 3;
    while (out < 0) {
      const bool suspect = (__ldg(&P.s_bits[v >> 5]) >> (v & 31)) & 1u;
      const uint4 x = node_draw(a, v, P.k0, P.k1);
      if (suspect && (!HAS_P || source_coin(x.y, __ldg(&P.p32[v])))) { out = 1; break; }
      const uint4 nd = __ldg(&P.T.node[v]);
      if (x.x >= nd.w) { out = 0; break; }
      const uint32_t e = nd.x + pick_in_edge(P.T.edge, nd, x.x);
      const uint32_t u = __ldg(&P.T.edge[e].x);
      if (HAS_REM && ((P.edge_removed && bit_at(P.edge_removed, e)) || (P.node_removed && bit_at(P.node_removed, u)))) {
        out = 3;
        break;
      }
      if (ck.seen(u)) { out = 2; break; }
      ck.keep(u, len);
      v = u;
      if (++len > P.step_cap) { atomicOr(P.ctl + SC_STATUS, ST_STEP_CAP); out = 0; break; }
    }
    outcome[i] = (int8_t)out;
    length[i] = (int32_t)len;
  }
}

// ------------------------------------------------------------------ host
__global__ void k_set_bits(const int32_t* __restrict__ src, const uint32_t* __restrict__ p, int32_t cnt,
                           uint32_t* __restrict__ bits, uint32_t* __restrict__ p32) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += gridDim.x * blockDim.x) {
    const uint32_t v = (uint32_t)src[i];
    atomicOr(&bits[v >> 5], 1u << (v & 31));
    if (p32) p32[v] = p[i];
  }
}

hsaw_status query_upload(const Graph& g, const hsaw_query* q, QueryDev& qd, cudaStream_t s) {
  if (!q) return fail(HSAW_E_INVALID, "query: NULL");
  if (q->n_sources < 1 || !q->sources) return fail(HSAW_E_INVALID, "query: need at least one source");
  std::vector<uint8_t> seen((size_t)g.n, 0);
  for (int32_t i = 0; i < q->n_sources; ++i) {
    int32_t v = q->sources[i];
    if (v < 0 || v >= g.n) return fail(HSAW_E_RANGE, "query: source outside [0, n)");
    if (seen[v]) return fail(HSAW_E_INVALID, "query: duplicate source");
    seen[v] = 1;
  }
  const size_t words = (size_t)(g.n + 31) / 32;
  HSAW_TRY(dmalloc((void**)&qd.s_bits, words * 4, s));
  HSAW_CK(cudaMemsetAsync(qd.s_bits, 0, words * 4, s));
  if (q->p_fixed) {
    HSAW_TRY(dmalloc((void**)&qd.p32, (size_t)g.n * 4, s));
    HSAW_CK(cudaMemsetAsync(qd.p32, 0, (size_t)g.n * 4, s));
  }
  // the source list stays with the query (walk-pool queries read their sources' lists);
  // on failure the caller's query_release frees what was allocated
  HSAW_TRY(dmalloc((void**)&qd.s_list, (size_t)q->n_sources * 4, s));
  qd.n_src = q->n_sources;
  HSAW_CK(cudaMemcpyAsync(qd.s_list, q->sources, (size_t)q->n_sources * 4, cudaMemcpyHostToDevice, s));
  uint32_t* d_p = nullptr;
  if (q->p_fixed) {
    HSAW_TRY(dmalloc((void**)&d_p, (size_t)q->n_sources * 4, s));
    if (cudaMemcpyAsync(d_p, q->p_fixed, (size_t)q->n_sources * 4, cudaMemcpyHostToDevice, s) != cudaSuccess) {
      dfree(d_p, s);
      return fail(HSAW_E_DEVICE, "query: probability upload failed");
    }
  }
  count_launch();
  k_set_bits<<<grid_for(q->n_sources, 256, 1024), 256, 0, s>>>(qd.s_list, d_p, q->n_sources, qd.s_bits, qd.p32);
  const cudaError_t le = cudaGetLastError();
  dfree(d_p, s);
  if (le != cudaSuccess) return fail(HSAW_E_DEVICE, "query: suspect bits launch failed");
  qd.seed = q->seed;
  double real = 0.0;  // expected number of real sources
  for (int32_t i = 0; i < q->n_sources; ++i) real += q->p_fixed ? (double)q->p_fixed[i] / 4294967296.0 : 1.0;
  qd.start_rate = real / (double)g.n;
  return HSAW_OK;
}

// Removal masks are kept as bits: the walk reads one per draw at random, and m bytes would
// push walk records out of L2 (R-MAT 22 eSI residual estimate of 100 K hits, 1,000 edges
// removed: 67 MB of bytes against 8.4 MB of bits).
__global__ void k_pack_mask(const uint8_t* __restrict__ bytes, size_t len, uint32_t* __restrict__ bits) {
  const size_t words = (len + 31) / 32;
  for (size_t w = blockIdx.x * (size_t)blockDim.x + threadIdx.x; w < words; w += (size_t)gridDim.x * blockDim.x) {
    uint32_t b = 0;
    if (w * 32 + 32 <= len) {  // bytes starts on a 16-byte boundary (an allocation of its own)
      const uint4* p = reinterpret_cast<const uint4*>(bytes + w * 32);
      const uint4 q[2] = {p[0], p[1]};
      const uint32_t* x = reinterpret_cast<const uint32_t*>(q);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) b |= ((x[i] >> (8 * j)) & 0xFFu) ? 1u << (4 * i + j) : 0u;
    } else {
      for (size_t i = w * 32; i < len; ++i) b |= bytes[i] ? 1u << (i & 31) : 0u;
    }
    bits[w] = b;
  }
}

hsaw_status pack_mask(const uint8_t* bytes, size_t len, uint32_t** bits, cudaStream_t s) {
  HSAW_TRY(dmalloc((void**)bits, (len + 31) / 32 * 4, s));
  count_launch();
  k_pack_mask<<<grid_for((len + 31) / 32, 256, 8192), 256, 0, s>>>(bytes, len, *bits);
  HSAW_CK(cudaGetLastError());
  return HSAW_OK;
}

void query_release(QueryDev& qd, cudaStream_t s) {
  dfree(qd.s_bits, s);
  dfree(qd.s_list, s);
  dfree(qd.p32, s);
  if (qd.owns_removed) {
    dfree(qd.edge_removed, s);
    dfree(qd.node_removed, s);
  }
  qd = QueryDev();
}

void Stream::release(cudaStream_t s) {
  aid.release(s); len.release(s); node_off.release(s); nodes.release(s); edges.release(s);
  chunk_hits.release(s); chunk_off.release(s); chunk_kept.release(s); kept.release(s); ctrs.release(s); recs.release(s); tmp64.release(s);
  pbits.release(s); pcnt.release(s);
}

hsaw_status stream_init(Stream& st, uint64_t first_attempt, uint64_t max_attempts, cudaStream_t s) {
  st.count = 0;
  st.total_nodes = 0;
  st.first_attempt = first_attempt;
  st.next_attempt = first_attempt;
  st.steps = 0;
  st.max_attempts = max_attempts ? max_attempts : (1ull << 62);
  HSAW_TRY(st.node_off.ensure(1024, s));
  HSAW_CK(cudaMemsetAsync(st.node_off.p, 0, sizeof(int64_t), s));
  HSAW_TRY(st.ctrs.ensure(8, s));
  return HSAW_OK;
}

static SampleParams make_params(const Graph& g, const QueryDev& qd) {
  SampleParams P{};
  P.T = g.tables();
  P.s_bits = qd.s_bits;
  P.p32 = qd.p32;
  P.edge_removed = qd.edge_removed;
  P.node_removed = qd.node_removed;
  P.n = (uint32_t)g.n;
  P.k0 = (uint32_t)qd.seed;
  P.k1 = (uint32_t)(qd.seed >> 32);
  P.keys = philox_round_keys(P.k0, P.k1);
  P.step_cap = (uint32_t)std::min<uint64_t>(4ull * (uint64_t)g.n + 64ull, 0xFFFFFFF0ull);
  return P;
}

static int sample_blocks_per_sm() {
  static const int cached = [] {
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_sample<false, false, REC16>, 256, 0);
    return b > 0 ? b : 1;
  }();
  return cached;
}

// Blocks per SM: all that fit, 6.  G draws/s with 4 and 6 blocks, R-MAT: equal weights at scale
// 17 to 23: 173/185, 153/173, 111/112, 101/100, 67/65, 49/48, 39/40; random weights at 16 to 22:
// 71/84, 71/83, 47/59, 37/40, 34/37.  (With two loads a record, 3 blocks were the faster on
// graphs far beyond L2; one load does not need that.)  HSAW_SAMPLE_BLOCKS=b in the environment
// asks for b (measurement).
static int sample_blocks() {
  const int full = sample_blocks_per_sm();
  const char* f = getenv("HSAW_SAMPLE_BLOCKS");
  const int b = f ? atoi(f) : 0;
  return b > 0 ? std::min(full, b) : full;
}

template <Layout L>
static void launch_sample_as(const SampleParams& P, unsigned grid, cudaStream_t s) {
  const bool hp = P.p32 != nullptr, hr = (P.edge_removed || P.node_removed);
  count_launch();
  if (hp && hr) k_sample<true, true, L><<<grid, 256, 0, s>>>(P);
  else if (hp) k_sample<true, false, L><<<grid, 256, 0, s>>>(P);
  else if (hr) k_sample<false, true, L><<<grid, 256, 0, s>>>(P);
  else k_sample<false, false, L><<<grid, 256, 0, s>>>(P);
}

static void launch_sample(const Graph& g, const SampleParams& P, unsigned grid, cudaStream_t s) {
  switch (g.layout) {
    case REC16: launch_sample_as<REC16>(P, grid, s); break;
    case REC32: launch_sample_as<REC32>(P, grid, s); break;
    case TAIL4: launch_sample_as<TAIL4>(P, grid, s); break;
    case EDGE8: launch_sample_as<EDGE8>(P, grid, s); break;
  }
}

// Attempts per chunk: 256, or fewer (32 at least) where that leaves resident warps without one.
// A lane then walks one attempt or few, so a short launch ends with its longest walk instead of
// the longest sum of eight: 4,096 attempts on a 16 K-node graph, 105 -> 60 us.
static uint32_t chunk_shift_for(uint64_t attempts) {
  const uint64_t warps = (uint64_t)sm_count() * sample_blocks_per_sm() * SAMPLE_WARPS;
  uint32_t shift = 8;
  while (shift > 5 && (attempts >> shift) < warps) --shift;
  return shift;
}

// One sampler launch over attempts [st.next_attempt, + batch): hits are recorded per chunk
// and compacted in attempt order into aid/len at st.count; *new_hits receives their number,
// *new_nodes their nodes.
static hsaw_status sample_window(const Graph& g, const QueryDev& qd, Stream& st, uint64_t batch, uint32_t* new_hits,
                                 int64_t* new_nodes, cudaStream_t s) {
  SampleParams P = make_params(g, qd);
  const uint32_t shift = chunk_shift_for(batch), chunk = 1u << shift;
  const uint32_t n_chunks = (uint32_t)((batch + chunk - 1) >> shift);
  // with no hit yet, the rate is below a few in the attempts so far
  const uint64_t used = st.next_attempt - st.first_attempt;
  uint32_t cap = hit_records(st.hit_rate > 0.0 ? st.hit_rate : used ? 1.0 / (double)used : 1.0, chunk);
  for (;;) {
    HSAW_TRY(st.chunk_hits.ensure((size_t)SC_WORDS + n_chunks, s));
    HSAW_TRY(st.recs.ensure((size_t)n_chunks * cap, s));
    const double elements = st.count ? st.hit_rate * (double)batch * (double)st.total_nodes / (double)st.count : 0.0;
    const bool keep = !st.ids_only && !lean() && (st.count || !used) && (uint64_t)n_chunks * cap <= kept_records(elements);
    HSAW_TRY(st.chunk_kept.ensure(keep ? 2 * (size_t)n_chunks * cap : 0, s));
    uint32_t* const ctl = st.chunk_hits.p;
    HSAW_CK(cudaMemsetAsync(ctl, 0, ((size_t)SC_WORDS + n_chunks) * 4, s));
    P.a0 = st.next_attempt;
    P.n_attempts = (uint32_t)batch;
    P.chunk_shift = shift;
    P.n_chunks = n_chunks;
    P.cap = cap;
    P.ctl = ctl;
    P.chunk_hits = ctl + SC_WORDS;
    P.recs = st.recs.p;
    P.kept = keep ? st.chunk_kept.p : nullptr;
    const int bps = sample_blocks();
    const unsigned grid = (unsigned)std::max(1, std::min<int>(sm_count() * bps, (int)((n_chunks + 7) / 8)));
    void* prof = profile_begin(s);
    launch_sample(g, P, grid, s);
    profile_end(prof, s, batch);
    HSAW_CK(cudaGetLastError());
    // the counts' offsets in place (a chunk with more hits than records makes the launch run
    // again, whatever they say)
    HSAW_TRY(exclusive_scan_u32(P.chunk_hits, n_chunks, ctl + SC_HITS, s));
    uint32_t h[SC_WORDS];
    HSAW_CK(cudaMemcpyAsync(h, ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
    HSAW_CK(cudaStreamSynchronize(s));
    unsigned long long hs = 0, hn = 0;
    std::memcpy(&hs, h + SC_STEPS, 8);
    std::memcpy(&hn, h + SC_NODES, 8);
    if (h[SC_STATUS] & ST_STEP_CAP) return fail(HSAW_E_STEP_CAP, "sampling: a walk exceeded its step guard");
    if ((h[SC_STATUS] & ST_OVERFLOW) && cap < chunk) {
      cap = chunk;  // rare: rerun this launch with room for every attempt to hit
      continue;
    }
    st.steps += hs;
    profile_add_steps(hs);
    if (getenv("HSAW_LOG_LAUNCHES"))  // measurement aid: attempts and live-edge draws of each sampler launch
      fprintf(stderr, "hsaw: k_sample launch attempts=%llu draws=%llu blocks_per_sm=%d\n", (unsigned long long)batch,
              hs, bps);
    *new_hits = h[SC_HITS];
    *new_nodes = (int64_t)hn;
    if (*new_hits) {
      HSAW_TRY(st.aid.ensure((size_t)st.count + *new_hits, s, true));
      HSAW_TRY(st.len.ensure((size_t)st.count + *new_hits, s, true));
      HSAW_TRY(st.kept.ensure(keep ? 2 * (size_t)*new_hits : 0, s));
      st.kept_hits = keep ? *new_hits : 0;
      count_launch();
      k_compact<<<grid_for((size_t)n_chunks * 32, 256, 8192), 256, 0, s>>>(
          P.chunk_hits, ctl + SC_HITS, st.recs.p, cap, n_chunks, st.next_attempt, P.kept, st.aid.p + st.count,
          st.len.p + st.count, st.kept.p);
      HSAW_CK(cudaGetLastError());
    }
    return HSAW_OK;
  }
}

hsaw_status stream_extend(const Graph& g, const QueryDev& qd, Stream& st, int64_t want, cudaStream_t s) {
  st.elem_range[0] = g.n;
  st.elem_range[1] = g.m;
  const uint32_t CHUNK = 256;
  // the walk pool serves this query's attempts below pool.attempts when the walk seed
  // matches and the graph is not a residual one
  const bool pool_ok = g.pool.ent && g.pool.seed == qd.seed && qd.s_list && !qd.edge_removed && !qd.node_removed;
  while (st.count < want) {
    if (cancel_requested()) return fail(HSAW_E_CANCELLED, "sampling: query cancelled");
    const uint64_t used = st.next_attempt - st.first_attempt;
    if (used >= st.max_attempts) return fail(HSAW_E_TIMEOUT, "sampling: attempt budget exhausted before enough hits");
    // window size from the hit rate so far (2^20 .. 2^28 attempts; doubling while no hit; down
    // to 2^16 where the walks of a window past the last hit asked for are of no use to the
    // caller, the first then by 16 times the rate that start nodes alone give: most walks see
    // more nodes than that, and one that falls short costs a launch),
    // with a margin of 4 standard deviations of the rate estimate (st.count hits seen) and
    // of the window's own hit count (need): attempts past the last hit a solve uses are
    // wasted, and a window that falls short only costs one more launch
    const double need = (double)(want - st.count);
    st.hit_rate = used ? (double)st.count / (double)used : 0.0;
    const double margin = std::min(1.25, 1.0 + 4.0 / std::sqrt(std::max(1.0, (double)st.count)) + 4.0 / std::sqrt(need));
    const double least = st.least_window;
    double target = st.hit_rate > 0 ? need / st.hit_rate * margin + 4096.0
                    : used          ? std::max(1048576.0, 2.0 * (double)used)
                                    : std::min(1048576.0, need / 16.0 / std::max(qd.start_rate, 1e-12));
    target = std::max(target, least);
    target = std::min(target, (double)MOST_ATTEMPTS);
    uint64_t batch = (uint64_t)target;
    batch = std::min<uint64_t>(batch, st.max_attempts - used);
    uint32_t new_hits = 0;
    int64_t new_nodes = 0;
    if (pool_ok && st.next_attempt < g.pool.attempts) {
      // whole blocks of the index where the pool and the budget allow
      const uint64_t B = 1ull << g.pool.shift;
      uint64_t a1 = std::min<uint64_t>(g.pool.attempts, (st.next_attempt + batch + B - 1) / B * B);
      a1 = std::min<uint64_t>(a1, st.next_attempt + (st.max_attempts - used));
      batch = a1 - st.next_attempt;
      HSAW_TRY(pool_hits(g, qd, st, st.next_attempt, a1, &new_hits, &new_nodes, s));
    } else {
      batch = (batch + CHUNK - 1) / CHUNK * CHUNK;
      HSAW_TRY(sample_window(g, qd, st, batch, &new_hits, &new_nodes, s));
    }
    HSAW_TRY(stream_take_hits(g, qd, st, new_hits, new_nodes, s));
    st.next_attempt += batch;
  }
  return HSAW_OK;
}

hsaw_status stream_take_hits(const Graph& g, const QueryDev& qd, Stream& st, uint32_t new_hits, int64_t new_nodes,
                             cudaStream_t s) {
  if (!new_hits) return HSAW_OK;
  if (st.ids_only) {
    st.count += new_hits;
    return HSAW_OK;
  }
  const uint32_t k0 = (uint32_t)qd.seed, k1 = (uint32_t)(qd.seed >> 32);
  // walk offsets, then the hits' nodes and edges re-drawn from their attempt ids
  HSAW_TRY(st.node_off.ensure((size_t)st.count + new_hits + 1, s, true));
  HSAW_TRY(len_offsets(st.len.p + st.count, new_hits, st.total_nodes, st.node_off.p + st.count, st.tmp64, s));
  if (new_nodes < 0) {
    int64_t end = 0;
    HSAW_CK(cudaMemcpyAsync(&end, st.node_off.p + st.count + new_hits, 8, cudaMemcpyDeviceToHost, s));
    HSAW_CK(cudaStreamSynchronize(s));
    new_nodes = end - st.total_nodes;
  }
  const int64_t tot = st.total_nodes + new_nodes;
  HSAW_TRY(st.nodes.ensure((size_t)tot, s, true));
  HSAW_TRY(st.edges.ensure((size_t)tot, s, true));
  // by segments where walks are long enough for their start-up (a node record each) to pay
  const bool segments = st.kept_hits == new_hits && new_nodes >= 16 * (int64_t)new_hits;
  st.kept_hits = 0;
  count_launch();
  if (segments) {
    const decltype(&k_rewalk_segments<REC16>) by_layout[] = {k_rewalk_segments<REC16>, k_rewalk_segments<REC32>,
                                                             k_rewalk_segments<TAIL4>, k_rewalk_segments<EDGE8>};
    by_layout[g.layout]<<<grid_for((size_t)new_hits * SEGMENTS, 128, 1u << 16), 128, 0, s>>>(
        g.tables(), (uint32_t)g.n, k0, k1, st.aid.p, st.len.p, st.node_off.p, reinterpret_cast<uint32_t*>(st.kept.p),
        st.count, st.count + new_hits, st.nodes.p, st.edges.p);
  } else {
    const decltype(&k_rewalk<REC16>) by_layout[] = {k_rewalk<REC16>, k_rewalk<REC32>, k_rewalk<TAIL4>, k_rewalk<EDGE8>};
    by_layout[g.layout]<<<grid_for(new_hits, 128, 1u << 16), 128, 0, s>>>(
        g.tables(), (uint32_t)g.n, k0, k1, st.aid.p, st.len.p, st.node_off.p, st.count, st.count + new_hits, st.nodes.p,
        st.edges.p);
  }
  HSAW_CK(cudaGetLastError());
  st.total_nodes = tot;
  st.count += new_hits;
  return HSAW_OK;
}

hsaw_status classify_attempts(const Graph& g, const QueryDev& qd, uint64_t first, int64_t count, int8_t* outcome,
                              int32_t* length, cudaStream_t s) {
  SampleParams P = make_params(g, qd);
  uint32_t* d_ctr = nullptr;
  HSAW_TRY(dmalloc((void**)&d_ctr, 16, s));
  HSAW_CK(cudaMemsetAsync(d_ctr, 0, 16, s));
  P.ctl = d_ctr;
  const unsigned grid = grid_for(count, 128, 1u << 16);
  const bool hp = P.p32 != nullptr, hr = (P.edge_removed || P.node_removed);
  if (hp && hr) { count_launch(); k_classify<true, true><<<grid, 128, 0, s>>>(P, first, count, outcome, length); }
  else if (hp) { count_launch(); k_classify<true, false><<<grid, 128, 0, s>>>(P, first, count, outcome, length); }
  else if (hr) { count_launch(); k_classify<false, true><<<grid, 128, 0, s>>>(P, first, count, outcome, length); }
  else { count_launch(); k_classify<false, false><<<grid, 128, 0, s>>>(P, first, count, outcome, length); }
  HSAW_CK(cudaGetLastError());
  uint32_t h[2] = {0, 0};
  HSAW_CK(cudaMemcpyAsync(h, d_ctr, 8, cudaMemcpyDeviceToHost, s));
  HSAW_CK(cudaStreamSynchronize(s));
  dfree(d_ctr, s);
  if (h[1] & ST_STEP_CAP) return fail(HSAW_E_STEP_CAP, "classify: a walk exceeded its step guard");
  return HSAW_OK;
}

}  // namespace hsaw

// ------------------------------------------------------------------ allocation-free variant
// Scratch of hsaw_sample_hits_static: file-scope device arrays sized for at most
// HSAW_STATIC_MAX_ATTEMPTS attempts per call (about 2 MiB in total).  Every GPU that loads
// this library holds them until the process exits.  Host code cannot pass these names to
// a kernel (in host code they are stand-ins, not device addresses); their device
// addresses are looked up once per device with cudaGetSymbolAddress.
namespace hsaw {

constexpr uint32_t STATIC_CHUNKS = HSAW_STATIC_MAX_ATTEMPTS / 32;  // chunks of at least 32 attempts

static __device__ __align__(256) uint32_t g_static_ctl[SC_WORDS + STATIC_CHUNKS];  // control words, chunk hits
static __device__ __align__(256) uint2 g_static_recs[HSAW_STATIC_MAX_ATTEMPTS];

struct StaticScratch {
  uint32_t* ctl = nullptr;
  uint2* recs = nullptr;
  bool ready = false;
};
static StaticScratch g_static_dev[64];
static std::mutex g_static_mu;

// Device addresses of the static scratch on the current device (set-up on first use).
static hsaw_status static_scratch(StaticScratch** out) {
  int dev = 0;
  HSAW_CK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(HSAW_E_DEVICE, "static sampler: device index out of range");
  std::lock_guard<std::mutex> lk(g_static_mu);
  StaticScratch& s = g_static_dev[dev];
  if (!s.ready) {
    HSAW_CK(cudaGetSymbolAddress((void**)&s.ctl, g_static_ctl));
    HSAW_CK(cudaGetSymbolAddress((void**)&s.recs, g_static_recs));
    s.ready = true;
  }
  *out = &s;
  return HSAW_OK;
}

// The hits of all chunks in attempt order, as k_compact, with no scan before it: a block owns
// STATIC_BLOCK chunks and sums the counts of those before them itself (at most 32 KB, from L2).
// Writes nothing when there are more than out_cap hits; the total goes to ctl.
constexpr uint32_t STATIC_BLOCK = 128;
__global__ void __launch_bounds__(256) k_static_finish(const uint32_t* __restrict__ chunk_hits, uint32_t n_chunks,
                                                       const uint2* __restrict__ recs, uint32_t chunk_shift,
                                                       uint64_t a0, int64_t out_cap, uint32_t* __restrict__ ctl,
                                                       uint64_t* __restrict__ out_aid,
                                                       uint32_t* __restrict__ out_len) {
  __shared__ uint32_t before_w[8], total_w[8], own[STATIC_BLOCK], off[STATIC_BLOCK];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t c0 = blockIdx.x * STATIC_BLOCK;
  uint32_t before = 0, total = 0;
  for (uint32_t i = threadIdx.x; i < n_chunks; i += blockDim.x) {
    const uint32_t c = chunk_hits[i];
    total += c;
    if (i < c0) before += c;
    if (i >= c0 && i < c0 + STATIC_BLOCK) own[i - c0] = c;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  total = __reduce_add_sync(0xffffffffu, total);
  if (lane == 0) {
    before_w[w] = before;
    total_w[w] = total;
  }
  __syncthreads();
  before = total = 0;
  for (int i = 0; i < 8; ++i) {
    before += before_w[i];
    total += total_w[i];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl[SC_HITS] = total;
  if ((int64_t)total > out_cap || (ctl[SC_STATUS] & ST_STEP_CAP)) return;
  const uint32_t mine = min(STATIC_BLOCK, n_chunks - c0);
  if (w == 0) {  // offsets of the block's chunks
    uint32_t run = before;
    for (uint32_t i0 = 0; i0 < mine; i0 += 32) {
      const uint32_t v = i0 + lane < mine ? own[i0 + lane] : 0u;
      uint32_t x = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (i0 + lane < mine) off[i0 + lane] = run + x - v;
      run += __shfl_sync(0xffffffffu, x, 31);
    }
  }
  __syncthreads();
  for (uint32_t ck = w; ck < mine; ck += 8) {
    const uint32_t c = own[ck];
    const uint2* r = recs + ((size_t)(c0 + ck) << chunk_shift);
    for (uint32_t i = lane; i < c; i += 32) {
      const uint2 me = r[i];
      uint32_t rank = 0;
      for (uint32_t j = 0; j < c; ++j) rank += (r[j].x < me.x) ? 1u : 0u;
      out_aid[off[ck] + rank] = a0 + me.x;
      out_len[off[ck] + rank] = me.y;
    }
  }
}

}  // namespace hsaw

extern "C" hsaw_status hsaw_sample_hits_static(hsaw_graph g, const uint32_t* suspect_bits, uint64_t seed,
                                               uint64_t first_attempt, int64_t n_attempts, uint64_t* aid_out,
                                               uint32_t* len_out, int64_t out_cap, int64_t* n_hits, void* stream) {
  using namespace hsaw;
  if (!g || !suspect_bits || !n_hits || (out_cap > 0 && (!aid_out || !len_out)))
    return fail(HSAW_E_INVALID, "static sampler: NULL argument");
  *n_hits = 0;
  if (n_attempts < 0 || n_attempts > (int64_t)HSAW_STATIC_MAX_ATTEMPTS)
    return fail(HSAW_E_INVALID, "static sampler: n_attempts must be in [0, HSAW_STATIC_MAX_ATTEMPTS]");
  if (n_attempts == 0) return HSAW_OK;
  const Graph& G = g->g;
  int cur_dev = -1;
  HSAW_CK(cudaGetDevice(&cur_dev));
  if (cur_dev != G.device) return fail(HSAW_E_DEVICE, "static sampler: the current device is not the graph's device");
  StaticScratch* sc = nullptr;
  HSAW_TRY(static_scratch(&sc));
  cudaStream_t s = (cudaStream_t)stream;
  SampleParams P{};
  P.T = G.tables();
  P.s_bits = suspect_bits;
  P.n = (uint32_t)G.n;
  P.k0 = (uint32_t)seed;
  P.k1 = (uint32_t)(seed >> 32);
  P.keys = philox_round_keys(P.k0, P.k1);
  P.step_cap = (uint32_t)std::min<uint64_t>(4ull * (uint64_t)G.n + 64ull, 0xFFFFFFF0ull);
  const uint32_t shift = chunk_shift_for((uint64_t)n_attempts);
  const uint32_t n_chunks = (uint32_t)((n_attempts + (1 << shift) - 1) >> shift);
  P.a0 = first_attempt;
  P.n_attempts = (uint32_t)n_attempts;
  P.chunk_shift = shift;
  P.n_chunks = n_chunks;
  P.cap = 1u << shift;  // room for every attempt of a chunk to hit: no overflow
  P.ctl = sc->ctl;
  P.chunk_hits = sc->ctl + SC_WORDS;
  P.recs = sc->recs;
  // the shared scratch keeps the previous call's contents: clear what must start at zero
  HSAW_CK(cudaMemsetAsync(sc->ctl, 0, ((size_t)SC_WORDS + n_chunks) * sizeof(uint32_t), s));
  const unsigned grid = (unsigned)std::max(1, std::min<int>(sm_count() * sample_blocks_per_sm(),
                                                             (int)((n_chunks + 7) / 8)));
  launch_sample(G, P, grid, s);
  HSAW_CK(cudaGetLastError());
  count_launch();
  k_static_finish<<<(n_chunks + STATIC_BLOCK - 1) / STATIC_BLOCK, 256, 0, s>>>(P.chunk_hits, n_chunks, sc->recs, shift,
                                                                             first_attempt, out_cap, sc->ctl, aid_out,
                                                                             len_out);
  HSAW_CK(cudaGetLastError());
  uint32_t h[SC_WORDS] = {0};
  HSAW_CK(cudaMemcpyAsync(h, sc->ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
  HSAW_CK(cudaStreamSynchronize(s));
  if (h[SC_STATUS] & ST_STEP_CAP) return fail(HSAW_E_STEP_CAP, "static sampler: a walk exceeded its step guard");
  *n_hits = h[SC_HITS];
  if ((int64_t)h[SC_HITS] > out_cap) return fail(HSAW_E_INVALID, "static sampler: more hits than out_cap");
  return HSAW_OK;
}
