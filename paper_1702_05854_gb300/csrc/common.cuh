// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <string>

#include "../../include/hsaw.h"

namespace hsaw {

// ------------------------------------------------------------------ errors
void set_error(const std::string& msg);
hsaw_status fail(hsaw_status st, const std::string& msg);
hsaw_status cuda_fail(cudaError_t e, const char* what, const char* file, int line);

#define HSAW_CK(call)                                                        \
  do {                                                                       \
    cudaError_t e_ = (call);                                                 \
    if (e_ != cudaSuccess) return ::hsaw::cuda_fail(e_, #call, __FILE__, __LINE__); \
  } while (0)

#define HSAW_TRY(expr)                 \
  do {                                 \
    hsaw_status s_ = (expr);           \
    if (s_ != HSAW_OK) return s_;      \
  } while (0)

// ------------------------------------------------------------------ device memory
// Stream-ordered allocations from the device's default memory pool; freed blocks stay
// cached in the pool (release threshold raised at first use), so per-call temporaries
// cost no driver round trip after warm-up.
hsaw_status dmalloc(void** p, size_t bytes, cudaStream_t s);
void dfree(void* p, cudaStream_t s);

// One allocation that a call's small buffers are cut from: while it lives, dmalloc on its thread
// and stream takes what fits from it and dfree leaves that alone.  A small solve makes about 30
// allocations and as many frees, each a microsecond or two and a lock that solves on other
// threads want too.  Buffers cut from it must be gone before it is.
class Slab {
 public:
  explicit Slab(cudaStream_t s);
  ~Slab();
  Slab(const Slab&) = delete;
  Slab& operator=(const Slab&) = delete;
  void* cut(size_t bytes, cudaStream_t s);
  bool holds(const void* p) const { return p >= base_ && p < base_ + cap_; }
  static constexpr size_t BYTES = 32ull << 20;

 private:
  cudaStream_t s_;
  char* base_ = nullptr;
  size_t cap_ = 0, used_ = 0;
  Slab* outer_;
};

// A call that ran out of device memory is made once more without the scratch that only buys time: no
// slab, no counts by element id, no greedy by peaks, no checkpoints of walks, no payload in the edge
// sort.  lean() is true meanwhile, on the call's thread.  call: makes and releases all that it holds.
bool lean();
bool begin_lean(hsaw_status st);  // false: not for a failure that was injected, nor twice
struct LeanEnd {
  ~LeanEnd();
};
template <typename F>
hsaw_status within_memory(F&& call) {
  const hsaw_status st = call();
  if (!begin_lean(st)) return st;
  LeanEnd end;
  return call();
}

template <typename T>
struct DBuf {  // grow-only device buffer
  T* p = nullptr;
  size_t cap = 0;  // elements
  hsaw_status ensure(size_t n, cudaStream_t s, bool keep = false) {
    if (n <= cap) return HSAW_OK;
    size_t nc = cap ? cap : 1024;
    while (nc < n) nc *= 2;
    void* np = nullptr;
    HSAW_TRY(dmalloc(&np, nc * sizeof(T), s));
    if (keep && p && cap) HSAW_CK(cudaMemcpyAsync(np, p, cap * sizeof(T), cudaMemcpyDeviceToDevice, s));
    dfree(p, s);
    p = static_cast<T*>(np);
    cap = nc;
    return HSAW_OK;
  }
  void release(cudaStream_t s) {
    dfree(p, s);
    p = nullptr;
    cap = 0;
  }
};

// ------------------------------------------------------------------ graph
// Device in-adjacency (Sec. 2.1).  node[v] = {first in-edge, in-degree, uniform weight
// (0 if the in-weights differ), in-sum}; edge[e] = {tail node u of (u, v), running sum of
// v's in-weights through e}.  In-edge j of v is live for a draw r iff
// thr[j-1] <= r < thr[j]; none is live when r >= in-sum.
// What a walk reads at each draw depends on where the graph's tables lie (Layout):
//   REC16, REC32: walk records, larger than L2 or well inside it.  A record gives the tail
//     node of an edge and everything the next draw at that node needs in one read, so a walk
//     makes one dependent access per live-edge draw at equal-weight nodes (the tail's node
//     record is replicated per in-edge).  REC16, where every node with in-weight has equal
//     in-weights (as weighted cascade gives): erec[e] = {u, node[u].x, node[u].y, node[u].z}
//     of edge e = (u, v); the in-sum is in-degree times weight.  REC32: erec[2e], erec[2e+1] =
//     {u, node[u].x, node[u].y, node[u].z}, {node[u].w, thr[e], 0, 0}, sector aligned, and for
//     nodes with unequal weights grec[2p], grec[2p+1] (p = first(v) + b), the walk record of
//     the live in-edge j0 of the smallest draw of bucket b = floor(r * deg / in-sum), with j0
//     in the second half's third word: the answer for any r of the bucket is at or after it
//     (Chen & Asau's guide table), usually within a step or two through erec.
//   TAIL4, EDGE8: two or three small reads that L2 holds instead of one that it does not.
//     TAIL4 (equal weights): tail[e] = u, then node[u].  EDGE8: the first in-edge to look at
//     from guide[] (one entry per four in-edges of a node, from guide_base), edges from there
//     four at a time (a sector), then node[u].
// Dependent random reads measured 290 G/s on tables that L2 holds, 83 G/s on 0.27 GB, 55 on
// 0.54 GB, 41 on 2.1 GB and 38 beyond 8 GB.
enum Layout { REC16 = 0, REC32 = 1, TAIL4 = 2, EDGE8 = 3 };
struct WalkTables {
  const uint4* __restrict__ node;
  const uint2* __restrict__ edge;
  const uint4* __restrict__ erec;
  const uint4* __restrict__ grec;
  const uint32_t* __restrict__ tail;
  const uint32_t* __restrict__ guide;
};

// Walk pool (query-independent traces, kept as an inverted index): for walk seed `seed`,
// trace a (a < attempts) is attempt a's walk ignoring sources - its nodes until no live
// in-edge or a detected cycle.  A query's HSAW of attempt a is the trace's prefix up to its
// first real source (the source test is per node, with the same node-keyed coin), so
// attempt a hits exactly when its trace holds a real source.  Attempts are grouped in
// blocks of 2^shift; for block b and node v, ent[boff[b] + noff[b (n + 1) + v] ..
// boff[b] + noff[b (n + 1) + v + 1]) lists (in no particular order, possibly twice) the
// attempts a - (b << shift) of the block whose trace passes through v.
struct WalkPool {
  uint64_t seed = 0;
  uint64_t attempts = 0;
  uint32_t shift = 0;
  uint32_t blocks = 0;
  uint64_t entries = 0;
  uint64_t* boff = nullptr;  // blocks + 1
  uint32_t* noff = nullptr;  // blocks * (n + 1)
  uint32_t* ent = nullptr;   // entries
};

struct Graph {
  int64_t n = 0, m = 0;
  WalkPool pool;
  uint4* node = nullptr;
  uint2* edge = nullptr;
  Layout layout = REC32;
  uint4* erec = nullptr;      // REC16, REC32
  uint4* grec = nullptr;      // REC32
  uint32_t* tail = nullptr;   // TAIL4
  uint32_t* guide = nullptr;  // EDGE8
  WalkTables tables() const { return {node, edge, erec, grec, tail, guide}; }
  int64_t* input_index = nullptr;  // CSR position -> input edge index (NULL = identity)
  int device = 0;
};

// ------------------------------------------------------------------ Philox4x32-10
// Salmon, Moraes, Dror, Shaw, SC'11: 10 rounds of two 32x32->64 multiplies with the
// published multipliers, key bumped by the published Weyl constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

// The same generator with its ten round keys (key + i * the Weyl constants, i = 0..9)
// computed once per launch: a kernel that keeps them in its parameters (constant bank)
// saves the two key additions of every round.
struct PhiloxKeys {
  uint32_t k0[10], k1[10];
};
inline PhiloxKeys philox_round_keys(uint32_t k0, uint32_t k1) {
  PhiloxKeys K;
  for (int i = 0; i < 10; ++i) {
    K.k0[i] = k0 + (uint32_t)i * 0x9E3779B9u;
    K.k1[i] = k1 + (uint32_t)i * 0xBB67AE85u;
  }
  return K;
}
__device__ __forceinline__ uint4 philox4x32_10_rk(uint4 c, const PhiloxKeys& K) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ K.k0[i], lo1, hi0 ^ c.w ^ K.k1[i], lo0);
  }
  return c;
}

// Draw of node v in attempt a (one live-edge world per attempt).
__device__ __forceinline__ uint4 node_draw(uint64_t a, uint32_t v, uint32_t k0, uint32_t k1) {
  return philox4x32_10(make_uint4((uint32_t)a, (uint32_t)(a >> 32), v, 0u), k0, k1);
}
// Start node of attempt a: floor(x0 * n / 2^32).
__device__ __forceinline__ uint32_t start_node(uint64_t a, uint32_t n, uint32_t k0, uint32_t k1) {
  const uint4 x = philox4x32_10(make_uint4((uint32_t)a, (uint32_t)(a >> 32), 0u, 1u), k0, k1);
  return __umulhi(x.x, n);
}
__device__ __forceinline__ bool source_coin(uint32_t x1, uint32_t p32) {
  return p32 == 0xFFFFFFFFu || x1 < p32;
}
// Live in-edge index j in [0, deg) of a node with record nd for draw r < nd.w (in-sum):
// the first j with r < thr[j] (equal weights: j = r / w; otherwise binary search).
__device__ __forceinline__ uint32_t pick_in_edge(const uint2* __restrict__ edge, uint4 nd, uint32_t r) {
  if (nd.z) return r / nd.z;  // equal weights: thr[j] = (j+1) w
  uint32_t lo = 0, hi = nd.y;  // first j with r < thr[j]
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    const uint32_t t = __ldg(&edge[nd.x + mid].y);
    if (r < t) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// Guide-table bucket of draw r at a node with in-degree deg and in-sum insum (r < insum).
__device__ __forceinline__ uint32_t guide_bucket(uint32_t r, uint32_t deg, uint32_t insum) {
  return (uint32_t)(((uint64_t)r * deg) / insum);
}

// Exact cycle detection in registers: the walk keeps the nodes it saw at positions
// 0, 1, 2, 3, 4, 5, 6, 7, 8, 10, 12, 15, 18, ... (each 1.25x the last), the 8 newest in
// registers.  A tail node equal to a kept node is a revisit, so the world's backward chain
// is a cycle (miss); a cycle entered at position mu is seen within about 0.25 mu + lambda
// draws, against mu + lambda for a whole-walk check and about 2 (mu + lambda) for Brent.
struct Ckpt {
  uint32_t c0, c1, c2, c3, c4, c5, c6, c7;  // newest first
  uint32_t next;
  __device__ __forceinline__ void reset(uint32_t v) {
    c0 = c1 = c2 = c3 = c4 = c5 = c6 = c7 = v;
    next = 1;
  }
  __device__ __forceinline__ bool seen(uint32_t u) const {
    return (u == c0) | (u == c1) | (u == c2) | (u == c3) | (u == c4) | (u == c5) | (u == c6) | (u == c7);
  }
  // u is the node at walk position pos (>= 1)
  __device__ __forceinline__ void keep(uint32_t u, uint32_t pos) {
    if (pos < next) return;
    c7 = c6; c6 = c5; c5 = c4; c4 = c3; c3 = c2; c2 = c1; c1 = c0; c0 = u;
    next = after(next);
  }
  // the position kept after `pos`: 1, 2, ..., 8, 10, 12, 15, ...
  static __device__ __forceinline__ uint32_t after(uint32_t pos) { return pos + max(1u, pos >> 2); }
};

// ------------------------------------------------------------------ primitives (primitives.cu)
// Exclusive prefix sum in place; *total (device, may be NULL) receives the sum.
hsaw_status exclusive_scan_u32(uint32_t* d, size_t n, uint32_t* total, cudaStream_t s);
hsaw_status exclusive_scan_u64(uint64_t* d, size_t n, uint64_t* total, cudaStream_t s);
// Stable LSD radix sort of (key, value) pairs on the low `bits` bits of the key.  The
// result ends in (keys, vals) or (keys_alt, vals_alt); *in_alt tells which.
hsaw_status radix_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* keys_alt, uint32_t* vals_alt, size_t n,
                             int bits, cudaStream_t s, bool* in_alt);
// The edge list (src, dst, w) sorted by dst, stable: edge = {src, w} and index = input position in
// sorted order; *sorted_dst is keys or keys_alt.  A node at or above `nodes` (2 at least) sets bit
// 0 of *err.  keys, keys_alt, vals, vals_alt, pay: room for m each; m >= 1.
hsaw_status radix_sort_edges(const int32_t* src, const int32_t* dst, const uint32_t* w, size_t m, uint32_t nodes,
                             uint32_t* keys, uint32_t* keys_alt, uint32_t* vals, uint32_t* vals_alt, uint2* pay,
                             uint2* edge, int64_t* index, uint32_t** sorted_dst, uint32_t* err, cudaStream_t s);
int bit_width(uint64_t x);  // bits needed for values in [0, x]

// ------------------------------------------------------------------ launch helpers
inline unsigned grid_for(size_t n, unsigned block, unsigned cap = 1u << 30) {
  size_t g = (n + block - 1) / block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (unsigned)g;
}
int sm_count();

// Launch accounting (profiling): every kernel launch of the library calls count_launch();
// sampler launches are bracketed by profile_begin / profile_end.
void count_launch();
void* profile_begin(cudaStream_t s);
void profile_end(void* token, cudaStream_t s, uint64_t attempts);
void profile_add_steps(uint64_t steps);
// Phase timing (profiling only): 0 sampling, 1 counting + index, 2 greedy, 3 coverage.
enum { PH_SAMPLE = 0, PH_COUNT = 1, PH_GREEDY = 2, PH_COVERAGE = 3 };
void* phase_begin(cudaStream_t s);
void phase_end(void* token, cudaStream_t s, int phase);

// ------------------------------------------------------------------ walk-record steps
// One 32-byte walk record in ONE 256-bit load (p is 32-byte aligned: records start at a
// cudaMalloc base).  As two 16-byte loads every record costs two L1 and two L2 requests for
// the same sector: dependent random reads measured 29-32 G/s that way on tables of 2-34 GB
// and 205 G/s in L2, against 38-41 and 290 G/s as one load (6 blocks of 256 per SM).  volatile:
// without it the compiler may take the read for free of effects and hoist it above the test
// that makes its address valid.
__device__ __forceinline__ void load_record(const uint4* __restrict__ p, uint4& a, uint4& b) {
  asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
      : "l"(p));
}

// floor(r / w), w >= 1, from a float estimate that is never above it: the conversions, the
// factor and the approximate quotient (2 ulp) are off by less than 2^-20 together, which the
// factor takes off, so the estimate is the quotient or, below 2^19, at most one less.  About
// half the instructions of the integer division.
__device__ __forceinline__ uint32_t quotient(uint32_t r, uint32_t w) {
  uint32_t q = __float2uint_rz(__fdividef(__uint2float_rn(r) * (1.0f - 0x1p-20f), __uint2float_rn(w)));
  uint32_t rem = r - q * w;
  if (rem >= w) {
    ++q;
    rem -= w;
    if (rem >= w) q = r / w;
  }
  return q;
}

// EDGE8: node v's guide entries start here, one per four in-edges (rounded up), which bases of
// consecutive nodes leave room for.
__device__ __forceinline__ uint32_t guide_base(uint32_t first, uint32_t v) { return (first >> 2) + v; }
// The guide entry of draw r < insum.  The float arithmetic is off by less than 2^-21 of the
// bucket's number, so r >= b insum / buckets (1 - 2^-20): guide[] is built for that draw.
__device__ __forceinline__ uint32_t guide_entry(uint32_t r, uint32_t deg, uint32_t insum) {
  const uint32_t buckets = (deg + 3) >> 2;
  const uint32_t b = __float2uint_rz(__uint2float_rz(r) *
                                     __fdividef(__uint2float_rn(buckets), __uint2float_rn(insum)));
  return min(b, buckets - 1);
}

// The live in-edge e of node v with record rec = {first in-edge, in-degree, equal weight or
// 0, in-sum} for a draw r < rec.w, read through the graph's tables (the same choice as
// pick_in_edge: j = r / w at equal weights, otherwise the first j with r < thr[j]).  u
// receives e's tail, next the tail's record.
template <Layout L>
__device__ __forceinline__ uint32_t record_step(const WalkTables& T, uint32_t v, uint4 rec, uint32_t r, uint32_t& u,
                                                uint4& next) {
  uint32_t e;
  if (L == REC16) {
    e = rec.x + quotient(r, rec.z);
    const uint4 x = __ldg(&T.erec[e]);
    u = x.x;
    next = make_uint4(x.y, x.z, x.w, x.z * x.w);
  } else if (L == TAIL4) {
    e = rec.x + quotient(r, rec.z);
    u = __ldg(&T.tail[e]);
    next = __ldg(&T.node[u]);
  } else if (L == REC32) {
    uint4 ra, rb;
    if (rec.z) {
      e = rec.x + quotient(r, rec.z);
      load_record(T.erec + 2 * (size_t)e, ra, rb);
    } else {
      load_record(T.grec + 2 * ((size_t)rec.x + guide_bucket(r, rec.y, rec.w)), ra, rb);
      e = rec.x + rb.z;
      while (r >= rb.y) {
        ++e;
        load_record(T.erec + 2 * (size_t)e, ra, rb);
      }
    }
    u = ra.x;
    next = make_uint4(ra.y, ra.z, ra.w, rb.x);
  } else {
    if (rec.z) {
      e = rec.x + quotient(r, rec.z);
      u = __ldg(&T.edge[e].x);
    } else {
      e = rec.x + __ldg(&T.guide[guide_base(rec.x, v) + guide_entry(r, rec.y, rec.w)]);
      for (;;) {  // r < thr of the list's last edge, so the search ends inside the list
        const uint32_t at = e & ~3u;
        uint4 a, b;  // edges at .. at + 3, {tail, running sum} each
        load_record(reinterpret_cast<const uint4*>(T.edge + at), a, b);
        uint32_t past = (r < a.y ? 1u : 0u) | (r < a.w ? 2u : 0u) | (r < b.y ? 4u : 0u) | (r < b.w ? 8u : 0u);
        past &= 0xFu << (e & 3u);
        if (past) {
          const uint32_t i = __ffs(past) - 1;
          e = at + i;
          u = i == 0 ? a.x : i == 1 ? a.z : i == 2 ? b.x : b.z;
          break;
        }
        e = at + 4;
      }
    }
    next = __ldg(&T.node[u]);
  }
  return e;
}

}  // namespace hsaw

// Opaque handle types of the ABI.
struct hsaw_graph_s {
  hsaw::Graph g;
};
