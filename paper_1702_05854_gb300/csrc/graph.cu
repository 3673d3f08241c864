// Graph ingest (Sec. 2.1): edge list or CSR -> device in-adjacency with running uint32
// in-weight sums, per-node records and validation of the LT in-weight condition.
#include <cuda_runtime.h>

#include <atomic>
#include <cstring>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "common.cuh"

namespace hsaw {

// ------------------------------------------------------------------ errors / memory
static thread_local std::string t_err;
void set_error(const std::string& msg) { t_err = msg; }
const char* last_error() { return t_err.c_str(); }
hsaw_status fail(hsaw_status st, const std::string& msg) {
  t_err = msg;
  return st;
}
static thread_local bool t_lean = false, t_refused = false;  // the allocator had no memory
bool lean() { return t_lean; }
bool begin_lean(hsaw_status st) {
  const bool again = st == HSAW_E_NOMEM && t_refused && !t_lean;
  t_refused = false;
  if (again) t_lean = true;
  return again;
}
LeanEnd::~LeanEnd() { t_lean = false; }
hsaw_status cuda_fail(cudaError_t e, const char* what, const char* file, int line) {
  char buf[512];
  snprintf(buf, sizeof(buf), "%s failed: %s (%s:%d)", what, cudaGetErrorString(e), file, line);
  t_err = buf;
  if (e == cudaErrorMemoryAllocation) t_refused = true;
  return (e == cudaErrorMemoryAllocation) ? HSAW_E_NOMEM : HSAW_E_DEVICE;
}

static std::once_flag g_pool_once;
static std::atomic<long long> g_fail_countdown{0};  // test hook: > 0 counts down to a failing allocation

// Scratch allocator: CUDA's stream-ordered pool, or the caller's (hsaw_set_allocator).  The
// allocator changes only while no scratch block is held and no other call runs, so every
// block goes back to the allocator it came from; allocations read it without a lock.
struct ScratchAllocator {
  hsaw_alloc_fn alloc;
  hsaw_free_fn release;
  void* ctx;
};
static std::mutex g_alloc_set_mu;                          // serialises changes
static std::vector<std::unique_ptr<ScratchAllocator>> g_alloc_all;  // every one installed, kept to exit
static std::atomic<const ScratchAllocator*> g_alloc{nullptr};
static std::atomic<long long> g_held{0};                   // scratch blocks handed out, not yet released

static thread_local Slab* t_slab = nullptr;
static hsaw_status allocate(void** p, size_t bytes, cudaStream_t s);

Slab::Slab(cudaStream_t s) : s_(s), outer_(t_slab) {
  void* p = nullptr;
  if (!lean() && allocate(&p, BYTES, s) == HSAW_OK) {
    base_ = static_cast<char*>(p);
    cap_ = BYTES;
  } else {
    set_error("");  // small buffers are then allocated one by one
    t_refused = false;
  }
  t_slab = this;
}

Slab::~Slab() {
  t_slab = nullptr;
  dfree(base_, s_);
  t_slab = outer_;
}

void* Slab::cut(size_t bytes, cudaStream_t s) {
  bytes = (bytes + 255) & ~(size_t)255;
  if (s != s_ || bytes > cap_ - used_) return nullptr;
  void* p = base_ + used_;
  used_ += bytes;
  return p;
}

hsaw_status dmalloc(void** p, size_t bytes, cudaStream_t s) {
  if (g_fail_countdown.load(std::memory_order_relaxed) > 0 && g_fail_countdown.fetch_sub(1) == 1) {
    *p = nullptr;
    t_refused = false;
    t_err = "device allocation failed (injected by hsaw_debug_fail_alloc_after)";
    return HSAW_E_NOMEM;
  }
  if (bytes == 0) bytes = 16;
  if (t_slab && (*p = t_slab->cut(bytes, s))) return HSAW_OK;
  return allocate(p, bytes, s);
}

// From the allocator itself.
static hsaw_status allocate(void** p, size_t bytes, cudaStream_t s) {
  if (const ScratchAllocator* a = g_alloc.load(std::memory_order_acquire)) {
    *p = a->alloc(bytes, (void*)s, a->ctx);
    if (!*p) {
      t_refused = true;
      char buf[128];
      snprintf(buf, sizeof(buf), "device allocation of %zu bytes failed (caller's allocator)", bytes);
      t_err = buf;
      return HSAW_E_NOMEM;
    }
    g_held.fetch_add(1);
    return HSAW_OK;
  }
  std::call_once(g_pool_once, [] {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
      uint64_t thr = UINT64_MAX;
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
  });
  cudaError_t e = cudaMallocAsync(p, bytes, s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    t_refused = true;
    char buf[128];
    snprintf(buf, sizeof(buf), "device allocation of %zu bytes failed: %s", bytes, cudaGetErrorString(e));
    t_err = buf;
    return HSAW_E_NOMEM;
  }
  g_held.fetch_add(1);
  return HSAW_OK;
}
void dfree(void* p, cudaStream_t s) {
  if (!p || (t_slab && t_slab->holds(p))) return;
  if (const ScratchAllocator* a = g_alloc.load(std::memory_order_acquire))
    a->release(p, (void*)s, a->ctx);
  else
    cudaFreeAsync(p, s);
  g_held.fetch_sub(1);
}

// ------------------------------------------------------------------ kernels
enum : uint32_t { ERR_RANGE = 1u, ERR_WEIGHT = 2u, ERR_ROWPTR = 4u };

__global__ void k_validate_nodes(const int32_t* __restrict__ a, int64_t m, int64_t n, uint32_t* __restrict__ err) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
    if (a[e] < 0 || a[e] >= n) atomicOr(err, ERR_RANGE);
}

__global__ void k_iota_dst(const int32_t* __restrict__ dst, int64_t m, uint32_t* __restrict__ keys,
                           uint32_t* __restrict__ vals) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    keys[e] = (uint32_t)dst[e];
    vals[e] = (uint32_t)e;
  }
}

// row_start[v] = first CSR position of v (lower bound of v in the sorted destinations).
__global__ void k_row_from_sorted(const uint32_t* __restrict__ sorted_dst, int64_t m, int64_t n,
                                  uint32_t* __restrict__ row_start) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v <= n; v += (int64_t)gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = m;
    while (lo < hi) {
      int64_t mid = (lo + hi) >> 1;
      if ((int64_t)sorted_dst[mid] < v) lo = mid + 1; else hi = mid;
    }
    row_start[v] = (uint32_t)lo;
  }
}

__global__ void k_gather_edges(const uint32_t* __restrict__ perm, const int32_t* __restrict__ src,
                               const uint32_t* __restrict__ w, int64_t m, uint2* __restrict__ edge,
                               int64_t* __restrict__ input_index) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < m; q += (int64_t)gridDim.x * blockDim.x) {
    uint32_t e = perm[q];
    edge[q] = make_uint2((uint32_t)src[e], w[e]);
    if (input_index) input_index[q] = e;
  }
}

__global__ void k_csr_rows(const int64_t* __restrict__ rp, int64_t n, int64_t m, uint32_t* __restrict__ row_start,
                           uint32_t* __restrict__ err) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v <= n; v += (int64_t)gridDim.x * blockDim.x) {
    int64_t a = rp[v];
    if (a < 0 || a > m || (v < n && rp[v + 1] < a) || (v == 0 && a != 0) || (v == n && a != m))
      atomicOr(err, ERR_ROWPTR);
    row_start[v] = (uint32_t)(a < 0 ? 0 : (a > m ? m : a));
  }
}

__global__ void k_copy_edges(const int32_t* __restrict__ src, const uint32_t* __restrict__ w, int64_t m, int64_t n,
                             uint2* __restrict__ edge, uint32_t* __restrict__ err) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < m; q += (int64_t)gridDim.x * blockDim.x) {
    int32_t a = src[q];
    if (a < 0 || a >= n) atomicOr(err, ERR_RANGE);
    edge[q] = make_uint2((uint32_t)a, w[q]);
  }
}

// Running in-weight sums (exact, 64-bit carry), the in-sum check (<= 2^32 - 1), equal-weight
// detection and the node record: a warp per 32 nodes, and a block per hub (a node of more
// than HUB_DEGREE in-edges), which the warp pass only lists.  In the warp pass the longest list
// alone set the pass's time (R-MAT 22: 3.1 ms, R-MAT 20: 1.3 ms).  err[1] counts the nodes with in-weight whose in-weights differ.
constexpr uint32_t HUB_DEGREE = 1024;

// Hubs of the graph: count, then node ids (at most m / HUB_DEGREE of them).
struct Hubs {
  uint32_t* count;
  uint32_t* node;
};

__device__ __forceinline__ uint32_t clamp32(uint64_t x) { return x > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)x; }

__device__ __forceinline__ void write_node(uint4* __restrict__ node, int64_t v, uint32_t first, uint32_t deg,
                                           bool uniform, uint32_t w0, uint64_t sum, uint32_t* __restrict__ err) {
  node[v] = make_uint4(first, deg, (uniform && deg) ? w0 : 0u, clamp32(sum));
  if (sum > 0xFFFFFFFFull) atomicOr(err, ERR_WEIGHT);
}

// A warp takes 32 nodes, a lane each for lists of up to SHORT_LIST edges; longer lists are taken
// 32 edges at a time by the whole warp, the next 32 (of the same node or the next) being read
// meanwhile.  Where 32 in-weights are equal their sums are multiples, without a scan.  Bound by
// instructions before (a warp a node, a 64-bit scan for every 32 edges):
// R-MAT 22, equal weights, 656 -> 324 us; R-MAT 20, random weights, 292 -> 232 us.
__global__ void __launch_bounds__(256) k_thresholds(const uint32_t* __restrict__ row_start, int64_t n,
                                                    uint2* __restrict__ edge, uint4* __restrict__ node, Hubs hubs,
                                                    uint32_t* __restrict__ err) {
  constexpr uint32_t SHORT_LIST = 8;
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v0 = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * 32; v0 < n; v0 += warps * 32) {
    const int64_t v = v0 + lane;
    const uint32_t b = v < n ? row_start[v] : 0u, e = v < n ? row_start[v + 1] : 0u, deg = e - b;
    const bool hub = deg > HUB_DEGREE;
    if (hub) hubs.node[atomicAdd(hubs.count, 1u)] = (uint32_t)v;
    uint64_t sum = 0;
    uint32_t w0 = 0;
    bool uniform = true;
    if (deg && deg <= SHORT_LIST) {
      uint32_t w[SHORT_LIST];
#pragma unroll
      for (uint32_t i = 0; i < SHORT_LIST; ++i) w[i] = i < deg ? edge[b + i].y : 0u;
      w0 = w[0];
#pragma unroll
      for (uint32_t i = 0; i < SHORT_LIST; ++i) {
        if (i >= deg) break;
        sum += w[i];
        uniform &= w[i] == w0;
        edge[b + i].y = clamp32(sum);
      }
    }
    unsigned left = __ballot_sync(FULL, deg > SHORT_LIST && !hub);
    int cur = left ? __ffs(left) - 1 : -1;
    uint32_t first = __shfl_sync(FULL, b, cur & 31), end = __shfl_sync(FULL, e, cur & 31), base = first;
    uint32_t w = cur >= 0 && base + lane < end ? edge[base + lane].y : 0u;
    uint64_t carry = 0;
    uint32_t start_w = 0;
    bool same = true;  // all of the node's in-weights so far
    while (cur >= 0) {
      int next = cur;
      uint32_t next_first = first, next_end = end, next_base = base + 32;
      if (next_base >= end) {
        left &= left - 1;
        next = left ? __ffs(left) - 1 : -1;
        next_first = next_base = __shfl_sync(FULL, b, next & 31);
        next_end = __shfl_sync(FULL, e, next & 31);
      }
      const uint32_t next_w = next >= 0 && next_base + lane < next_end ? edge[next_base + lane].y : 0u;
      if (base == first) {
        carry = 0;
        same = true;
        start_w = __shfl_sync(FULL, w, 0);
      }
      const bool in = base + lane < end;
      uint64_t x, all;
      if (__all_sync(FULL, !in || w == start_w)) {
        x = (uint64_t)start_w * (lane + 1);
        all = (uint64_t)start_w * min(32u, end - base);
      } else {
        same = false;
        x = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint64_t y = __shfl_up_sync(FULL, x, o);
          if (lane >= o) x += y;
        }
        all = __shfl_sync(FULL, x, 31);
      }
      if (in) edge[base + lane].y = clamp32(carry + x);
      carry += all;
      if (next != cur && lane == cur) {
        sum = carry;
        w0 = start_w;
        uniform = same;
      }
      cur = next;
      first = next_first;
      end = next_end;
      base = next_base;
      w = next_w;
    }
    if (v < n && !hub) write_node(node, v, b, deg, uniform, w0, sum, err);
    const unsigned unequal = __ballot_sync(FULL, !uniform && clamp32(sum));
    if (lane == 0 && unequal) atomicAdd(err + 1, (uint32_t)__popc(unequal));
  }
}

// A block a hub, a tile of 2 K edges at a time, the next tile's in-weights being read while this
// one's sums are made: many hubs have a tile or two, so four small blocks an SM, not one of 1,024
// threads (R-MAT 22 358 -> 240 us, R-MAT 20 93 -> 70 us; 301 and 72 us with tiles of 8 K).
constexpr int HUB_WARPS = 8;
__global__ void __launch_bounds__(HUB_WARPS * 32, 4) k_hub_thresholds(const uint32_t* __restrict__ row_start,
                                                         uint2* __restrict__ edge, uint4* __restrict__ node, Hubs hubs,
                                                         uint32_t* __restrict__ err) {
  constexpr uint32_t ITEMS = 8, TILE = ITEMS * HUB_WARPS * 32;
  __shared__ uint64_t sums[2][HUB_WARPS];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t count = *hubs.count;
  for (uint32_t h = blockIdx.x; h < count; h += gridDim.x) {
    const uint32_t v = hubs.node[h];
    const uint32_t b = row_start[v], e = row_start[v + 1];
    const uint32_t w0 = edge[b].y;
    uint32_t x[ITEMS];
#pragma unroll
    for (uint32_t i = 0; i < ITEMS; ++i) {
      const uint32_t q = b + threadIdx.x * ITEMS + i;
      x[i] = q < e ? edge[q].y : 0u;
    }
    __syncthreads();  // every thread has read edge[b] before it is written
    uint64_t carry = 0;
    bool uniform = true;
    uint32_t turn = 0;
    for (uint32_t base = b; base < e; base += TILE, turn ^= 1) {
      const uint32_t q = base + threadIdx.x * ITEMS;
      uint32_t next[ITEMS];
      uint64_t sum = 0;
#pragma unroll
      for (uint32_t i = 0; i < ITEMS; ++i) {
        const uint64_t p = (uint64_t)q + TILE + i;
        next[i] = p < e ? edge[p].y : 0u;
      }
#pragma unroll
      for (uint32_t i = 0; i < ITEMS; ++i) {
        if (q + i < e && x[i] != w0) uniform = false;
        sum += x[i];
      }
      uint64_t inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) sums[turn][w] = inc;
      __syncthreads();  // the other turn's sums are read before this, and written after the next
      uint64_t mine = lane < HUB_WARPS ? sums[turn][lane] : 0ull;
#pragma unroll
      for (int o = 1; o < HUB_WARPS; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, mine, o);
        if (lane >= o) mine += y;
      }
      const uint64_t before = __shfl_sync(0xffffffffu, mine, (w + 31) & 31);
      uint64_t at = carry + (w ? before : 0ull) + inc - sum;
      carry += __shfl_sync(0xffffffffu, mine, HUB_WARPS - 1);
#pragma unroll
      for (uint32_t i = 0; i < ITEMS; ++i) {
        at += x[i];
        if (q + i < e) edge[q + i].y = clamp32(at);
        x[i] = next[i];
      }
    }
    uniform = __syncthreads_and(uniform);
    if (threadIdx.x == 0) {
      write_node(node, v, b, e - b, uniform, w0, carry, err);
      if (!uniform && clamp32(carry)) atomicAdd(err + 1, 1u);
    }
  }
}

// Walk records (see Graph::erec).
template <bool EQ>
__global__ void k_walk_records(const uint2* __restrict__ edge, const uint4* __restrict__ node, int64_t m,
                               uint4* __restrict__ erec) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    const uint2 ed = edge[e];
    const uint4 nu = node[ed.x];
    if (EQ) {
      erec[e] = make_uint4(ed.x, nu.x, nu.y, nu.z);
    } else {
      erec[2 * e] = make_uint4(ed.x, nu.x, nu.y, nu.z);
      erec[2 * e + 1] = make_uint4(nu.w, ed.y, 0u, 0u);
    }
  }
}

// Bucket record b of a node with unequal in-weights (see Graph::grec): the walk record of the
// live in-edge of the bucket's smallest draw.
__device__ __forceinline__ void guide_record(uint4 nd, uint32_t b, const uint2* __restrict__ edge,
                                             const uint4* __restrict__ erec, uint4* __restrict__ grec) {
  const uint32_t lb = (uint32_t)(((uint64_t)b * nd.w + nd.y - 1) / nd.y);  // ceil(b * insum / deg)
  uint32_t lo = 0, hi = nd.y;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (lb < edge[nd.x + mid].y) hi = mid; else lo = mid + 1;
  }
  const size_t p = 2 * ((size_t)nd.x + b), e = 2 * ((size_t)nd.x + lo);
  grec[p] = erec[e];
  uint4 second = erec[e + 1];
  second.z = lo;
  grec[p + 1] = second;
}

// EDGE8: guide entry b of a node with unequal in-weights, the live in-edge of the smallest draw
// that may look it up (see guide_entry).
__device__ __forceinline__ void guide_first(uint4 nd, uint32_t v, uint32_t b, const uint2* __restrict__ edge,
                                            uint32_t* __restrict__ guide) {
  const uint32_t buckets = (nd.y + 3) >> 2;
  const uint32_t at = (uint32_t)((uint64_t)b * nd.w / buckets), off = (at >> 20) + 1;
  const uint32_t lb = at > off ? at - off : 0u;
  uint32_t lo = 0, hi = nd.y;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (lb < edge[nd.x + mid].y) hi = mid; else lo = mid + 1;
  }
  guide[guide_base(nd.x, v) + b] = lo;
}

// One warp per node, and a block per slice of a hub's buckets (one warp on the longest list
// took the whole pass: 4.7 ms on R-MAT 20).  grec: bucket records (REC32), else guide (EDGE8).
__global__ void k_guide(const uint4* __restrict__ node, const uint2* __restrict__ edge, int64_t n,
                        const uint4* __restrict__ erec, uint4* __restrict__ grec, uint32_t* __restrict__ guide) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
    const uint4 nd = node[v];
    if (nd.z != 0 || nd.w == 0 || nd.y > HUB_DEGREE) continue;  // equal weights, no in-weight, or a hub
    if (grec)
      for (uint32_t b = lane; b < nd.y; b += 32) guide_record(nd, b, edge, erec, grec);
    else
      for (uint32_t b = lane; b < (nd.y + 3) >> 2; b += 32) guide_first(nd, (uint32_t)v, b, edge, guide);
  }
}

__global__ void __launch_bounds__(256) k_hub_guide(const uint4* __restrict__ node, const uint2* __restrict__ edge,
                                                   Hubs hubs, const uint4* __restrict__ erec,
                                                   uint4* __restrict__ grec, uint32_t* __restrict__ guide) {
  constexpr uint32_t SLICES = 16;
  const uint64_t items = (uint64_t)*hubs.count * SLICES;
  for (uint64_t i = blockIdx.x; i < items; i += gridDim.x) {
    const uint32_t v = hubs.node[i / SLICES];
    const uint4 nd = node[v];
    if (nd.z != 0 || nd.w == 0) continue;
    const uint32_t buckets = grec ? nd.y : (nd.y + 3) >> 2;
    for (uint32_t b = (uint32_t)(i % SLICES) * blockDim.x + threadIdx.x; b < buckets; b += SLICES * blockDim.x) {
      if (grec) guide_record(nd, b, edge, erec, grec);
      else guide_first(nd, v, b, edge, guide);
    }
  }
}

__global__ void k_tails(const uint2* __restrict__ edge, int64_t m, uint32_t* __restrict__ tail) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
    tail[e] = edge[e].x;
}

// ------------------------------------------------------------------ host
// d_err: error bits, then the count of unequal nodes (k_thresholds) into *unequal.
static hsaw_status check_err(uint32_t* d_err, cudaStream_t s, uint32_t* unequal = nullptr) {
  uint32_t word[2] = {0, 0};
  HSAW_CK(cudaMemcpyAsync(word, d_err, sizeof(word), cudaMemcpyDeviceToHost, s));
  HSAW_CK(cudaStreamSynchronize(s));
  const uint32_t h = word[0];
  if (unequal) *unequal = word[1];
  if (h & ERR_RANGE) return fail(HSAW_E_RANGE, "graph: a node index is outside [0, n)");
  if (h & ERR_ROWPTR) return fail(HSAW_E_INVALID, "graph: in_row_ptr is not a valid CSR offset array");
  if (h & ERR_WEIGHT) return fail(HSAW_E_WEIGHT_SUM, "graph: a node's in-weight sum exceeds 2^32 - 1");
  return HSAW_OK;
}

// True for page-locked (pinned or registered) host memory, whose copies run asynchronously.
static bool host_pinned(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeHost;
}

template <typename T>
static hsaw_status stage(const T* p, size_t count, bool on_device, cudaStream_t s, T** dev, bool* owned) {
  *owned = false;
  if (on_device || count == 0) {
    *dev = const_cast<T*>(p);
    return HSAW_OK;
  }
  HSAW_TRY(dmalloc((void**)dev, count * sizeof(T), s));
  *owned = true;
  const cudaError_t e = cudaMemcpyAsync(*dev, p, count * sizeof(T), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) {
    dfree(*dev, s);
    *dev = nullptr;
    *owned = false;
    return cuda_fail(e, "cudaMemcpyAsync(graph input)", __FILE__, __LINE__);
  }
  return HSAW_OK;
}

void pool_release(WalkPool& p);

static void destroy_graph(Graph& g) {
  pool_release(g.pool);
  if (g.node) cudaFree(g.node);
  if (g.edge) cudaFree(g.edge);
  if (g.input_index) cudaFree(g.input_index);
  if (g.erec) cudaFree(g.erec);
  if (g.grec) cudaFree(g.grec);
  if (g.tail) cudaFree(g.tail);
  if (g.guide) cudaFree(g.guide);
  g.erec = nullptr;
  g.grec = nullptr;
  g.tail = nullptr;
  g.guide = nullptr;
  g.node = nullptr;
  g.edge = nullptr;
  g.input_index = nullptr;
}

static hsaw_status alloc_graph(Graph& g, int64_t n, int64_t m, bool with_index) {
  g.n = n;
  g.m = m;
  cudaGetDevice(&g.device);
  HSAW_CK(cudaMalloc((void**)&g.node, (size_t)n * sizeof(uint4)));
  HSAW_CK(cudaMalloc((void**)&g.edge, (size_t)(m + 4) / 4 * 4 * sizeof(uint2)));
  if (with_index) HSAW_CK(cudaMalloc((void**)&g.input_index, (size_t)(m ? m : 1) * sizeof(int64_t)));
  return HSAW_OK;
}

// A second stream (with one event) for copies that overlap work on the call's stream; it is
// drained and destroyed when the call returns, before its temporaries are freed.
struct SideStream {
  cudaStream_t s = nullptr;
  cudaEvent_t ev = nullptr;
  hsaw_status create() {
    HSAW_CK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    HSAW_CK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    return HSAW_OK;
  }
  ~SideStream() {
    if (s) {
      cudaStreamSynchronize(s);
      cudaStreamDestroy(s);
    }
    if (ev) cudaEventDestroy(ev);
  }
};

struct Temps {
  std::vector<void*> ptrs;
  cudaStream_t s;
  explicit Temps(cudaStream_t st) : s(st) {}
  template <typename T>
  hsaw_status get(T** p, size_t count) {
    HSAW_TRY(dmalloc((void**)p, (count ? count : 1) * sizeof(T), s));
    ptrs.push_back(*p);
    return HSAW_OK;
  }
  void keep(void* p) { ptrs.push_back(p); }
  ~Temps() {
    for (void* p : ptrs) dfree(p, s);
  }
};

// Walk tables by size (see Layout): the small ones where the records do not fit L2 and the
// small ones do, or nearly.  Sampler, G draws/s, records against small tables, R-MAT edge
// factor 16 (L2 129 MB): equal weights, scale 18 to 23: 171/135, 111/122, 70/98, 51/63, 44/46,
// 40/36; random weights, scale 16 to 22: 78/84, 73/85, 65/82, 54/73, 46/58, 40/40, 36/30.
// M attempts/s at other edge factors, records against small tables: equal weights, edge factor 4, scale
// 21 to 24: 7168/7674, 5521/6712, 4588/5045, 3939/3648; 8, scale 20 to 24: 4586/4807, 3065/4024,
// 2305/2747, 1998/2003, 1912/1631; 32, scale 18 to 22: 2615/3046, 1393/2117, 957/1396, 779/903, 620/607;
// 64, scale 17 to 21: 2422/2753, 1297/2252, 874/1350, 666/813, 520/526.  Random weights, edge factor 4,
// scale 18 to 23: 52808/55342, 48652/49642, 44449/51295, 37367/44164, 31268/32594, 27746/24153; 64, scale
// 15 to 21: 23974/28090, 21248/27152, 18875/26483, 16529/22904, 15543/17713, 14644/13173, 14191/10589.
// The rule takes the faster of the two or one within 4% of it at 73 of 76 sizes; right at 16 M = L2 it
// leaves up to 17% (edge factor 32, scale 18).
static Layout choose_layout(int64_t n, int64_t m, bool eq) {
  static const double l2 = [] {
    int dev = 0, bytes = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&bytes, cudaDevAttrL2CacheSize, dev);
    return (double)bytes;
  }();
  const double N = (double)n, M = (double)m;
  if (eq) return 16 * M > l2 && 4 * M + 16 * N <= 3.0 * l2 ? TAIL4 : REC16;
  return 64 * M > 0.25 * l2 && 9 * M + 20 * N <= 2.6 * l2 ? EDGE8 : REC32;
}

static hsaw_status finish_graph(Graph& g, uint32_t* row_start, uint32_t* d_err, Temps& T, cudaStream_t s) {
  const int64_t n = g.n;
  Hubs hubs;
  HSAW_TRY(T.get(&hubs.count, 1 + (size_t)(g.m / HUB_DEGREE)));
  hubs.node = hubs.count + 1;
  HSAW_CK(cudaMemsetAsync(hubs.count, 0, sizeof(uint32_t), s));
  count_launch();
  k_thresholds<<<grid_for((size_t)n, 256, 1u << 20), 256, 0, s>>>(row_start, n, g.edge, g.node, hubs, d_err);
  HSAW_CK(cudaGetLastError());
  if (g.m > HUB_DEGREE) {
    count_launch();
    k_hub_thresholds<<<grid_for((size_t)(g.m / HUB_DEGREE), 1, 4 * sm_count()), HUB_WARPS * 32, 0, s>>>(
        row_start, g.edge, g.node, hubs, d_err);
    HSAW_CK(cudaGetLastError());
  }
  uint32_t unequal = 0;
  HSAW_TRY(check_err(d_err, s, &unequal));
  if (!g.m) return HSAW_OK;
  g.layout = choose_layout(n, g.m, unequal == 0);
  if (g.layout == TAIL4) {
    HSAW_CK(cudaMalloc((void**)&g.tail, (size_t)g.m * sizeof(uint32_t)));
    count_launch();
    k_tails<<<grid_for(g.m, 256, 1u << 16), 256, 0, s>>>(g.edge, g.m, g.tail);
    HSAW_CK(cudaGetLastError());
    return HSAW_OK;
  }
  if (g.layout == EDGE8) {
    HSAW_CK(cudaMalloc((void**)&g.guide, ((size_t)g.m / 4 + (size_t)n + 1) * sizeof(uint32_t)));
  } else {
    HSAW_CK(cudaMalloc((void**)&g.erec, (size_t)g.m * (g.layout == REC16 ? 1 : 2) * sizeof(uint4)));
    count_launch();
    if (g.layout == REC16) {
      k_walk_records<true><<<grid_for(g.m, 256, 1u << 16), 256, 0, s>>>(g.edge, g.node, g.m, g.erec);
      HSAW_CK(cudaGetLastError());
      return HSAW_OK;
    }
    k_walk_records<false><<<grid_for(g.m, 256, 1u << 16), 256, 0, s>>>(g.edge, g.node, g.m, g.erec);
    HSAW_CK(cudaGetLastError());
    if (cudaMalloc((void**)&g.grec, (size_t)g.m * 2 * sizeof(uint4)) != cudaSuccess) {
      cudaGetLastError();
      g.grec = nullptr;
      t_refused = true;
      return fail(HSAW_E_NOMEM, "graph: guide records do not fit in device memory");
    }
  }
  count_launch();
  k_guide<<<grid_for((size_t)n * 32, 256, 1u << 20), 256, 0, s>>>(g.node, g.edge, n, g.erec, g.grec, g.guide);
  HSAW_CK(cudaGetLastError());
  if (g.m > HUB_DEGREE) {
    count_launch();
    k_hub_guide<<<8 * sm_count(), 256, 0, s>>>(g.node, g.edge, hubs, g.erec, g.grec, g.guide);
    HSAW_CK(cudaGetLastError());
  }
  return HSAW_OK;
}

static hsaw_status from_edges(int64_t n, int64_t m, const int32_t* src, const int32_t* dst, const uint32_t* w,
                              uint32_t flags, cudaStream_t s, Graph& g) {
  if (n < 1 || m < 0 || n >= (1ll << 31) || m >= (1ll << 31)) return fail(HSAW_E_INVALID, "graph: need 1 <= n < 2^31, 0 <= m < 2^31");
  if (m > 0 && (!src || !dst || !w)) return fail(HSAW_E_INVALID, "graph: NULL edge array");
  const bool dev = flags & HSAW_INPUT_DEVICE;
  Temps T(s);
  // pinned host input: the destinations are copied first and sorted on s while the
  // sources and weights are copied on a side stream (drained before T frees); pageable
  // input is copied first, all of it, on s (its copies do not overlap kernels)
  SideStream side;
  const bool overlap = !dev && m > 0 && host_pinned(src) && host_pinned(w);
  int32_t *d_src = nullptr, *d_dst = nullptr;
  uint32_t* d_w = nullptr;
  bool o1 = false, o2 = false, o3 = false;
  if (!overlap) {
    HSAW_TRY(stage(src, (size_t)m, dev, s, &d_src, &o1));
    if (o1) T.keep(d_src);
    HSAW_TRY(stage(w, (size_t)m, dev, s, &d_w, &o3));
    if (o3) T.keep(d_w);
  }
  HSAW_TRY(stage(dst, (size_t)m, dev, s, &d_dst, &o2));
  if (o2) T.keep(d_dst);
  uint32_t* d_err = nullptr;
  HSAW_TRY(T.get(&d_err, 2));
  HSAW_CK(cudaMemsetAsync(d_err, 0, 2 * sizeof(uint32_t), s));
  uint32_t *keys, *vals, *keys2, *vals2, *row_start;
  HSAW_TRY(T.get(&row_start, n + 1));
  if (!overlap && m > 0 && n > 1 && !lean()) {  // the whole list is here: tails and weights ride along
    HSAW_TRY(alloc_graph(g, n, m, true));
    uint2* pay = nullptr;
    uint32_t* sorted = nullptr;
    HSAW_TRY(T.get(&keys, m));
    HSAW_TRY(T.get(&vals, m));
    HSAW_TRY(T.get(&keys2, m));
    HSAW_TRY(T.get(&vals2, m));
    HSAW_TRY(T.get(&pay, m));
    HSAW_TRY(radix_sort_edges(d_src, d_dst, d_w, (size_t)m, (uint32_t)n, keys, keys2, vals, vals2, pay, g.edge,
                              g.input_index, &sorted, d_err, s));
    count_launch();
    k_row_from_sorted<<<grid_for(n + 1, 256, 8192), 256, 0, s>>>(sorted, m, n, row_start);
    HSAW_CK(cudaGetLastError());
    return finish_graph(g, row_start, d_err, T, s);
  }
  if (m) {
    count_launch();
    k_validate_nodes<<<grid_for(m, 256, 8192), 256, 0, s>>>(d_dst, m, n, d_err);
    if (!overlap) {
      count_launch();
      k_validate_nodes<<<grid_for(m, 256, 8192), 256, 0, s>>>(d_src, m, n, d_err);
    }
    HSAW_CK(cudaGetLastError());
    HSAW_TRY(check_err(d_err, s));
  }
  HSAW_TRY(T.get(&keys, m));
  HSAW_TRY(T.get(&vals, m));
  HSAW_TRY(T.get(&keys2, m));
  HSAW_TRY(T.get(&vals2, m));
  if (m) {
    count_launch();
    k_iota_dst<<<grid_for(m, 256, 8192), 256, 0, s>>>(d_dst, m, keys, vals);
    HSAW_CK(cudaGetLastError());
  }
  bool alt = false;
  HSAW_TRY(radix_sort_pairs(keys, vals, keys2, vals2, (size_t)m, bit_width((uint64_t)(n - 1)), s, &alt));
  uint32_t* sk = alt ? keys2 : keys;
  uint32_t* sv = alt ? vals2 : vals;
  count_launch();
  k_row_from_sorted<<<grid_for(n + 1, 256, 8192), 256, 0, s>>>(sk, m, n, row_start);
  HSAW_CK(cudaGetLastError());
  if (overlap) {  // the destinations' copy finished at the validation's synchronisation
    HSAW_TRY(side.create());
    HSAW_TRY(stage(src, (size_t)m, dev, side.s, &d_src, &o1));
    if (o1) T.keep(d_src);
    HSAW_TRY(stage(w, (size_t)m, dev, side.s, &d_w, &o3));
    if (o3) T.keep(d_w);
    HSAW_CK(cudaEventRecord(side.ev, side.s));
    HSAW_CK(cudaStreamWaitEvent(s, side.ev, 0));
    count_launch();
    k_validate_nodes<<<grid_for(m, 256, 8192), 256, 0, s>>>(d_src, m, n, d_err);
    HSAW_CK(cudaGetLastError());
    HSAW_TRY(check_err(d_err, s));
  }
  HSAW_TRY(alloc_graph(g, n, m, true));
  if (m) {
    count_launch();
    k_gather_edges<<<grid_for(m, 256, 8192), 256, 0, s>>>(sv, d_src, d_w, m, g.edge, g.input_index);
    HSAW_CK(cudaGetLastError());
  }
  return finish_graph(g, row_start, d_err, T, s);
}

static hsaw_status from_csr(int64_t n, int64_t m, const int64_t* rp, const int32_t* src, const uint32_t* w,
                            uint32_t flags, cudaStream_t s, Graph& g) {
  if (n < 1 || m < 0 || n >= (1ll << 31) || m >= (1ll << 31)) return fail(HSAW_E_INVALID, "graph: need 1 <= n < 2^31, 0 <= m < 2^31");
  if (!rp || (m > 0 && (!src || !w))) return fail(HSAW_E_INVALID, "graph: NULL CSR array");
  const bool dev = flags & HSAW_INPUT_DEVICE;
  Temps T(s);
  int64_t* d_rp;
  int32_t* d_src;
  uint32_t* d_w;
  bool o1, o2, o3;
  HSAW_TRY(stage(rp, (size_t)n + 1, dev, s, &d_rp, &o1));
  if (o1) T.keep(d_rp);
  HSAW_TRY(stage(src, (size_t)m, dev, s, &d_src, &o2));
  if (o2) T.keep(d_src);
  HSAW_TRY(stage(w, (size_t)m, dev, s, &d_w, &o3));
  if (o3) T.keep(d_w);
  uint32_t *d_err, *row_start;
  HSAW_TRY(T.get(&d_err, 2));
  HSAW_TRY(T.get(&row_start, n + 1));
  HSAW_CK(cudaMemsetAsync(d_err, 0, 2 * sizeof(uint32_t), s));
  count_launch();
  k_csr_rows<<<grid_for(n + 1, 256, 8192), 256, 0, s>>>(d_rp, n, m, row_start, d_err);
  HSAW_CK(cudaGetLastError());
  HSAW_TRY(check_err(d_err, s));
  HSAW_TRY(alloc_graph(g, n, m, false));
  if (m) {
    count_launch();
    k_copy_edges<<<grid_for(m, 256, 8192), 256, 0, s>>>(d_src, d_w, m, n, g.edge, d_err);
    HSAW_CK(cudaGetLastError());
    HSAW_TRY(check_err(d_err, s));
  }
  return finish_graph(g, row_start, d_err, T, s);
}

// node record -> host CSR export
static hsaw_status export_graph(const Graph& g, int64_t* rp, int32_t* src, int32_t* dst, uint32_t* thr, int64_t* ii,
                                cudaStream_t s) {
  std::vector<uint4> node((size_t)g.n);
  HSAW_CK(cudaMemcpyAsync(node.data(), g.node, (size_t)g.n * sizeof(uint4), cudaMemcpyDeviceToHost, s));
  std::vector<uint2> edge;
  if (src || thr) {
    edge.resize((size_t)g.m);
    if (g.m) HSAW_CK(cudaMemcpyAsync(edge.data(), g.edge, (size_t)g.m * sizeof(uint2), cudaMemcpyDeviceToHost, s));
  }
  if (ii && g.m) {
    if (g.input_index)
      HSAW_CK(cudaMemcpyAsync(ii, g.input_index, (size_t)g.m * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  }
  HSAW_CK(cudaStreamSynchronize(s));
  if (ii && !g.input_index)
    for (int64_t e = 0; e < g.m; ++e) ii[e] = e;
  if (rp) {
    for (int64_t v = 0; v < g.n; ++v) rp[v] = node[v].x;
    rp[g.n] = g.m;
  }
  if (dst)
    for (int64_t v = 0; v < g.n; ++v)
      for (uint32_t q = node[v].x; q < node[v].x + node[v].y; ++q) dst[q] = (int32_t)v;
  for (int64_t q = 0; q < g.m; ++q) {
    if (src) src[q] = (int32_t)edge[q].x;
    if (thr) thr[q] = edge[q].y;
  }
  return HSAW_OK;
}

}  // namespace hsaw

using namespace hsaw;

extern "C" {

const char* hsaw_last_error(void) { return hsaw::last_error(); }
const char* hsaw_version(void) { return "hsaw-gb300 0.1 (sm_103a)"; }

hsaw_status hsaw_graph_from_edges(int64_t n, int64_t m, const int32_t* src, const int32_t* dst, const uint32_t* w_fixed,
                                  uint32_t flags, void* stream, hsaw_graph* out) {
  if (!out) return fail(HSAW_E_INVALID, "graph: NULL out");
  *out = nullptr;
  auto* h = new (std::nothrow) hsaw_graph_s();
  if (!h) return fail(HSAW_E_NOMEM, "graph: host allocation");
  const hsaw_status st = within_memory([&] {
    const hsaw_status r = from_edges(n, m, src, dst, w_fixed, flags, (cudaStream_t)stream, h->g);
    if (r != HSAW_OK) {
      cudaStreamSynchronize((cudaStream_t)stream);
      destroy_graph(h->g);
    }
    return r;
  });
  if (st != HSAW_OK) {
    delete h;
    return st;
  }
  *out = h;
  return HSAW_OK;
}

hsaw_status hsaw_graph_from_csr(int64_t n, int64_t m, const int64_t* in_row_ptr, const int32_t* in_src,
                                const uint32_t* w_fixed, uint32_t flags, void* stream, hsaw_graph* out) {
  if (!out) return fail(HSAW_E_INVALID, "graph: NULL out");
  *out = nullptr;
  auto* h = new (std::nothrow) hsaw_graph_s();
  if (!h) return fail(HSAW_E_NOMEM, "graph: host allocation");
  hsaw_status st = from_csr(n, m, in_row_ptr, in_src, w_fixed, flags, (cudaStream_t)stream, h->g);
  if (st != HSAW_OK) {
    cudaStreamSynchronize((cudaStream_t)stream);
    destroy_graph(h->g);
    delete h;
    return st;
  }
  *out = h;
  return HSAW_OK;
}

hsaw_status hsaw_graph_destroy(hsaw_graph g) {
  if (!g) return HSAW_OK;
  cudaDeviceSynchronize();
  destroy_graph(g->g);
  delete g;
  return HSAW_OK;
}

hsaw_status hsaw_set_allocator(hsaw_alloc_fn alloc, hsaw_free_fn release, void* ctx) {
  if ((alloc == nullptr) != (release == nullptr))
    return fail(HSAW_E_INVALID, "allocator: give both alloc and release, or neither");
  std::lock_guard<std::mutex> lk(g_alloc_set_mu);
  const long long held = g_held.load();
  if (held != 0) {
    char buf[160];
    snprintf(buf, sizeof(buf), "allocator: %lld scratch blocks of the current allocator are still held", held);
    t_err = buf;
    return HSAW_E_INVALID;
  }
  const ScratchAllocator* next = nullptr;
  if (alloc) {
    g_alloc_all.emplace_back(new ScratchAllocator{alloc, release, ctx});
    next = g_alloc_all.back().get();
  }
  g_alloc.store(next, std::memory_order_release);
  return HSAW_OK;
}

hsaw_status hsaw_debug_fail_alloc_after(int64_t n) {
  g_fail_countdown.store(n > 0 ? n : 0);
  return HSAW_OK;
}

hsaw_status hsaw_graph_edge(hsaw_graph g, int64_t edge_id, int32_t* src, int32_t* dst, int64_t* input_index) {
  if (!g) return fail(HSAW_E_INVALID, "graph: NULL handle");
  if (edge_id < 0 || edge_id >= g->g.m) return fail(HSAW_E_RANGE, "graph: edge id outside [0, m)");
  uint2 ed;
  HSAW_CK(cudaMemcpy(&ed, g->g.edge + edge_id, sizeof(uint2), cudaMemcpyDeviceToHost));
  if (src) *src = (int32_t)ed.x;
  if (dst) {  // the node whose in-range holds edge_id: binary search over the node records
    int64_t lo = 0, hi = g->g.n - 1;
    while (lo < hi) {
      const int64_t mid = (lo + hi + 1) / 2;
      uint4 nd;
      HSAW_CK(cudaMemcpy(&nd, g->g.node + mid, sizeof(uint4), cudaMemcpyDeviceToHost));
      if ((int64_t)nd.x <= edge_id) lo = mid; else hi = mid - 1;
    }
    // nodes without in-edges share their first position with the next node: take the
    // last node starting at or before edge_id whose range is non-empty
    uint4 nd;
    HSAW_CK(cudaMemcpy(&nd, g->g.node + lo, sizeof(uint4), cudaMemcpyDeviceToHost));
    while (lo > 0 && (int64_t)nd.x + nd.y <= edge_id) {
      --lo;
      HSAW_CK(cudaMemcpy(&nd, g->g.node + lo, sizeof(uint4), cudaMemcpyDeviceToHost));
    }
    *dst = (int32_t)lo;
  }
  if (input_index) {
    if (g->g.input_index) {
      HSAW_CK(cudaMemcpy(input_index, g->g.input_index + edge_id, sizeof(int64_t), cudaMemcpyDeviceToHost));
    } else {
      *input_index = edge_id;
    }
  }
  return HSAW_OK;
}

hsaw_status hsaw_graph_info(hsaw_graph g, int64_t* n, int64_t* m) {
  if (!g) return fail(HSAW_E_INVALID, "graph: NULL handle");
  if (n) *n = g->g.n;
  if (m) *m = g->g.m;
  return HSAW_OK;
}

hsaw_status hsaw_graph_export(hsaw_graph g, int64_t* in_row_ptr, int32_t* in_src, int32_t* in_dst, uint32_t* thr,
                              int64_t* input_index, void* stream) {
  if (!g) return fail(HSAW_E_INVALID, "graph: NULL handle");
  return export_graph(g->g, in_row_ptr, in_src, in_dst, thr, input_index, (cudaStream_t)stream);
}

}  // extern "C"
