// Internal state of a query: device suspect set, the ordered HSAW stream and the
// counting / greedy workspaces (not part of the ABI).
#pragma once
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace hsaw {

// Device view of the suspects V_I = (V_I, p) (Sec. 2.2) and of an optional residual graph.
struct QueryDev {
  uint32_t* s_bits = nullptr;     // n bits: v in V_I
  uint32_t* p32 = nullptr;        // n words or NULL (p == 1)
  int32_t* s_list = nullptr;      // n_src node ids of V_I
  int32_t n_src = 0;
  uint32_t* edge_removed = nullptr;  // m bits or NULL
  uint32_t* node_removed = nullptr;  // n bits or NULL
  uint64_t seed = 0;
  bool owns_removed = false;
  double start_rate = 0.0;  // chance that a start node is a real source
};

hsaw_status query_upload(const Graph& g, const hsaw_query* q, QueryDev& qd, cudaStream_t s);
void query_release(QueryDev& qd, cudaStream_t s);
// Bit x of *bits = (bytes[x] != 0), x < len; bytes is a device array.
hsaw_status pack_mask(const uint8_t* bytes, size_t len, uint32_t** bits, cudaStream_t s);

// The ordered HSAW stream R_1, R_2, ... of Alg. 3: hit j has attempt id aid[j], l_j =
// len[j] nodes nodes[node_off[j] .. node_off[j+1]) and l_j - 1 edges starting at
// edges[node_off[j] - j].
struct Stream {
  int64_t count = 0;
  int64_t total_nodes = 0;
  uint64_t first_attempt = 0;
  uint64_t next_attempt = 0;  // first attempt id not examined yet
  uint64_t steps = 0;         // live-edge draws executed
  uint64_t max_attempts = 0;
  DBuf<uint64_t> aid;
  DBuf<uint32_t> len;
  DBuf<int64_t> node_off;  // count + 1
  DBuf<int32_t> nodes;
  DBuf<int32_t> edges;
  // per-launch workspace
  DBuf<uint32_t> chunk_hits, chunk_off, ctrs;
  DBuf<uint2> recs;
  DBuf<uint4> chunk_kept;  // checkpoints of the records' walks, two per record
  DBuf<uint4> kept;        // and of the hits just found, in order
  uint32_t kept_hits = 0;  // hits that kept holds
  DBuf<uint64_t> tmp64;
  DBuf<uint32_t> pbits;  // walk pool: one bit per attempt of a window
  DBuf<uint64_t> pcnt;   // walk pool: entries per (source, block), then their prefix
  double hit_rate = 0.0;  // running estimate for launch sizing
  double least_window = 1048576.0;  // attempts per sampler launch; a caller's handle holds all hits of its windows
  bool ids_only = false;  // only attempt ids and lengths are wanted, no walks
  int64_t elem_range[2] = {0, 0};  // [node mode, edge mode]: element ids lie in [0, n) / [0, m)
  void release(cudaStream_t s);
};

// Hit records that a sampler launch has room for per chunk of attempts: a few standard deviations above
// the hits expected at `rate` a attempt, at most all.  A launch that needs more runs again with all.
inline uint32_t hit_records(double rate, uint32_t chunk) {
  const double hits = std::max(rate, 0.0) * chunk;
  return (uint32_t)std::min<double>(chunk, std::ceil(hits + 6.0 * std::sqrt(hits + 1.0) + 8.0));
}
// Checkpoints (32 bytes a record) are kept for launches of up to this many records: 134 MB, or half of what
// the counts and the index of the walks expected will take (48 bytes an element); without them the walks
// are drawn again from their starts.
inline uint64_t kept_records(double elements) { return std::max(1ull << 22, (unsigned long long)(0.75 * elements)); }
constexpr uint64_t MOST_ATTEMPTS = 1ull << 28;  // of a launch

hsaw_status stream_init(Stream& st, uint64_t first_attempt, uint64_t max_attempts, cudaStream_t s);
// Extend the stream until it holds at least want hits (Alg. 3 loop).
hsaw_status stream_extend(const Graph& g, const QueryDev& qd, Stream& st, int64_t want, cudaStream_t s);
// Adopt new_hits hits whose attempt ids and lengths are already at aid/len[st.count ..]:
// their walk offsets, nodes and edges (re-drawn from the attempt ids), and the count.
// new_nodes: their nodes, or -1 if not known.
hsaw_status stream_take_hits(const Graph& g, const QueryDev& qd, Stream& st, uint32_t new_hits, int64_t new_nodes,
                             cudaStream_t s);
hsaw_status classify_attempts(const Graph& g, const QueryDev& qd, uint64_t first, int64_t count, int8_t* outcome,
                              int32_t* length, cudaStream_t s);

// Walks and walk elements that a Cover may have.  Its kernels count them in 32 bits and step by up to 2^21
// at a time: a step past the end must not wrap, or a loop would never end.
constexpr int64_t MOST_ENTRIES = (1ll << 32) - (1ll << 22);

// Occurrence counts and inverted index over walks [first, first + count) (a5, a6).
struct Cover {
  int64_t walks = 0, entries = 0, unique = 0;
  DBuf<uint32_t> keys, vals, keys2, vals2;  // sort workspace
  DBuf<uint32_t> run_flag;                  // entries
  DBuf<int32_t> uid;                        // unique element ids, increasing
  DBuf<uint32_t> cnt;                       // occurrence count per unique element
  DBuf<uint32_t> inv_off;                   // unique + 1
  DBuf<uint32_t> inv_walk;                  // entries: local walk index, grouped by element
  DBuf<uint32_t> entry_uidx;                // entries: unique index of each walk entry
  DBuf<uint32_t> walk_eoff;                 // walks + 1: entry offsets of the walks
  DBuf<uint32_t> cnt_work;                  // greedy's running counts
  DBuf<uint32_t> covered;  // greedy: per walk, 0 or 1 + the pick that covered it
  DBuf<uint8_t> dirty;     // greedy (grid version): group dirty flags
  DBuf<uint4> inv_ent;           // cluster greedy: inverted-index entries with their walk's entry range; peaks: pairs
  DBuf<uint4> peak_list;         // greedy by peaks: the phase's elements
  DBuf<uint32_t> g_idx, g_list, g_cnt, g_entry;  // greedy on the heavy elements: index map, list, counts, entries
  DBuf<uint2> g_rng;             // greedy: each element's entries of inv_ent
  DBuf<unsigned long long> partial;
  // counts by element id (for_greedy): keys holds the counts of `elements` ids, the entries of
  // the walks are el[*from - from_sub ...], and entries, unique, uid and the inverted index are
  // not made
  bool by_id = false;
  bool short_walks = false;  // mean walk below 16 elements, about
  const int32_t* el = nullptr;
  const int64_t* from = nullptr;
  int64_t from_sub = 0, elements = 0;
  const struct Stream* stream = nullptr;  // where the walks lie, for an index made after all
  hsaw_mode mode = HSAW_EDGE;
  int64_t first = 0;
  int64_t about = 0;      // walk elements of the range (counts by id: about)
  bool crowded = false;   // by peaks would be the slower greedy (cover_build)
  void release_index(cudaStream_t s);  // uid, cnt and the inverted index, which counts by id do not make
  void release(cudaStream_t s);
};

// Whether the greedy's counts are by element id (M elements in all, `elements` in the walks).
bool counts_by_id(int64_t M, int64_t elements);
// k > 0: only cover_greedy of k picks follows (any element a candidate if all), so counts by element
// id do where they are the cheaper.
hsaw_status cover_build(const Stream& st, hsaw_mode mode, int64_t first, int64_t count, Cover& cv, cudaStream_t s,
                        int32_t k = 0, bool all = true);
// Entry offsets of walks [first, first + count) from the range's first, in cv.walk_eoff.
hsaw_status walk_offsets(const Stream& st, bool edges, int64_t first, int64_t count, Cover& cv, cudaStream_t s);
hsaw_status count_by_id(const Stream& st, bool edges, int64_t first, int64_t count, int64_t M, Cover& cv,
                        cudaStream_t s);
int peak_cluster();  // CTAs of the cluster that the greedy by peaks runs on; 0: it cannot
uint64_t peak_room(int64_t walks);  // pairs that its CTAs hold
// Greedy (Alg. 4 / 7) on a built Cover; cand (device, M bytes) may be NULL.  *aid_host (may be
// NULL) receives *aid_dev with the picks.
hsaw_status cover_greedy(Cover& cv, const uint8_t* cand_dev, int64_t M, int32_t k, int64_t* ids_host,
                         uint32_t* gains_host, cudaStream_t s, const uint64_t* aid_dev = nullptr,
                         uint64_t* aid_host = nullptr);
// The same picks by peaks, many at a time (peaks.cu), for cover_greedy: the first *rounds <= k
// ids and gains (device, k of each); *done = false when no cluster can run it, or it is left to the
// greedy that takes one pick at a time.
// The greedy by peaks keeps a phase whose elements do not fit its CTAs whole while their (element, walk)
// pairs are at most this many, and its rounds have not looked at 16 times as many and PEAK_PICK a pick;
// otherwise the greedy that takes one pick at a time has it.  Greedy by peaks against one pick at a
// time, ms, where the lists are longer: 4 M node walks of R-MAT 18 (115 M elements), k = 100, 700
// against 65; 1 M of R-MAT 13 (8.2 M), k = 1,000, 102 against 9.9; 1 M on a path of 30, k = 1, 0.85
// against 0.26; though also 200 K edge walks of the 16 K Chung-Lu graph, k = 100, 1.3 against 4.5
// (16 picks cover all: the list does not tell).  Within it: 4 M edge walks of R-MAT 18 (111 M
// elements, 310 K pairs), k = 1,000, 3.9 against 15.7; 1 M of R-MAT 13 with random weights (1.6 M,
// 443 K pairs), k = 1,000, 3.6 against 5.1; 100 K node walks of R-MAT 13 (224 K pairs), k = 10, 0.75
// against 0.64.  Where the mean candidate is in fewer than 32 walks, few picks touch each other and
// lists may be longer: 1 M node walks of a 1 M Chung-Lu graph with random weights (16 walks a candidate,
// 1.1 M pairs), k = 100, 1.7 against 2.6.
constexpr uint64_t PEAK_PICK = 1ull << 15;
inline uint64_t peak_pairs(int64_t walks, int64_t elements, int32_t k) {
  return peak_room(walks) / 8 * 7 + (uint64_t)elements / 20 + 200ull * k;
}
constexpr uint32_t PEAK_SPARSE = 32;  // elements / candidates below which a list may be longer,
inline uint32_t peak_sparse_pairs(int32_t k) {  // by this many pairs: fewer where many picks mean many rounds
  return (uint32_t)std::min<uint64_t>(10000ull * k, 1000000000ull / (1000 + (uint64_t)k));
}
// Elements that a phase lists, about: half as many again as the picks wanted, and a few.
__host__ __device__ inline uint64_t peak_list_goal(uint64_t k) { return k + k / 2 + 64; }
struct PickBlock {  // one device buffer, so that one copy brings a greedy's results back
  static constexpr int CTL = 16, WORK = 4096;
  int64_t* ids;       // k
  uint32_t* gains;    // k
  uint64_t* last_aid; // an attempt id for the caller
  uint32_t* ctl;      // CTL words
  uint32_t* work;     // WORK words, not copied
  static size_t copied_words(int32_t k) { return ((size_t)3 * k + 1) / 2 * 2 + 2 + CTL; }
  static PickBlock at(uint32_t* p, int32_t k) {
    uint32_t* e = p + ((size_t)3 * k + 1) / 2 * 2;
    return {reinterpret_cast<int64_t*>(p), p + 2 * (size_t)k, reinterpret_cast<uint64_t*>(e), e + 2, e + 2 + CTL};
  }
};
// host: room for PickBlock::copied_words(k) words; *copied: the picks are there already.
hsaw_status peak_greedy(Cover& cv, const uint8_t* cand, int32_t k, const PickBlock& out, uint32_t* host,
                        int32_t* rounds, bool* done, bool* copied, cudaStream_t s);
// #walks in [first, first + count) that contain an element of T (T host, k ids).  aids (may be
// NULL) receives the attempt ids of walks at[0] and at[1] with it.
hsaw_status cover_count(const Stream& st, hsaw_mode mode, int64_t first, int64_t count, const int64_t* T, int32_t k,
                        uint64_t* cov, cudaStream_t s, const int64_t* at = nullptr, uint64_t* aids = nullptr);

// Walk pool (pool.cu).
void pool_release(WalkPool& p);
hsaw_status pool_build(Graph& g, uint64_t seed, uint64_t attempts, cudaStream_t s);
// Append to st (aid, len at st.count) the hits among attempts [a0, a1) (a1 <= pool.attempts),
// in attempt order; *new_hits receives their number, *new_nodes their nodes.
hsaw_status pool_hits(const Graph& g, const QueryDev& qd, Stream& st, uint64_t a0, uint64_t a1, uint32_t* new_hits,
                      int64_t* new_nodes, cudaStream_t s);

// Cancellation of the calling thread's current solve (set by the server's workers):
// checked between sampler launches and between stopping-rule rounds.
void set_cancel_flag(const volatile int* flag);
bool cancel_requested();

// One full solve on `s` (the body of hsaw_solve).
hsaw_status solve_one(const Graph& g, const hsaw_query* q, hsaw_result* r, cudaStream_t s);
// The fixed-N solve from a stream that already holds at least q->n_hsaw hits: counting,
// greedy (Alg. 4 / 7) and the result fields.
hsaw_status solve_fixed_from_stream(const Graph& g, const hsaw_query* q, Stream& st, hsaw_result* r, cudaStream_t s);
// Batched fixed-N sampling (batch.cu): extends every stream i to want[i] hits with
// multi-instance sampler launches.
// status[i] (in: HSAW_OK to take part) becomes HSAW_E_TIMEOUT when instance i's attempt
// budget runs out first; the return value reports failures of the launches themselves.
// staged[i] receives the number of hits appended to stream i's aid/len after its count:
// stream_take_hits(..., staged[i]) draws their walks.
hsaw_status batch_sample(const Graph* const* gs, const QueryDev* const* qds, Stream* const* sts, const int64_t* want,
                         int32_t count, hsaw_status* status, int64_t* staged, cudaStream_t s);
// Query checks shared by every solve: mode, 1 <= k <= |C|.
hsaw_status validate_query(const Graph& g, const hsaw_query* q);

// Stopping-rule constants (Sec. 5.1) and Check (Alg. 5), host FP64.
void stop_constants(int64_t M, int32_t k, double eps, double delta, double out6[6]);
int check_bound(double c, double cp, double size_rp, int32_t t, double eps, double lambda1, double* eps_t);

}  // namespace hsaw

struct hsaw_walks_s {
  hsaw::Stream st;
  hsaw::QueryDev qd;
  int device = 0;
};
