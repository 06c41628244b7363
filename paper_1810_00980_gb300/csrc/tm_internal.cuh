// Internal declarations of libtmotif (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include <atomic>
#include <string>
#include <vector>

#include "../../include/tm.h"

namespace tmo {

constexpr int kWarp = 32;
constexpr unsigned kFull = 0xffffffffu;

// ----------------------------------------------------------------------------
// bounds-checked build
// ----------------------------------------------------------------------------
// Compiled with -DTM_CHECKED (libtmotif_checked.so), the indices the kernels derive from data
// (work items, first edges, candidates, windows, pair segments, sort positions) are checked
// against the sizes of the arrays they index.  A failed check sets its bit in the
// translation unit's device error word and the access goes to element 0 instead, so the
// kernel never touches memory outside its arrays and runs to the end; the host reads and
// clears the words with tm_check_status.  Without TM_CHECKED the checks compile to nothing.
enum CheckBit : unsigned {
    kChkQueue = 1u,     // work item / first edge beyond the batch's counts
    kChkWindow = 2u,    // window slot or query index beyond the batch's tables
    kChkView = 4u,      // position beyond an adjacency view (m entries)
    kChkNode = 8u,      // node id beyond n (offsets arrays hold n + 1 entries)
    kChkRange = 16u,    // a candidate or pair range not inside [0, m]
    kChkSort = 32u,     // a sort or scan output position beyond its array
    kChkSelf = 64u,     // the self-test's deliberate out-of-range index
};
#ifdef TM_CHECKED
static __device__ unsigned int g_tm_check_word;   // one per translation unit
__device__ __forceinline__ int64_t chk_idx(int64_t i, int64_t n, unsigned bit) {
    if ((unsigned long long)i >= (unsigned long long)n) {
        atomicOr(&g_tm_check_word, bit);
        return 0;
    }
    return i;
}
#define TM_CHK_IDX(i, n, bit) ::tmo::chk_idx((int64_t)(i), (int64_t)(n), (bit))
#define TM_CHK(cond, bit) \
    do { if (!(cond)) atomicOr(&::tmo::g_tm_check_word, (bit)); } while (0)
// the translation unit's error word, read (and cleared) from the host
#define TM_DEFINE_CHECK_WORD(fn)                                                             \
    int fn(unsigned* w, bool clear) {                                                        \
        if (cudaMemcpyFromSymbol(w, ::tmo::g_tm_check_word, sizeof(unsigned)) != cudaSuccess) \
            return TM_ECUDA;                                                                 \
        unsigned z = 0;                                                                      \
        if (clear && cudaMemcpyToSymbol(::tmo::g_tm_check_word, &z, sizeof(unsigned)) != cudaSuccess) \
            return TM_ECUDA;                                                                 \
        return TM_OK;                                                                        \
    }
#else
#define TM_CHK_IDX(i, n, bit) (i)
#define TM_CHK(cond, bit) do {} while (0)
#define TM_DEFINE_CHECK_WORD(fn) \
    int fn(unsigned* w, bool) { *w = 0; return TM_OK; }
#endif
int check_word_match(unsigned* w, bool clear);
int check_word_graph(unsigned* w, bool clear);
int check_word_prims(unsigned* w, bool clear);
int check_selftest();
#ifdef TM_CHECKED
// tm_check_expire: the nth launch from now of a kernel that waits between tiles runs without its first
// tile (nobody gets that ticket) and with few polls
int check_expire(int nth);   // returns what was left of the last one (0: it has happened)
#endif

// ----------------------------------------------------------------------------
// error plumbing
// ----------------------------------------------------------------------------
void set_error(const std::string& msg);
int cuda_status(cudaError_t e, const char* what, const char* file, int line);

#define TM_CUDA(call)                                                             \
    do {                                                                          \
        cudaError_t _e = (call);                                                  \
        if (_e != cudaSuccess) return ::tmo::cuda_status(_e, #call, __FILE__, __LINE__); \
    } while (0)

#define TM_TRY(call)                   \
    do {                               \
        int _s = (call);               \
        if (_s != TM_OK) return _s;    \
    } while (0)

// ----------------------------------------------------------------------------
// device graph: edges sorted by time plus three time-sorted adjacency views
// ----------------------------------------------------------------------------
// Type-erased device graph: the time arrays hold int32 when every normalised
// time fits (tbytes = 4), else int64 (tbytes = 8).
struct GraphDev {
    int64_t m;
    int32_t n;
    int32_t tbytes;         // 4 or 8: element size of t, out_t, in_t, pair_t
    int64_t P;              // distinct (src, dst) pairs
    const int32_t* src;     // [m]
    const int32_t* dst;     // [m]
    const void* t;          // [m] normalised, non-decreasing
    const int64_t* out_off; // [n+1]
    const int32_t* out_nbr; // [m] destination
    const void* out_t;      // [m]
    const int64_t* in_off;  // [n+1]
    const int32_t* in_nbr;  // [m] source
    const void* in_t;       // [m]
    const int32_t* pair_dst;// [m] destination of each pair-view entry
    const int32_t* pair_beg;// [m] start and end of the segment of the entry's pair
    const int32_t* pair_end;// [m]
    const void* pair_t;     // [m]
    const int32_t* out_src; // [m] source of each out-view entry (the sort key)
    const int32_t* in_dst;  // [m] destination of each in-view entry
    // pair table: hparts parts of hmask + 1 slots, open addressing inside a part; a slot is the key
    // (src << 32 | dst), then (length << 32 | begin) of the pair's segment
    const unsigned long long* hslots;
    uint32_t hparts, hmask;
    // pair filter: two bits per pair in one 32-bit word; a lookup whose two bits are not both
    // set has no pair (most lookups of absent pairs end in this L2-resident array)
    const uint32_t* pfilt;             // [pfmask+1] or null
    unsigned long long pfmask;         // words - 1 (power of two)
    int32_t loops;          // 1 if some edge has src == dst
    float per_tick;         // 1 / (largest normalised time + 1)
};

// The same graph with its time arrays typed (TT = int32_t or int64_t).
template <typename TT>
struct GraphDevT {
    int64_t m;
    int32_t n;
    int64_t P;
    const int32_t* src;
    const int32_t* dst;
    const TT* t;
    const int64_t* out_off;
    const int32_t* out_nbr;
    const TT* out_t;
    const int64_t* in_off;
    const int32_t* in_nbr;
    const TT* in_t;
    const int32_t* pair_dst;
    const int32_t* pair_beg;
    const int32_t* pair_end;
    const TT* pair_t;
    const int32_t* out_src;
    const int32_t* in_dst;
    const unsigned long long* hslots;
    uint32_t hparts, hmask;
    const uint32_t* pfilt;
    unsigned long long pfmask;
    int32_t loops;
    float per_tick;
    // two-node tables (set by the batch that needs them): over pair-view positions e,
    // exclusive prefix sums of the number of edges of e's own pair (ex_own) and of its
    // reverse pair (ex_rev) with time < t_e
    const int64_t* ex_own;  // [m+1] or null
    const int64_t* ex_rev;  // [m+1] or null
};

template <typename TT>
inline GraphDevT<TT> typed(const GraphDev& g) {
    GraphDevT<TT> r;
    r.m = g.m; r.n = g.n; r.P = g.P;
    r.src = g.src; r.dst = g.dst; r.t = (const TT*)g.t;
    r.out_off = g.out_off; r.out_nbr = g.out_nbr; r.out_t = (const TT*)g.out_t;
    r.in_off = g.in_off; r.in_nbr = g.in_nbr; r.in_t = (const TT*)g.in_t;
    r.pair_dst = g.pair_dst; r.pair_beg = g.pair_beg; r.pair_end = g.pair_end; r.pair_t = (const TT*)g.pair_t;
    r.out_src = g.out_src; r.in_dst = g.in_dst;
    r.hslots = g.hslots; r.hparts = g.hparts; r.hmask = g.hmask; r.loops = g.loops;
    r.pfilt = g.pfilt; r.pfmask = g.pfmask; r.per_tick = g.per_tick;
    r.ex_own = nullptr; r.ex_rev = nullptr;
    return r;
}

constexpr unsigned long long kHashEmpty = ~0ull;

}  // namespace tmo

struct tm_graph {
    int device;
    int64_t m;
    int32_t n;
    int64_t P;
    int64_t t_min;
    int64_t t_max;          // normalised
    int64_t bytes;
    void* block;            // one device allocation holding every array
    void* hash_block;       // the pair filter, after a small graph's pair table
    void* table_block;      // a large graph's pair table (or null)
    void* ex_own_block;     // the two-node tables ([m+1] each), built on first use (or null)
    void* ex_rev_block;
    // records that a round of a batch on this graph has needed room for, beyond the set capacity
    mutable std::atomic<int64_t> ride_need{0};
    tmo::GraphDev dev;
};

namespace tmo {

// ----------------------------------------------------------------------------
// motif plans
// ----------------------------------------------------------------------------
enum View : int8_t { kPair = 0, kOut = 1, kIn = 2, kAll = 3 };

struct LevelPlan {
    int8_t view;    // which adjacency view lists the candidates of this motif edge
    int8_t su, sv;  // motif node labels of u_i, v_i
    int8_t bind_u;  // u_i is first seen at this edge
    int8_t bind_v;  // v_i is first seen at this edge
    int8_t nb;      // labels 0..nb-1 are bound before this edge
    int8_t pad[2];
};

}  // namespace tmo

struct tm_motif {
    int32_t l, k;
    int32_t mu[TM_L_MAX];
    int32_t mv[TM_L_MAX];
    tmo::LevelPlan lv[TM_L_MAX];
};

namespace tmo {

// order in which a query enumerates first edges: by time (windows), or grouped
// by source / destination (positions of the out / in view) for exact queries
enum FirstOrder : int32_t { kOrdTime = 0, kOrdOut = 1, kOrdIn = 2, kOrdPair = 3 };

// QPlan::ex23 bits: a motif on two nodes with three edges, (u,v) first; the middle and
// the last edge each either repeat (u,v) or reverse it (v,u)
enum Ex23Bits : int32_t { kEx23On = 1, kEx23MidRev = 2, kEx23LastRev = 4 };

// one shift of an estimate riding along with an exact query
struct alignas(16) RideEnt {
    int64_t shift;        // window origin -(shift draw mod cd) - t_off
    int64_t wbase;        // the shift's first window slot
    int64_t cd, delta;
    const uint64_t* wtab; // as QPlan::wtab
    // (t1 - shift) / cd as (t1 - shift) * mul >> sh for every time of the graph, by the rounded-up
    // reciprocal of Granlund and Montgomery (1994); sh = 0: divide
    uint32_t mul, sh;
    int32_t all_kept;     // uniform p = 1: no keep flag to read
    int32_t pad0[3];
};

struct QPlan {
    int32_t l, k;
    int32_t mode;        // TM_MODE_*
    int32_t b;
    int32_t q_mode;
    int32_t order;       // FirstOrder
    int32_t hoist;       // 1: the last motif edge joins the first edge's two nodes
    int32_t rev;         // 1: three edges, the second binds one new node x and the last
                         //    joins x to a first-edge node: instances can be closed from
                         //    either the second or the last edge's candidates
    int32_t rev2;        // 1: four or more edges, and the same holds for the last two
    int32_t full;        // 1: windows enumerate node-grouped positions through perm
    int32_t hrev;        // 1: three edges, closing pair fixed by the first edge, and the second
                         //    edge either joins the first edge's nodes or adds one node: the
                         //    closing pair's entries can be the items instead
    int32_t ex23;        // kEx23*: two-node three-edge motif counted from the pair tables
    const int32_t* perm; // [b*m] per shift: view positions stably partitioned by window
    const int64_t* woff; // [b*(J+1)] per shift: start of each window's positions in perm
    int64_t delta;
    int64_t cd;          // c * delta (estimate), 0 for exact
    int64_t J;           // windows per shift (estimate), 1 for exact
    int64_t win_base;    // first window slot of this query
    double p;
    uint64_t seed;
    const uint64_t* wtab;// [2*(delta+1)] Q64 weights c delta / (c delta - Delta), or null
    // a segment of a streamed graph (defaults: the whole graph)
    int64_t t_off;       // window time origin minus the graph's time origin
    int64_t j_lo;        // windows j_lo+1 .. j_lo+J of every shift are processed
    int64_t own_lo;      // exact queries: first edges with time in [own_lo, own_hi)
    int64_t own_hi;
    int64_t m_total;     // |T| in q_j = r |T_j| / |T|
    int64_t sum_base;    // first per-shift sums slot of this query
    int64_t part_base;   // first partial record of the fold (shifts x slices) of this query
    // exact three-edge queries of the same motif at smaller spans, counted in the same
    // enumeration (spans dsub[0..nsub) < delta; their counts go to the A_X* accumulators)
    int32_t nsub;
    // estimate with every window kept (uniform p = 1): first edges of the whole graph in node
    // order, each clamped to its own window ((t1 - s) / cd), one accumulator slot per shift
    int32_t wclamp;
    int64_t dsub[3];
    int64_t J_all;       // wclamp: the windows per shift (J is then 1 slot)
    // estimates of the same motif riding along with this exact query: every instance this
    // query enumerates is also added, with the rider's weight, to the rider's window when it
    // lies inside a kept window of the rider and within the rider's span
    int32_t nride;       // entries of `rides`: one per shift of every rider
    int32_t riding;      // 1: this estimate rides along with an exact query (no first edges)
    const RideEnt* rides;
    // (a stride of 320 bytes: plans staged in shared memory at 328 made the replay of a batch 1.5 %
    // slower)
    int64_t pad0[3];
    LevelPlan lv[TM_L_MAX];
};
constexpr int kMaxSub = 3;
constexpr int kMaxRide = 4096;                           // riders of one exact query
constexpr int64_t kMaxRideShifts = (int64_t)1 << 22;     // and their shifts (64 bytes each)
static_assert(sizeof(QPlan) == 320, "plan stride");

struct Tuning {
    int block_threads = 256;
    int blocks_per_sm = 6;   // (launch_match gives the times)
    int chunk_items = 256;
    int enum_threshold = 48;
};
Tuning& tuning();
constexpr int64_t kRideCapacity = (int64_t)1 << 23, kRideCapacityMost = (int64_t)1 << 27;
std::atomic<int64_t>& ride_capacity();

// one query's part of a segment of a streamed graph
struct SegSpec {
    int64_t t_off;           // global time of the segment graph's time 0
    int64_t j_lo, J;         // estimate: windows j_lo+1 .. j_lo+J of every shift
    int64_t own_lo, own_hi;  // exact: first edges with (segment) time in [own_lo, own_hi)
    int64_t m_total;         // edges of the whole graph
};

// one shift's sums over the windows a batch processed (additive across segments)
struct ShiftSums {
    unsigned long long count, wlo, whi, first, cand, last, inst, kept;
    double zq, vq;
};
// a += b (the weight sum as one 128-bit integer)
__host__ __device__ inline void add_shift_sums(ShiftSums& a, const ShiftSums& b) {
    unsigned long long lo = a.wlo + b.wlo;
    a.whi += b.whi + (lo < a.wlo ? 1ull : 0ull);
    a.wlo = lo;
    a.count += b.count; a.first += b.first; a.cand += b.cand; a.last += b.last;
    a.inst += b.inst; a.kept += b.kept; a.zq += b.zq; a.vq += b.vq;
}

struct BatchOut {                 // optional per-window readback for one query
    int query = -1;
    int32_t k = 0;
    bool all_windows = false;
    tm_window_rec* recs = nullptr;
    int64_t cap = 0;
    int64_t n_out = 0;
    int64_t shift = 0;
    const SegSpec* seg = nullptr; // per query, or null (whole graph)
    ShiftSums* sums = nullptr;    // host: per query, per shift (exact: one), or null
    const std::vector<std::vector<int>>* riders = nullptr;   // per query: plan indices of its riders
    int hidden = 0;                           // trailing queries whose results nobody asked for
    int64_t hidden_records = 0;               // most deferred records made room for on their behalf
    int64_t need_records = 0;                 // deferred records to make room for, past the usual capacity
    const int32_t* nsub = nullptr;            // per query: spans counted alongside (exact)
    const int64_t* sub_delta = nullptr;       // [nq][kMaxSub]
    unsigned long long* sub_count = nullptr;  // host out: [nq][kMaxSub]
};

// Most deferred records made room for on behalf of estimates that could do without (12.9 GB)
constexpr int64_t kHiddenRecords = (int64_t)1 << 29;
// hidden_records: of estimates that share an enumeration nobody asked for; 0: they do not
int run_batch(const tm_graph* g, const tm_query* qs, int nq, tm_result* res,
              cudaStream_t st, BatchOut* dbg, int64_t hidden_records = kHiddenRecords);
// bytes of the record buffer that a batch of these queries takes when it shares enumerations (0: it
// does not)
int64_t share_bytes(const tm_graph* g, const tm_query* qs, int nq);
int count_plain(const tm_graph* g, const tm_motif* m, int64_t delta, int64_t* count);
// query checks of tm_run_batch against a graph whose normalised times end at t_max
int check_query(int64_t t_max, const tm_query& q, std::string& why);

// primitives (prims.cu)
int scan_exclusive_i64(const int64_t* in, int64_t* out, int64_t n, int64_t* d_total,
                       cudaStream_t st);
int radix_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* keys_tmp, uint32_t* vals_tmp,
                     int64_t n, int bits, uint32_t* d_err, cudaStream_t st);   // *d_err as SortWs::err

// The radix sort in parts, for callers that produce the keys themselves and sort several lists
// of n triples (key, a, t) by the same number of bits:
//   sort_digits    how the bits are cut into passes
//   sort_ws        places the scratch of `sorts` sorts, `counted` of them with counts of their
//                  own, in sort_ws_bytes(...) bytes; sort_clear zeroes it
//   count_digits   (device) adds a key to the block's counts [pass][digit] in shared memory, which
//                  the caller adds to W.counts + (c * passes << db) for counted list c
//   sort_bases     counts -> starts of the digits' runs
//   sort_run       the passes of sorts [first, first + sorts) side by side in one launch per pass
//                  (SortIo::counts names the counted list with the same keys)
// Asynchronous; *W.err is non-zero afterwards if a wait between tiles expired (the lists are then
// incomplete: gave_up).
struct SortDigits { int bits, passes, db; };
struct SortWs {
    SortDigits D;
    int64_t n;
    int counted;
    uint32_t* err;
    uint32_t* counts;
    uint32_t* words;
    size_t bytes;
};
struct SortIo {
    const uint32_t *key_in, *a_in;
    const void* t_in;
    uint32_t *key_out, *a_out;    // the sorted lists
    void* t_out;
    uint32_t *key_tmp, *a_tmp;    // between passes (unused by a single pass)
    void* t_tmp;
    int counts;
    bool keep_key;                // false: the last pass leaves key_out unwritten
};
struct SortJob {
    const uint32_t *key_in, *a_in;
    const void* t_in;
    uint32_t *key_out, *a_out;
    void* t_out;
    uint32_t *ticket, *words;
    const uint32_t* base;
};
constexpr int kMaxSortJobs = 2;
struct SortJobs {
    SortJob job[kMaxSortJobs];
    int jobs;
    int limit;   // polls of a wait
    uint32_t* err;
};
SortDigits sort_digits(int bits);
size_t sort_ws_bytes(int64_t n, const SortDigits& D, int sorts, int counted);
SortWs sort_ws(void* mem, int64_t n, const SortDigits& D, int sorts, int counted);
int sort_clear(const SortWs& W, cudaStream_t st);
int sort_bases(const SortWs& W, cudaStream_t st);
int sort_run(const SortWs& W, const SortIo* io, int sorts, int first, int tbytes, cudaStream_t st);
__device__ __forceinline__ void count_digits(uint32_t* sm, const SortDigits& D, uint32_t key) {
    for (int p = 0; p < D.passes; p++)
        atomicAdd(sm + (p << D.db) + ((key >> (p * D.db)) & ((1u << D.db) - 1u)), 1u);
}
// exclusive scan with the tile sums in caller workspace (2 * ceil(n/2048) int64, n <= 2048^2)
int scan_exclusive_i64_ws(const int64_t* in, int64_t* out, int64_t n, int64_t* d_total,
                          int64_t* ws, int64_t ws_elems, cudaStream_t st);

int64_t scan_dn_ws_elems(int64_t n_max);
// Exclusive scan of 32-bit range lengths into 64-bit offsets (the first *d_n, or n_max when d_n is
// null) with, in cf, the element that holds every grain-th item (as far as ncf goes).  words:
// scan_once_words(n_max) zeroed words; when that is 0 (too many tiles for one launch) ws of
// scan_dn_ws_elems(n_max), or null to allocate it on the stream.  *err: as SortWs::err; in one
// launch *d_total, zeroed before, ends below zero then
// The matcher's chunks are whole grains.  Few first edges: 32 items, so that small batches cut
// small chunks, with entries for 64 items per first edge; many: 256, where every chunk is at
// least that long anyway, for as many items in an eighth of the memory.  (The bound counts: a
// captured batch of 18 queries on 1e5 edges has one of 2.1e6, and at 256 took 275 instead of
// 234 us.)
__host__ __device__ inline int item_grain_log(int64_t n_max) { return n_max <= (int64_t)1 << 22 ? 5 : 8; }
__host__ __device__ inline int item_grain(int64_t n_max) { return 1 << item_grain_log(n_max); }
inline size_t item_starts(size_t n_max) { return n_max <= (size_t)1 << 22 ? 2 * n_max + 2 : n_max / 4 + 2; }
constexpr int64_t kOnePassTiles = 1024;
size_t scan_once_words(int64_t n_max);
int scan_lengths(const int32_t* in, int64_t* out, int64_t n_max, const int64_t* d_n, int64_t* d_total,
                 int64_t* cf, int64_t ncf, unsigned long long* words, uint32_t* err, int64_t* ws, int64_t ws_elems,
                 cudaStream_t st);
// scan_exclusive_i64 in one launch when scan_once_words(n) > 0 (that many zeroed words)
int scan_once_i64(const int64_t* in, int64_t* out, int64_t n, int64_t* d_total, unsigned long long* words, uint32_t* err,
                  cudaStream_t st);

int sm_count();
// a graph from device arrays (tm_graph_load_device); h_t: the same times on the host when the
// caller has them there (their first and last are then read without waiting for the device)
int build_graph(const int32_t* d_src, const int32_t* d_dst, const int64_t* d_t, const int64_t* h_t, int64_t m,
                int32_t n_nodes, cudaStream_t st, tm_graph** out);
// the graph's two-node tables (own, rev: [m+1] each) that are asked for, each built on
// the first call that needs it (thread-safe; synchronises the stream when it builds);
// null for an empty graph or when not asked for
int ensure_ex_tables(tm_graph* g, cudaStream_t st, bool need_own, bool need_rev, const int64_t** own,
                     const int64_t** rev);
// device memory pool (prims.cu): raise the default pool's release threshold once
// per device; pool_free returns a stream-ordered block on an internal stream
int pool_prepare(int dev);
void pool_free(void* p, int dev);
int pool_trim();   // also frees the scratch arenas that no call holds
// scratch of one call, leased from a per-device grow-only arena (slot >= 0) or, when every
// arena is held, a pool block (slot < 0); usable on st from acquire to release
struct ScratchLease {
    void* p = nullptr;
    int slot = -1;
    int dev = 0;
};
int scratch_acquire(size_t bytes, cudaStream_t st, ScratchLease& L);
void scratch_release(ScratchLease& L, cudaStream_t st);

// profiling (abi.cu): phase events of the last batch / graph build, launch counter
bool profiling();
void store_profile_batch(double windows_ms, double level2_ms, double match_ms, double fold_ms,
                         double batch_ms, int64_t match_items, int64_t first_edges, double sizing_ms,
                         double scan_ms, double ride_ms = 0.0);
void store_profile_graph(double graph_ms);
void store_profile_ride_records(int64_t n);
void count_launch(int n = 1);

// NVTX ranges naming the host-side phases of a call (graph build, window partition, second-edge
// ranges, matcher, fold), one after another, so that a profiler can select them; without a tool
// attached each call costs a branch
struct NvtxPhases {
    nvtxRangeId_t id = 0;
    bool open = false;
    void next(const char* name) {
        if (open) nvtxRangeEnd(id);
        open = name != nullptr;
        if (open) id = nvtxRangeStartA(name);
    }
    ~NvtxPhases() { next(nullptr); }
};

// CUDA events on a stream, created only while profiling is on
struct PhaseEvents {
    static constexpr int kMax = 12;
    cudaEvent_t ev[kMax];
    int n = 0;
    bool on = false;
    explicit PhaseEvents(bool enable) : on(enable) {
        if (on)
            for (int i = 0; i < kMax; i++)
                if (cudaEventCreate(&ev[i]) != cudaSuccess) on = false;
    }
    ~PhaseEvents() {
        if (on)
            for (int i = 0; i < kMax; i++) cudaEventDestroy(ev[i]);
    }
    int mark(cudaStream_t st) {
        if (!on || n >= kMax) return -1;
        cudaEventRecord(ev[n], st);
        return n++;
    }
    double ms(int a, int b) const {
        if (!on || a < 0 || b < 0) return 0.0;
        float x = 0.f;
        cudaEventElapsedTime(&x, ev[a], ev[b]);
        return (double)x;
    }
};

// A launch that may begin before the stream's previous kernel has ended (programmatic dependent
// launch): its blocks set up what no kernel of the stream writes and then call grid_wait(), which
// returns once every earlier kernel has completed.  Every kernel launched this way calls it in
// every block, so that its own completion implies theirs.
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ----------------------------------------------------------------------------
// device helpers
// ----------------------------------------------------------------------------
// first index p in [lo, hi) with a[p] > v (a sorted non-decreasingly; any integer element type)
template <typename T>
__device__ __forceinline__ int64_t upper_bound_i64(const T* __restrict__ a, int64_t lo, int64_t hi,
                                                   int64_t v) {
    while (lo < hi) {
        int64_t mid = lo + ((hi - lo) >> 1);
        if ((int64_t)__ldg(a + mid) <= v) lo = mid + 1; else hi = mid;
    }
    return lo;
}
constexpr int64_t kTimeSearchMin = 32;
// first index p in [lo, hi) with a[p] >= v
template <typename T>
__device__ __forceinline__ int64_t lower_bound_i64(const T* __restrict__ a, int64_t lo, int64_t hi,
                                                   int64_t v) {
    while (lo < hi) {
        int64_t mid = lo + ((hi - lo) >> 1);
        if ((int64_t)__ldg(a + mid) < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ int64_t lower_bound_i32(const int32_t* __restrict__ a, int64_t lo,
                                                   int64_t hi, int32_t v) {
    while (lo < hi) {
        int64_t mid = lo + ((hi - lo) >> 1);
        if (__ldg(a + mid) < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Decoupled look-back.  A tile's word for one digit: 0 not yet known; count + 1 (below 2^31) once the tile
// has counted; kTilePrefix | sum over the tiles up to and including it once that is known (below
// 2^31, as n is).
constexpr uint32_t kTilePrefix = 0x80000000u;
constexpr int kSpinLimit = 1 << 22;   // polls of one word, about a second: then the error word is set

__device__ __forceinline__ uint32_t ld_tile(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_tile(uint32_t* p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Whether a wait of an earlier kernel of this call has expired.  What that kernel should have
// written is then missing, so every kernel behind a sort that takes an index, a range or a loop
// bound from there reads the word first and returns; the host reports it.  (A plain load: kernels
// that start with an empty L1, not overlapped launches.  Read past L1 by every warp, one word held
// up the small counts by 5 us and the build of 1e8 edges by 2 %.)  Behind a scan the total says so:
// it is negative, and there are no items (k_scan_once).
__device__ __forceinline__ bool gave_up(const uint32_t* err) { return err && *err != 0; }

// sum += the words of tiles tile-1, tile-2, ... at `stride` apart, back to the first that holds a
// prefix, kLookBack of them read at a time (the reads are a serial chain otherwise: prefixes
// travel forward at most that many tiles per memory latency).  Tiles are numbered in the order
// blocks start, so every word waited for belongs to a block that already runs; if one still
// never comes within `limit` polls the error word is set.  False then, and when another tile has
// set it: the caller writes nothing more.
constexpr int kLookBack = 4;
__device__ __forceinline__ bool look_back(const uint32_t* words, int64_t tile, int64_t stride, uint32_t* err, int limit,
                                          uint32_t& sum) {
    int64_t at = tile - 1;
    int spins = 0;
    while (at >= 0) {
        uint32_t v[kLookBack];
#pragma unroll
        for (int i = 0; i < kLookBack; i++) v[i] = at - i >= 0 ? ld_tile(words + (at - i) * stride) : kTilePrefix;
        bool open = true;   // no prefix and no missing word among those taken so far
#pragma unroll
        for (int i = 0; i < kLookBack; i++) {
            if (open) {
                if (v[i] & kTilePrefix) {
                    sum += v[i] & ~kTilePrefix;
                    return true;
                }
                open = v[i] != 0;
                if (open) {
                    sum += v[i] - 1;
                    at--;
                }
            }
        }
        if (v[0] == 0) {
            if (++spins > limit) {
                atomicOr(err, 1u);
                return false;
            }
            if ((spins & 63) == 0 && ld_tile(err) != 0) return false;
        } else {
            spins = 0;
        }
    }
    return true;
}

// upper_bound_i64 on a node's list of times (or the whole graph's): the first probe where v would be if
// the list's entries were spread evenly over the graph's time span, the second corrected by
// the same density from the time found there, then a bracket that grows from it and a bisection
// inside the bracket.  For evenly drawn times the second probe is off by about the fourth root of
// the list's length, so a search takes about 4 + log2(n) / 4 dependent loads instead of
// log2(n); bursts only widen the bracket (twice log2(n) at worst).  k_level2 of the benchmark batch
// on 1e7 edges 1.206 -> 1.124 ms, of a 1e8-edge hub graph 1.27 -> 1.17 ms, the matcher of 192 seeds of
// the 4-cycle 3.87 -> 3.60 ms; lists up to kTimeSearchMin entries are as quick by bisection.
template <typename T>
__device__ __forceinline__ int64_t time_ub(const T* __restrict__ a, int64_t lo, int64_t hi, int64_t v, float per_tick) {
    if (hi - lo > kTimeSearchMin) {
        const float d = (float)(hi - lo) * per_tick;
        int64_t g = lo + min((int64_t)((float)v * d), hi - lo - 1);
        g = min(max(g + (int64_t)((float)(v - (int64_t)__ldg(a + g)) * d), lo), hi - 1);
        int64_t step = (int64_t)1 << ((31 - __clz((int)(hi - lo))) >> 2);
        if ((int64_t)__ldg(a + g) <= v) {
            int64_t cur = g + step;
            lo = g + 1;
            while (cur < hi && (int64_t)__ldg(a + cur) <= v) {
                lo = cur + 1;
                step <<= 1;
                cur += step;
            }
            hi = min(hi, cur);
        } else {
            int64_t cur = g - step;
            hi = g;
            while (cur >= lo && (int64_t)__ldg(a + cur) > v) {
                hi = cur;
                step <<= 1;
                cur -= step;
            }
            lo = max(lo, cur + 1);
        }
    }
    return upper_bound_i64(a, lo, hi, v);
}

// SplitMix64 (Steele, Lea & Flood 2014): output n (n >= 1) of the generator
// seeded with s is mix(s + n * 0x9E3779B97F4A7C15).
__host__ __device__ __forceinline__ uint64_t sm64_mix(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__host__ __device__ __forceinline__ uint64_t sm64_output(uint64_t seed, uint64_t n) {
    return sm64_mix(seed + n * 0x9E3779B97F4A7C15ull);
}
// draw n of repetition k of a query seeded with `seed`
__host__ __device__ __forceinline__ uint64_t draw(uint64_t seed, uint64_t k, uint64_t n) {
    return sm64_output(sm64_output(seed, k + 1), n + 1);
}

// a pair's key, its bits in the filter (word (h >> 10) & pfmask), its part of the table (by the
// hash's upper half, in order) and its first slot there
__device__ __forceinline__ unsigned long long pair_key(int32_t u, int32_t v) {
    return ((unsigned long long)(uint32_t)u << 32) | (uint32_t)v;
}
__device__ __forceinline__ uint32_t pair_bits(unsigned long long h) { return (1u << (h & 31)) | (1u << ((h >> 5) & 31)); }
__device__ __forceinline__ uint32_t pair_part(unsigned long long h, uint32_t parts) { return __umulhi((uint32_t)(h >> 32), parts); }

// the time-sorted segment [a, b) of pair (u, v) in the pair view, by one hash lookup
// (after the pair filter, which answers most lookups of absent pairs from L2).  (Slots grouped by
// source, 8 bytes with the segment's end beside the entries, made the matcher 7 % slower: two
// more dependent loads; a table two thirds full 2 %: longer probe chains.)
template <typename TT>
__device__ __forceinline__ bool pair_segment(const GraphDevT<TT>& G, int32_t u, int32_t v, int64_t& a,
                                             int64_t& b, bool filter = true) {
    const unsigned long long key = pair_key(u, v);
    const unsigned long long h = sm64_mix(key);
    a = b = 0;
    if (filter && G.pfilt) {   // callers that know the pair exists skip the filter
        const uint32_t w = __ldg(G.pfilt + ((h >> 10) & G.pfmask));
        if (!((w >> (h & 31)) & (w >> ((h >> 5) & 31)) & 1u)) return false;
    }
    const ulonglong2* slots = reinterpret_cast<const ulonglong2*>(G.hslots) +
                              (size_t)pair_part(h, G.hparts) * ((size_t)G.hmask + 1);
    uint32_t x = (uint32_t)h & G.hmask;
    for (uint32_t it = 0; it <= G.hmask; it++) {
        const ulonglong2 sl = __ldg(slots + x);
        if (sl.x == key) {
            a = (int64_t)(uint32_t)sl.y;
            b = a + (int64_t)(sl.y >> 32);
            TM_CHK(b <= G.m, kChkRange);
#ifdef TM_CHECKED
            if (b > G.m) a = b = 0;   // an empty segment instead of one beyond the view
#endif
            return true;
        }
        if (sl.x == kHashEmpty) break;
        x = (x + 1) & G.hmask;
    }
    return false;
}

}  // namespace tmo
