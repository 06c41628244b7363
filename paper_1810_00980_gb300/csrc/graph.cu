// Graph ingest and adjacency build (temporal graph T and its static graph G,
// Section 2).  Everything after the input copy runs on the device: one read that
// validates, normalises t' = t - t_min (Algorithm 1 assumes times start at 0) and
// counts the sorts' digits, three stable radix sorts that leave every adjacency
// segment in time order, segment offsets and pair bounds found from the sorted
// keys, and the table of the static edges.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <new>

#include "tm_internal.cuh"

namespace tmo {
namespace {

constexpr int kThreads = 256;

unsigned grid_for(int64_t n, int per_sm = 8) {
    int64_t g = (n + kThreads - 1) / kThreads;
    int64_t cap = (int64_t)sm_count() * per_sm;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (unsigned)g;
}

// flags[0]: unsorted, flags[1]: id out of range (n_nodes given) or negative,
// flags[2]: max node id
__global__ void k_validate(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                           const int64_t* __restrict__ t, int64_t m, int32_t n_nodes,
                           int32_t* __restrict__ flags) {
    int32_t mx = -1;
    int bad_sort = 0, bad_id = 0, loop = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t s = src[i], d = dst[i];
        if (s < 0 || d < 0 || (n_nodes >= 0 && (s >= n_nodes || d >= n_nodes))) bad_id = 1;
        mx = max(mx, max(s, d));
        loop |= s == d;
        if (i > 0 && t[i] < t[i - 1]) bad_sort = 1;
    }
    if (__any_sync(kFull, bad_sort) && (threadIdx.x & 31) == 0) atomicOr(&flags[0], 1);
    if (__any_sync(kFull, bad_id) && (threadIdx.x & 31) == 0) atomicOr(&flags[1], 1);
    if (__any_sync(kFull, loop) && (threadIdx.x & 31) == 0) atomicOr(&flags[3], 1);
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(kFull, mx, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&flags[2], mx);
}

// Copies the edges into the graph (times minus tmin, in the graph's time type), counts the digits
// of both endpoints for the sorts and checks the input on the way: flags[0] unsorted, flags[1] id
// outside [0, n) (taken as node 0 until the build is given up), flags[3] some edge is a loop.
// One read of the input in place of three (check, copy, digit counts); bound by its 16 bytes in
// and 12 (16 with 64-bit times) out per edge.
constexpr int kIngestThreads = 512;
template <typename TT>
__global__ void __launch_bounds__(kIngestThreads) k_ingest(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                         const int64_t* __restrict__ t, int64_t m, int64_t tmin, int32_t n,
                         int32_t* __restrict__ gs, int32_t* __restrict__ gd, TT* __restrict__ gt,
                         uint32_t* __restrict__ flags, SortDigits D, uint32_t* __restrict__ counts) {
    extern __shared__ uint32_t sm_counts[];   // [source, destination][pass][digit]
    const int words = D.passes << D.db;
    for (int i = threadIdx.x; i < 2 * words; i += blockDim.x) sm_counts[i] = 0;
    __syncthreads();
    bool unsorted = false, bad = false, loop = false;
    constexpr int U = 4;   // independent loads in flight per thread
    const int64_t span = (int64_t)blockDim.x * U;
    for (int64_t base = blockIdx.x * span; base < m; base += gridDim.x * span) {
        int32_t s[U], d[U];
        int64_t tt[U], tp[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t i = base + (int64_t)u * blockDim.x + threadIdx.x;
            const bool in = i < m;
            s[u] = in ? src[i] : 0;
            d[u] = in ? dst[i] : 0;
            tt[u] = in ? t[i] : 0;
            tp[u] = in && i > 0 ? t[i - 1] : tt[u];
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t i = base + (int64_t)u * blockDim.x + threadIdx.x;
            if (i >= m) continue;
            unsorted |= tt[u] < tp[u];
            if ((uint32_t)s[u] >= (uint32_t)n || (uint32_t)d[u] >= (uint32_t)n) {
                bad = true;
                s[u] = d[u] = 0;
            }
            loop |= s[u] == d[u];
            gs[i] = s[u];
            gd[i] = d[u];
            gt[i] = (TT)(tt[u] - tmin);
            count_digits(sm_counts, D, (uint32_t)s[u]);
            count_digits(sm_counts + words, D, (uint32_t)d[u]);
        }
    }
    const bool any_unsorted = __syncthreads_or(unsorted), any_bad = __syncthreads_or(bad), any_loop = __syncthreads_or(loop);
    if (threadIdx.x == 0) {
        if (any_unsorted) atomicOr(flags, 1u);
        if (any_bad) atomicOr(flags + 1, 1u);
        if (any_loop) atomicOr(flags + 3, 1u);
    }
    for (int i = threadIdx.x; i < 2 * words; i += blockDim.x)
        if (sm_counts[i]) atomicAdd(counts + i, sm_counts[i]);
}

// off[v] = first position whose sorted key is >= v, for v in [0, n]; row 0 of the grid the out
// view's, row 1 the in view's.  Four keys per thread and load (one at a time, a thread waited out
// a memory latency per key: 38 us for 80 MB).
__global__ void k_offsets(const uint32_t* __restrict__ out_keys, const uint32_t* __restrict__ in_keys, int64_t m,
                          int32_t n, int64_t* __restrict__ out_off, int64_t* __restrict__ in_off, const uint32_t* err) {
    const uint32_t* keys = blockIdx.y ? in_keys : out_keys;
    int64_t* off = blockIdx.y ? in_off : out_off;
    const int64_t i0 = 4 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
    if (i0 > m || gave_up(err)) return;
    uint32_t k[4];
    if (i0 + 4 <= m) {
        const uint4 q = *reinterpret_cast<const uint4*>(keys + i0);   // the arrays start on 256 bytes
        k[0] = q.x; k[1] = q.y; k[2] = q.z; k[3] = q.w;
    } else {
#pragma unroll
        for (int x = 0; x < 4; x++) k[x] = i0 + x < m ? keys[i0 + x] : (uint32_t)n;   // position m ends the last node
    }
    int64_t prev = i0 == 0 ? -1 : (int64_t)keys[i0 - 1];
#pragma unroll
    for (int x = 0; x < 4; x++) {
        if (i0 + x > m) break;
        for (int64_t v = prev + 1; v <= (int64_t)k[x]; v++) off[TM_CHK_IDX(v, (int64_t)n + 1, kChkNode)] = i0 + x;
        prev = k[x];
    }
}

// ---- the pair table
// A small graph's table (one part, L2-resident) takes its pairs by compare-and-swap, one thread per
// pair.  Done that way for a large one, every pair waits for DRAM lines of its own, atomics and
// their retries on top: 0.36 ms for the 6.8M pairs of a 1e7-edge graph, 3.7 ms at 1e8, whether
// the pairs come in hash order or not (a probe: 0.30 ms in either order, 0.10 ms for the stores
// alone).  There the pairs are first sorted into lists by their part of the table, in two steps
// that write runs, and a block builds each part in shared memory and writes it out whole.
constexpr int kPartSlots = 4096;   // 64 KB of shared memory: three blocks per SM
constexpr int kPartPairs = 1900;   // on average: 46 % full, 50 standard deviations below a full part
constexpr int kBuckets = 64;       // first step's lists; the number of parts is a multiple
uint32_t pair_parts(int64_t pairs) {
    return kBuckets * (uint32_t)std::max<int64_t>(1, (pairs + kBuckets * kPartPairs - 1) / (kBuckets * kPartPairs));
}

__device__ __forceinline__ ulonglong2 pair_slot_value(int32_t u, int32_t v, int64_t beg, int64_t end) {
    return make_ulonglong2(pair_key(u, v), ((unsigned long long)(uint32_t)(end - beg) << 32) | (uint32_t)beg);
}

// one pair into the slots of its part by compare-and-swap (a part always keeps an empty slot)
__device__ __forceinline__ void pair_insert(unsigned long long* slots, uint32_t mask, const ulonglong2& e) {
    uint32_t x = (uint32_t)sm64_mix(e.x) & mask;
    for (uint32_t it = 0; it <= mask; it++) {
        if (atomicCAS(slots + 2 * (size_t)x, kHashEmpty, e.x) == kHashEmpty) {
            slots[2 * (size_t)x + 1] = e.y;
            return;
        }
        x = (x + 1) & mask;
    }
    TM_CHK(false, kChkRange);   // no empty slot
}

// every pair into a table of one part (emptied before)
__global__ void k_pair_insert(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, const int32_t* __restrict__ pair_beg,
                              const int32_t* __restrict__ pair_end, int64_t m, unsigned long long* __restrict__ slots,
                              uint32_t mask, const uint32_t* err) {
    if (gave_up(err)) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        if (pair_beg[i] == (int32_t)i) pair_insert(slots, mask, pair_slot_value(src[i], dst[i], i, pair_end[i]));
}

// First step's lists (filled by k_pairs): kBuckets lists of `cap` by the hash's upper bits
struct PairBuckets {
    ulonglong2* rec;       // [kBuckets][cap]
    uint32_t* count;       // [kBuckets]
    uint32_t cap;
    uint32_t* full;        // set when a list or a part had no room
};

// Second step: list b's pairs to their parts, each part's at the start of its own slots in the
// table.  A tile of 2,048 is put in part order in shared memory, so that runs are written.
constexpr int kSplitItems = 8;
constexpr int kSplitTile = kThreads * kSplitItems;
__global__ void __launch_bounds__(kThreads) k_pair_split(PairBuckets B, uint32_t parts, uint32_t* __restrict__ part_count,
                                                         ulonglong2* __restrict__ slots) {
    extern __shared__ __align__(16) unsigned char sm_split[];
    __shared__ uint32_t s_warp[kThreads / 32];
    ulonglong2* s_rec = (ulonglong2*)sm_split;                    // [tile] in part order
    uint32_t* s_cnt = (uint32_t*)(s_rec + kSplitTile);            // [sub] count, then tile start
    const uint32_t sub = parts / kBuckets;
    uint32_t* s_at = s_cnt + sub;                                 // [sub] place in the part's list
    const uint32_t per = (B.cap + kSplitTile - 1) / kSplitTile;   // tiles per list
    const uint32_t b = blockIdx.x / per, x0 = (blockIdx.x % per) * kSplitTile;
    const uint32_t n = min(B.count[b], B.cap);
    if (x0 >= n) return;
    const uint32_t tn = min(n - x0, (uint32_t)kSplitTile);
    for (uint32_t i = threadIdx.x; i < sub; i += kThreads) s_cnt[i] = 0;
    ulonglong2 rec[kSplitItems];
    uint32_t rank[kSplitItems], part[kSplitItems];
#pragma unroll
    for (int u = 0; u < kSplitItems; u++) {
        const uint32_t x = u * kThreads + threadIdx.x;
        if (x < tn) rec[u] = B.rec[(size_t)b * B.cap + x0 + x];
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kSplitItems; u++) {
        if (u * kThreads + threadIdx.x < tn) {
            part[u] = (uint32_t)TM_CHK_IDX(pair_part(sm64_mix(rec[u].x), parts) - b * sub, sub, kChkRange);
            rank[u] = atomicAdd(&s_cnt[part[u]], 1u);
        }
    }
    __syncthreads();
    // places in the parts' lists, and the tile's own order: an exclusive scan of the counts
    const uint32_t each = (sub + kThreads - 1) / kThreads, p0 = threadIdx.x * each;
    uint32_t sum = 0;
    for (uint32_t i = p0; i < min(p0 + each, sub); i++) sum += s_cnt[i];
    uint32_t inc = sum;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) s_warp[w] = inc;
    __syncthreads();
    uint32_t run = inc - sum;
    for (int i = 0; i < w; i++) run += s_warp[i];
    for (uint32_t i = p0; i < min(p0 + each, sub); i++) {
        const uint32_t c = s_cnt[i];
        // (minus the tile start: slot y of the tile then goes to place s_at + y of its part)
        s_at[i] = c ? atomicAdd(part_count + b * sub + i, c) - run : 0;
        s_cnt[i] = run;
        run += c;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kSplitItems; u++)
        if (u * kThreads + threadIdx.x < tn) s_rec[s_cnt[part[u]] + rank[u]] = rec[u];
    __syncthreads();
    for (uint32_t y = threadIdx.x; y < tn; y += kThreads) {
        const ulonglong2 e = s_rec[y];
        const uint32_t q = (uint32_t)TM_CHK_IDX(pair_part(sm64_mix(e.x), parts) - b * sub, sub, kChkRange), at = s_at[q] + y;
        if (at < (uint32_t)kPartSlots) slots[(size_t)(b * sub + q) * kPartSlots + at] = e;
        else *B.full = 1;
    }
}

// Third step: a block reads its part's list, builds the part in shared memory and writes it over
// the list.
__global__ void __launch_bounds__(kThreads) k_pair_build(const uint32_t* __restrict__ part_count, ulonglong2* __restrict__ slots,
                                                         uint32_t* __restrict__ full) {
    extern __shared__ __align__(16) unsigned char sm_part[];
    ulonglong2* part = (ulonglong2*)sm_part;   // [kPartSlots]
    ulonglong2* mine = slots + (size_t)blockIdx.x * kPartSlots;
    const uint32_t n = part_count[blockIdx.x];
    if (n >= (uint32_t)kPartSlots) {   // no empty slot would be left: the caller builds another table
        if (threadIdx.x == 0) *full = 1;
        return;
    }
    for (int i = threadIdx.x; i < kPartSlots; i += kThreads) part[i] = make_ulonglong2(kHashEmpty, kHashEmpty);
    __syncthreads();
    constexpr int U = 4;
    for (uint32_t i0 = 0; i0 < n; i0 += U * kThreads) {
        ulonglong2 e[U];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (i0 + u * kThreads + threadIdx.x < n) e[u] = mine[i0 + u * kThreads + threadIdx.x];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (i0 + u * kThreads + threadIdx.x < n) pair_insert((unsigned long long*)part, kPartSlots - 1, e[u]);
    }
    __syncthreads();   // the whole list has been read
    for (int i = threadIdx.x; i < kPartSlots; i += kThreads) mine[i] = part[i];
}

// Where each pair-view entry's pair starts and ends, and the pairs themselves into the pair filter
// (and, BUCKETS, into the lists that the pair table is built from), in one pass.  A pair starts
// where (source, destination) changes: ballots give one bit per entry, and an entry's start and
// end are the nearest set bits in its tile's 128 words; the segments that cross a tile's two
// borders are found by a binary search for the border entry's destination inside its source
// (sorted by destination), so that no tile waits on another.  (Numbering the pairs instead needs
// a scan over tiles: its look-back was half of that kernel's 0.12 ms on 1e7 edges, and every use
// of a pair's number was a further dependent load.)
constexpr int kPairItems = 16;
constexpr int kPairTile = kThreads * kPairItems;
constexpr int kPairWords = kPairTile / 32;
template <bool BUCKETS>
__global__ void __launch_bounds__(kThreads) k_pairs(const uint32_t* __restrict__ src, const int32_t* __restrict__ dst,
                        const int64_t* __restrict__ out_off, int64_t m, int32_t n, int32_t* __restrict__ pair_beg,
                        int32_t* __restrict__ pair_end, PairBuckets B, uint32_t* __restrict__ filt, unsigned long long fmask, unsigned long long* __restrict__ P, const uint32_t* err) {
    __shared__ uint32_t s_head[kPairWords];
    __shared__ int s_prev[kPairWords], s_next[kPairWords];   // last start before the word, first after it
    __shared__ int32_t s_beg, s_end;                         // of the segments crossing the tile's borders
    __shared__ uint32_t s_cnt[kBuckets], s_base[kBuckets];   // the tile's records per list, and their place
    if (gave_up(err)) return;
    if (BUCKETS && threadIdx.x < kBuckets) s_cnt[threadIdx.x] = 0;
    const int64_t tbase = (int64_t)blockIdx.x * kPairTile;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int k0 = w * kPairItems;   // the warp's first word
    const int64_t base = tbase + k0 * 32 + lane;
    uint32_t s[kPairItems];
    int32_t d[kPairItems];
#pragma unroll
    for (int r = 0; r < kPairItems; r++) {
        const int64_t i = base + r * 32;
        s[r] = i < m ? src[i] : 0;
        d[r] = i < m ? dst[i] : 0;
    }
    // the entry before the warp's first; every other one is a neighbouring lane's or round's
    uint32_t ls = 0;
    int32_t ld = 0;
    if (lane == 0 && base > 0 && base < m) {
        ls = src[base - 1];
        ld = dst[base - 1];
    }
    if (threadIdx.x == 0) s_beg = (int32_t)lower_bound_i32(dst, out_off[TM_CHK_IDX(s[0], n, kChkNode)], tbase, d[0]);
    if (threadIdx.x == 32) {
        const int64_t last = min(m, tbase + kPairTile) - 1;
        const int32_t dl = dst[last];
        int64_t lo = last + 1, hi = out_off[TM_CHK_IDX(src[last], n, kChkNode) + 1];
        while (lo < hi) {
            const int64_t mid = lo + ((hi - lo) >> 1);
            if (dst[mid] <= dl) lo = mid + 1; else hi = mid;
        }
        s_end = (int32_t)lo;
    }
#pragma unroll
    for (int r = 0; r < kPairItems; r++) {
        const int64_t i = base + r * 32;
        uint32_t ps = __shfl_up_sync(kFull, s[r], 1);
        int32_t pd = __shfl_up_sync(kFull, d[r], 1);
        if (lane == 0) {
            ps = ls;
            pd = ld;
        }
        const unsigned h = __ballot_sync(kFull, i < m && (i == 0 || s[r] != ps || d[r] != pd));
        if (lane == 0) s_head[k0 + r] = h;
        ls = __shfl_sync(kFull, s[r], 31);
        ld = __shfl_sync(kFull, d[r], 31);
    }
    __syncthreads();
    if (w == 0) {
        // per word the nearest starts outside it: running maximum from the left, minimum from the right
        constexpr int W = kPairWords / 32;
        int last = -1, first = kPairTile, pairs = 0;
#pragma unroll
        for (int x = 0; x < W; x++) {
            const uint32_t h = s_head[lane * W + x];
            pairs += __popc(h);
            if (h) {
                last = 32 * (lane * W + x) + 31 - __clz(h);
                if (first == kPairTile) first = 32 * (lane * W + x) + __ffs(h) - 1;
            }
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(kFull, last, o), b = __shfl_down_sync(kFull, first, o);
            if (lane >= o) last = max(last, a);
            if (lane + o < 32) first = min(first, b);
        }
        int before = __shfl_up_sync(kFull, last, 1), after = __shfl_down_sync(kFull, first, 1);
        if (lane == 0) before = -1;
        if (lane == 31) after = kPairTile;
#pragma unroll
        for (int x = 0; x < W; x++) {
            const int k = lane * W + x, y = lane * W + W - 1 - x;
            s_prev[k] = before;
            if (s_head[k]) before = 32 * k + 31 - __clz(s_head[k]);
            s_next[y] = after;
            if (s_head[y]) after = 32 * y + __ffs(s_head[y]) - 1;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(kFull, pairs, o);
        if (lane == 0 && pairs) atomicAdd(P, (unsigned long long)pairs);
    }
    __syncthreads();
    uint32_t place[kPairItems];   // BUCKETS: list << 16 | the record's rank among the tile's in it
#pragma unroll
    for (int r = 0; r < kPairItems; r++) {
        const int64_t i = base + r * 32;
        if (i >= m) continue;
        const int k = k0 + r;
        const uint32_t h = s_head[k];
        const uint32_t le = h & (0xffffffffu >> (31 - lane)), gt = h & (0xfffffffeu << lane);
        const int pb = le ? 32 * k + 31 - __clz(le) : s_prev[k];
        const int pe = gt ? 32 * k + __ffs(gt) - 1 : s_next[k];
        const int32_t end = pe < kPairTile ? (int32_t)(tbase + pe) : s_end;
        const int32_t beg = pb >= 0 ? (int32_t)(tbase + pb) : s_beg;
        TM_CHK(beg >= 0 && beg <= i && i < end && end <= m, kChkRange);
        pair_beg[i] = beg;
        pair_end[i] = end;
        if ((h >> lane) & 1u) {
            const unsigned long long key = pair_key((int32_t)s[r], d[r]), hash = sm64_mix(key);
            atomicOr(filt + ((hash >> 10) & fmask), pair_bits(hash));
            if constexpr (BUCKETS) {
                const uint32_t b = (uint32_t)((hash >> 32) / (0x100000000ull / kBuckets));
                place[r] = (b << 16) | atomicAdd(&s_cnt[b], 1u);
            }
        }
    }
    if constexpr (BUCKETS) {
        __syncthreads();
        if (threadIdx.x < kBuckets) s_base[threadIdx.x] = atomicAdd(B.count + threadIdx.x, s_cnt[threadIdx.x]);
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kPairItems; r++) {
            const int64_t i = base + r * 32;
            const int k = k0 + r;
            const uint32_t h = s_head[k];
            if (i >= m || !((h >> lane) & 1u)) continue;
            const uint32_t gt = h & (0xfffffffeu << lane);
            const int pe = gt ? 32 * k + __ffs(gt) - 1 : s_next[k];
            const int32_t end = pe < kPairTile ? (int32_t)(tbase + pe) : s_end;
            const uint32_t b = place[r] >> 16, at = s_base[b] + (place[r] & 0xffffu);
            if (at < B.cap)
                B.rec[(size_t)b * B.cap + at] = pair_slot_value((int32_t)s[r], d[r], i, end);
            else
                *B.full = 1;
        }
    }
}

// Edges from which the pair table is built part by part: below, a table with room for every edge
// (at most 2^22 slots, 64 MB) stays in L2, and one kernel that inserts is quicker than two steps of
// lists (about 20 us of insertion for 7e5 pairs).
constexpr int64_t kPartEdges = (int64_t)1 << 21;
constexpr size_t kSpareBytes = (size_t)4 << 20;   // a table of at most this size stays as it is

int bits_for(int32_t n) {
    int b = 0;
    while (b < 31 && ((int64_t)1 << b) < (int64_t)n) b++;
    return b;
}

// allows a kernel more dynamic shared memory than the 48 KB default, once per device
int allow_smem(const void* kernel, int bytes, int which) {
    static std::mutex mu;
    static bool done[64][2] = {};
    int dev = 0;
    TM_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(mu);
    if (dev >= 0 && dev < 64 && done[dev][which]) return TM_OK;
    TM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    if (dev >= 0 && dev < 64) done[dev][which] = true;
    return TM_OK;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// the input checks on their own, for callers that give no n_nodes or whose times span too much:
// max id through *n_ids
int check_edges(const int32_t* d_src, const int32_t* d_dst, const int64_t* d_t, int64_t m, int32_t n_nodes,
                cudaStream_t st, int32_t* n_ids) {
    int32_t* flags = nullptr;
    TM_CUDA(cudaMallocAsync((void**)&flags, 4 * sizeof(int32_t), st));
    int32_t hf[4] = {0, 0, -1, 0};
    cudaError_t e = cudaMemcpyAsync(flags, hf, sizeof(hf), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        k_validate<<<grid_for(m), kThreads, 0, st>>>(d_src, d_dst, d_t, m, n_nodes, flags); count_launch();
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);   // hf has been read
    if (e == cudaSuccess) e = cudaMemcpyAsync(hf, flags, sizeof(hf), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFreeAsync(flags, st);
    TM_CUDA(e);
    if (hf[0]) { set_error("timestamps are not sorted non-decreasingly"); return TM_EUNSORTED; }
    if (hf[1]) { set_error("node id outside [0, n_nodes)"); return TM_ERANGE; }
    *n_ids = hf[2] + 1;
    return TM_OK;
}

}  // namespace

int build_graph(const int32_t* d_src, const int32_t* d_dst, const int64_t* d_t, const int64_t* h_t, int64_t m,
                int32_t n_nodes, cudaStream_t st, tm_graph** out) {
    if (!out) { set_error("out is NULL"); return TM_EINVAL; }
    *out = nullptr;
    if (m < 0 || m >= ((int64_t)1 << 31) - 1) { set_error("m outside [0, 2^31-1)"); return TM_EINVAL; }
    if (m > 0 && (!d_src || !d_dst || !d_t)) { set_error("NULL edge array"); return TM_EINVAL; }
    if (n_nodes < -1) { set_error("n_nodes < -1"); return TM_EINVAL; }

    int dev = 0;
    TM_CUDA(cudaGetDevice(&dev));
    PhaseEvents pe(profiling());
    NvtxPhases nv;
    nv.next("tm_graph_build");
    int ev0 = pe.mark(st);
    int64_t tmin = 0, tmax = 0;
    int32_t n = n_nodes < 0 ? 0 : n_nodes;
    if (m > 0) {
        int64_t tt[2];
        if (h_t) {
            tt[0] = h_t[0];
            tt[1] = h_t[m - 1];
        } else {
            TM_CUDA(cudaMemcpyAsync(&tt[0], d_t, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
            TM_CUDA(cudaMemcpyAsync(&tt[1], d_t + (m - 1), sizeof(int64_t), cudaMemcpyDeviceToHost, st));
            TM_CUDA(cudaStreamSynchronize(st));
        }
        if (tt[1] < tt[0]) { set_error("timestamps are not sorted non-decreasingly"); return TM_EUNSORTED; }
        tmin = tt[0];
        const uint64_t span = (uint64_t)tt[1] - (uint64_t)tt[0];
        if (n <= 0 || span >= (uint64_t)1 << 61) {   // ids counted, or a wrong input told apart, first
            int32_t ids = 0;
            TM_TRY(check_edges(d_src, d_dst, d_t, m, n_nodes, st, &ids));
            if (span >= (uint64_t)1 << 61) { set_error("time span >= 2^61"); return TM_EINVAL; }
            if (n_nodes < 0) n = ids;
        }
        tmax = (int64_t)span;
    }

    // ---- one allocation for the resident graph
    size_t nN = (size_t)n + 1, M = (size_t)m;
    // time arrays hold int32 when every normalised time fits, else int64
    const int tb = tmax <= (int64_t)INT32_MAX ? 4 : 8;
    size_t sz_i32m = align256(4 * M), sz_off = align256(8 * nN);
    size_t sz_tm = align256((size_t)tb * M);
    size_t total = 2 * sz_i32m + sz_tm              // src, dst, t
                 + sz_off + 2 * sz_i32m + sz_tm     // out view
                 + sz_off + 2 * sz_i32m + sz_tm     // in view
                 + 3 * sz_i32m + sz_tm;             // pair view
    tm_graph* g = new (std::nothrow) tm_graph();
    if (!g) { set_error("host allocation failed"); return TM_ENOMEM; }
    g->device = dev;
    g->m = m;
    g->n = n;
    g->t_min = tmin;
    g->t_max = tmax;
    g->bytes = (int64_t)total;
    pool_prepare(dev);
    cudaError_t e = cudaMallocAsync(&g->block, total, st);
    if (e != cudaSuccess) {
        delete g;
        return cuda_status(e, "cudaMalloc(graph)", __FILE__, __LINE__);
    }
    char* p = (char*)g->block;
    auto take = [&](size_t bytes) { char* r = p; p += bytes; return (void*)r; };
    int32_t* gs = (int32_t*)take(sz_i32m);
    int32_t* gd = (int32_t*)take(sz_i32m);
    void* gt = take(sz_tm);
    int64_t* out_off = (int64_t*)take(sz_off);
    int32_t* out_src = (int32_t*)take(sz_i32m);
    int32_t* out_nbr = (int32_t*)take(sz_i32m);
    void* out_t = take(sz_tm);
    int64_t* in_off = (int64_t*)take(sz_off);
    int32_t* in_dst = (int32_t*)take(sz_i32m);
    int32_t* in_nbr = (int32_t*)take(sz_i32m);
    void* in_t = take(sz_tm);
    int32_t* pair_dst = (int32_t*)take(sz_i32m);
    int32_t* pair_beg = (int32_t*)take(sz_i32m);
    int32_t* pair_end = (int32_t*)take(sz_i32m);
    void* pair_t = take(sz_tm);

    GraphDev& G = g->dev;
    G.m = m; G.n = n; G.tbytes = tb; G.loops = 0;
    G.per_tick = 1.0f / ((float)tmax + 1.0f);
    G.src = gs; G.dst = gd; G.t = gt;
    G.out_off = out_off; G.out_nbr = out_nbr; G.out_t = out_t;
    G.in_off = in_off; G.in_nbr = in_nbr; G.in_t = in_t;
    G.pair_dst = pair_dst; G.pair_beg = pair_beg; G.pair_end = pair_end; G.pair_t = pair_t;
    G.out_src = out_src; G.in_dst = in_dst;
    G.hslots = nullptr; G.hparts = 0; G.hmask = 0;
    G.pfilt = nullptr; G.pfmask = 0;
    g->hash_block = nullptr;
    g->table_block = nullptr;
    g->ex_own_block = nullptr;
    g->ex_rev_block = nullptr;

    int rc = TM_OK;
    if (m == 0) {
        TM_CUDA(cudaMemsetAsync(out_off, 0, 8 * nN, st));
        TM_CUDA(cudaMemsetAsync(in_off, 0, 8 * nN, st));
        TM_CUDA(cudaStreamSynchronize(st));
        g->P = 0;
        G.P = 0;
        *out = g;
        return TM_OK;
    }

    // ---- pair filter: about 8 bits per edge (a power of two of 32-bit words, sized by the edges so
    // that the build need not wait for the number of pairs), at most 32 MB so that it stays in L2;
    // a small graph's pair table before it, of one part with room for every edge
    const bool parted = m >= kPartEdges;
    uint64_t cap = 2;
    while (2 * cap < 3 * (uint64_t)m) cap <<= 1;
    unsigned long long fw = 1;
    while (fw < ((unsigned long long)m + 7) / 8 && fw < (1ull << 23)) fw <<= 1;
    const size_t table_bytes = parted ? 0 : 16 * cap;
    e = cudaMallocAsync(&g->hash_block, table_bytes + 4 * fw, st);
    if (e != cudaSuccess) {
        cudaStreamSynchronize(st);
        pool_free(g->block, dev);
        delete g;
        return cuda_status(e, "cudaMalloc(pair table)", __FILE__, __LINE__);
    }
    g->bytes += (int64_t)(table_bytes + 4 * fw);
    uint32_t* filt = (uint32_t*)((char*)g->hash_block + table_bytes);
    G.pfilt = filt;
    G.pfmask = fw - 1;

    // ---- scratch: the lists between the passes of two sorts, the sorts' counts and tile words.
    // The sorts' spare words hold the flags and the pair count.
    const SortDigits D = sort_digits(bits_for(n));
    const size_t set = 2 * sz_i32m + sz_tm, ws_bytes = align256(sort_ws_bytes(m, D, 3, 2)) + 256;   // (256: the lists' counts)
    const size_t pc_bytes = align256(4 * (size_t)pair_parts(m));   // the parts' counts
    const size_t space = std::max(2 * set, parted ? 16 * ((size_t)m + m / 8 + 1024 * kBuckets) + pc_bytes : 0);
    ScratchLease lease;
    int lrc = scratch_acquire(space + ws_bytes, st, lease);
    if (lrc != TM_OK) {
        cudaStreamSynchronize(st);
        pool_free(g->block, dev);
        pool_free(g->hash_block, dev);
        pool_free(g->table_block, dev);
        delete g;
        return lrc;
    }
    char* q = (char*)lease.p;
    const SortWs W = sort_ws(q, m, D, 3, 2);
    uint32_t* flags = W.err + 8;   // 4 flags, then the pair count, list-full mark, ...
    PairBuckets B;                 // ... and in the sorts' space, free by then, the pair lists
    B.cap = (uint32_t)(m / kBuckets + m / (8 * kBuckets) + 1024);
    B.count = (uint32_t*)(q + ws_bytes) - kBuckets;
    B.full = W.err + 20;
    uint32_t* part_count = (uint32_t*)(q + ws_bytes);
    B.rec = (ulonglong2*)(q + ws_bytes + pc_bytes);
    unsigned long long* dP = (unsigned long long*)(W.err + 16);
    q += ws_bytes;
    SortIo io[2];   // out view: (source; destination, time) by source; in view the other way round
    for (int k = 0; k < 2; k++) {
        io[k].key_in = (const uint32_t*)(k ? gd : gs);
        io[k].a_in = (const uint32_t*)(k ? gs : gd);
        io[k].t_in = gt;
        io[k].key_out = (uint32_t*)(k ? in_dst : out_src);
        io[k].a_out = (uint32_t*)(k ? in_nbr : out_nbr);
        io[k].t_out = k ? in_t : out_t;
        io[k].key_tmp = (uint32_t*)q;
        io[k].a_tmp = (uint32_t*)(q + sz_i32m);
        io[k].t_tmp = q + 2 * sz_i32m;
        io[k].counts = k;
        io[k].keep_key = true;
        q += set;
    }
    // pair view: the in view stably re-sorted by source = (source, destination, time); its
    // sources are the out view's, so the last pass need not write them
    SortIo pr = io[0];
    pr.key_in = (const uint32_t*)in_nbr;
    pr.a_in = (const uint32_t*)in_dst;
    pr.t_in = in_t;
    pr.key_out = io[1].key_tmp;   // (three or more passes go through it)
    pr.a_out = (uint32_t*)pair_dst;
    pr.t_out = pair_t;
    pr.keep_key = false;

    auto launched = [&]() {
        count_launch();
        if (rc == TM_OK && cudaGetLastError() != cudaSuccess) {
            set_error("graph build launch failed");
            rc = TM_ECUDA;
        }
    };
    rc = sort_clear(W, st);
    if (rc == TM_OK && ((!parted && cudaMemsetAsync(g->hash_block, 0xff, table_bytes, st) != cudaSuccess) ||
                        cudaMemsetAsync(filt, 0, 4 * fw, st) != cudaSuccess ||
                        cudaMemsetAsync(B.count, 0, 4 * kBuckets, st) != cudaSuccess))
        rc = cuda_status(cudaGetLastError(), "pair table", __FILE__, __LINE__);
    if (rc == TM_OK) {
        const size_t sm = (size_t)8 * D.passes << D.db;
        const unsigned gi = (unsigned)std::min<int64_t>((m + 4 * kIngestThreads - 1) / (4 * kIngestThreads), (int64_t)sm_count() * 4);
        if (tb == 4)
            k_ingest<int32_t><<<gi, kIngestThreads, sm, st>>>(d_src, d_dst, d_t, m, tmin, n, gs, gd, (int32_t*)gt, flags, D, W.counts);
        else
            k_ingest<int64_t><<<gi, kIngestThreads, sm, st>>>(d_src, d_dst, d_t, m, tmin, n, gs, gd, (int64_t*)gt, flags, D, W.counts);
        launched();
    }
    if (rc == TM_OK) rc = sort_bases(W, st);
    if (rc == TM_OK) rc = sort_run(W, io, 2, 0, tb, st);
    if (rc == TM_OK) rc = sort_run(W, &pr, 1, 2, tb, st);
    if (rc == TM_OK) {
        k_offsets<<<dim3((unsigned)((m / 4 + kThreads) / kThreads), 2), kThreads, 0, st>>>(
            (const uint32_t*)out_src, (const uint32_t*)in_dst, m, n, out_off, in_off, W.err);
        launched();
    }
    if (rc == TM_OK) {
        const unsigned gp = (unsigned)((m + kPairTile - 1) / kPairTile);
        if (parted)
            k_pairs<true><<<gp, kThreads, 0, st>>>((const uint32_t*)out_src, pair_dst, out_off, m, n, pair_beg, pair_end, B, filt, fw - 1, dP, W.err);
        else
            k_pairs<false><<<gp, kThreads, 0, st>>>((const uint32_t*)out_src, pair_dst, out_off, m, n, pair_beg, pair_end, B, filt, fw - 1, dP, W.err);
        launched();
    }
    uint32_t h[24];   // error word, flags, pair count, list-full mark
    // waits for the build so far and takes the first thing that is wrong with it
    auto settle = [&]() {
        e = cudaMemcpyAsync(h, W.err, sizeof(h), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) rc = cuda_status(e, "graph build", __FILE__, __LINE__);
        else if (h[8]) { set_error("timestamps are not sorted non-decreasingly"); rc = TM_EUNSORTED; }
        else if (h[9]) { set_error("node id outside [0, n_nodes)"); rc = TM_ERANGE; }
        else if (h[0]) { set_error("graph build: a wait for an earlier tile expired"); rc = TM_ECUDA; }
    };
    auto insert_all = [&](void* table, uint64_t slots) {   // into an emptied table of one part
        G.hslots = (const unsigned long long*)table;
        G.hparts = 1;
        G.hmask = (uint32_t)(slots - 1);
        k_pair_insert<<<grid_for(m, 32), kThreads, 0, st>>>(out_src, pair_dst, pair_beg, pair_end, m, (unsigned long long*)table, G.hmask, W.err);
        launched();
    };
    if (rc == TM_OK && !parted) insert_all(g->hash_block, cap);
    if (rc == TM_OK && parted) {
        settle();
        uint64_t P = 0;
        if (rc == TM_OK) std::memcpy(&P, h + 16, 8);
        const uint32_t parts = pair_parts((int64_t)P);
        const size_t part_bytes = (size_t)16 * kPartSlots;
        if (rc == TM_OK) {
            e = cudaMallocAsync(&g->table_block, parts * part_bytes, st);
            if (e != cudaSuccess) rc = cuda_status(e, "cudaMalloc(pair table)", __FILE__, __LINE__);
        }
        const uint32_t sub = parts / kBuckets;
        const size_t split_sm = 16 * (size_t)kSplitTile + 8 * (size_t)sub;
        if (rc == TM_OK) rc = allow_smem((const void*)k_pair_split, 16 * kSplitTile + 160 * 1024, 0);
        if (rc == TM_OK) rc = allow_smem((const void*)k_pair_build, (int)part_bytes, 1);
        if (rc == TM_OK && cudaMemsetAsync(part_count, 0, 4 * (size_t)parts, st) != cudaSuccess)
            rc = cuda_status(cudaGetLastError(), "pair table", __FILE__, __LINE__);
        if (rc == TM_OK) {
            g->bytes += (int64_t)(parts * part_bytes);
            G.hslots = (const unsigned long long*)g->table_block;
            G.hparts = parts;
            G.hmask = kPartSlots - 1;
            const unsigned per = (B.cap + kSplitTile - 1) / kSplitTile;
            k_pair_split<<<per * kBuckets, kThreads, split_sm, st>>>(B, parts, part_count, (ulonglong2*)g->table_block);
            launched();
            k_pair_build<<<parts, kThreads, part_bytes, st>>>(part_count, (ulonglong2*)g->table_block, B.full);
            launched();
        }
    }
    int ev1 = pe.mark(st);
    if (rc == TM_OK) settle();
    if (rc == TM_OK && h[20]) {
        // more pairs hashed into one list or part than it holds: one part with room for every pair
        uint64_t P = 0, slots = 2;
        std::memcpy(&P, h + 16, 8);
        while (2 * slots < 3 * P) slots <<= 1;
        pool_free(g->table_block, dev);
        g->table_block = nullptr;
        g->bytes += 16 * ((int64_t)slots - (int64_t)G.hparts * kPartSlots);
        e = cudaMallocAsync(&g->table_block, 16 * slots, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(g->table_block, 0xff, 16 * slots, st);
        if (e != cudaSuccess) rc = cuda_status(e, "cudaMalloc(pair table)", __FILE__, __LINE__);
        if (rc == TM_OK) insert_all(g->table_block, slots);
        if (rc == TM_OK) settle();
    }
    // A small graph whose edges repeat few pairs would keep a table sized by its edges (up to 64 MB
    // where the pairs need kilobytes): beyond kSpareBytes the pairs move to one of their own size.
    // (Only then: waiting for their number first would cost every small build a round trip.)
    if (rc == TM_OK && !parted && table_bytes >= kSpareBytes) {
        uint64_t P = 0, slots = 2;
        std::memcpy(&P, h + 16, 8);
        while (2 * slots < 3 * P) slots <<= 1;
        void* block = nullptr;
        if (4 * slots <= cap && cudaMallocAsync(&block, 16 * slots + 4 * fw, st) == cudaSuccess) {
            uint32_t* f = (uint32_t*)((char*)block + 16 * slots);
            e = cudaMemsetAsync(block, 0xff, 16 * slots, st);
            if (e == cudaSuccess) e = cudaMemcpyAsync(f, filt, 4 * fw, cudaMemcpyDeviceToDevice, st);
            if (e != cudaSuccess) rc = cuda_status(e, "pair table", __FILE__, __LINE__);
            if (rc == TM_OK) insert_all(block, slots);
            if (rc == TM_OK) settle();
            else cudaStreamSynchronize(st);
            std::swap(block, g->hash_block);
            pool_free(block, dev);
            G.pfilt = f;
            g->bytes -= 16 * (int64_t)(cap - slots);
        }
        cudaGetLastError();   // no room for a second table: the first stays
    }
    int64_t P = 0;
    if (rc == TM_OK) {
        G.loops = h[11] ? 1 : 0;
        std::memcpy(&P, h + 16, 8);
        if (pe.on) store_profile_graph(pe.ms(ev0, ev1));
    }
    scratch_release(lease, st);
    if (rc != TM_OK) {
        cudaStreamSynchronize(st);
        pool_free(g->block, dev);
        pool_free(g->hash_block, dev);
        pool_free(g->table_block, dev);
        delete g;
        return rc;
    }
    g->P = P;
    G.P = P;
    *out = g;
    return TM_OK;
}

namespace {

// Two-node tables.  For pair-view position e of pair (u, v) at time t_e:
//   own[e] = number of (u, v) edges with time < t_e, rev[e] = number of (v, u) edges with
//   time < t_e;
// each then turned into exclusive prefix sums over all positions.  The source of pair-view
// position e is out_src[e]: both views group the edges by source in the same ranges.
template <typename TT>
__global__ void k_ex_rank(GraphDevT<TT> G, int reverse, int64_t* __restrict__ out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < G.m;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t te = (int64_t)G.pair_t[e];
        if (!reverse) {
            int64_t pa = G.pair_beg[e];
            int64_t r = e - pa;
            if (e > pa && (int64_t)G.pair_t[e - 1] == te) r = lower_bound_i64(G.pair_t, pa, e, te) - pa;
            out[e] = r;
        } else {
            int32_t u = G.out_src[e], v = G.pair_dst[e];
            int64_t ra, rb;
            out[e] = pair_segment(G, v, u, ra, rb) ? lower_bound_i64(G.pair_t, ra, rb, te) - ra : 0;
        }
    }
}

std::mutex g_ex_mu;

int build_ex_table(tm_graph* g, int reverse, cudaStream_t st, void** blk_out) {
    size_t n1 = (size_t)g->m + 1;
    void* blk = nullptr;
    TM_CUDA(cudaMallocAsync(&blk, align256(8 * n1), st));
    int64_t* a = (int64_t*)blk;
    int rc = TM_OK;
    cudaError_t e = cudaMemsetAsync(a + g->m, 0, 8, st);
    if (e == cudaSuccess) {
        if (g->dev.tbytes == 4) k_ex_rank<int32_t><<<grid_for(g->m), kThreads, 0, st>>>(typed<int32_t>(g->dev), reverse, a);
        else k_ex_rank<int64_t><<<grid_for(g->m), kThreads, 0, st>>>(typed<int64_t>(g->dev), reverse, a);
        count_launch();
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) rc = cuda_status(e, "two-node table", __FILE__, __LINE__);
    if (rc == TM_OK) rc = scan_exclusive_i64(a, a, (int64_t)n1, nullptr, st);
    if (rc == TM_OK) {
        e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) rc = cuda_status(e, "two-node table", __FILE__, __LINE__);
    }
    if (rc != TM_OK) {
        cudaStreamSynchronize(st);
        pool_free(blk, g->device);
        return rc;
    }
    g->bytes += (int64_t)align256(8 * n1);
    *blk_out = blk;
    return TM_OK;
}

}  // namespace

int ensure_ex_tables(tm_graph* g, cudaStream_t st, bool need_own, bool need_rev, const int64_t** own,
                     const int64_t** rev) {
    std::lock_guard<std::mutex> lk(g_ex_mu);
    *own = *rev = nullptr;
    if (g->m == 0) return TM_OK;
    int rc = TM_OK;
    if (need_own && !g->ex_own_block) rc = build_ex_table(g, 0, st, &g->ex_own_block);
    if (rc == TM_OK && need_rev && !g->ex_rev_block) rc = build_ex_table(g, 1, st, &g->ex_rev_block);
    if (rc != TM_OK) return rc;
    if (need_own) *own = (const int64_t*)g->ex_own_block;
    if (need_rev) *rev = (const int64_t*)g->ex_rev_block;
    return TM_OK;
}

}  // namespace tmo

extern "C" {

int tm_graph_load_device(const int32_t* d_src, const int32_t* d_dst, const int64_t* d_t, int64_t m,
                         int32_t n_nodes, void* stream, tm_graph** out) {
    return tmo::build_graph(d_src, d_dst, d_t, nullptr, m, n_nodes, (cudaStream_t)stream, out);
}

int tm_graph_load(const int32_t* src, const int32_t* dst, const int64_t* t, int64_t m,
                  int32_t n_nodes, tm_graph** out) {
    if (!out) { tmo::set_error("out is NULL"); return TM_EINVAL; }
    *out = nullptr;
    if (m < 0 || m >= ((int64_t)1 << 31) - 1) { tmo::set_error("m outside [0, 2^31-1)"); return TM_EINVAL; }
    if (m > 0 && (!src || !dst || !t)) { tmo::set_error("NULL edge array"); return TM_EINVAL; }
    cudaStream_t st;
    TM_CUDA(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
    size_t M = (size_t)(m > 0 ? m : 1);
    tmo::ScratchLease lease;   // the three staged arrays
    int rc = tmo::scratch_acquire(2 * tmo::align256(4 * M) + 8 * M, st, lease);
    if (rc != TM_OK) {
        cudaStreamDestroy(st);
        return rc;
    }
    int32_t* ds = (int32_t*)lease.p;
    int32_t* dd = (int32_t*)((char*)lease.p + tmo::align256(4 * M));
    int64_t* dt = (int64_t*)((char*)lease.p + 2 * tmo::align256(4 * M));
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess && m > 0) e = cudaMemcpyAsync(ds, src, 4 * (size_t)m, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && m > 0) e = cudaMemcpyAsync(dd, dst, 4 * (size_t)m, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && m > 0) e = cudaMemcpyAsync(dt, t, 8 * (size_t)m, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) rc = tmo::cuda_status(e, "tm_graph_load copy", __FILE__, __LINE__);
    if (rc == TM_OK) rc = tmo::build_graph(ds, dd, dt, t, m, n_nodes, st, out);
    tmo::scratch_release(lease, st);
    cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
    return rc;
}

void tm_graph_free(tm_graph* g) {
    if (!g) return;
    tmo::pool_free(g->block, g->device);
    tmo::pool_free(g->hash_block, g->device);
    tmo::pool_free(g->table_block, g->device);
    tmo::pool_free(g->ex_own_block, g->device);
    tmo::pool_free(g->ex_rev_block, g->device);
    delete g;
}

int tm_graph_get_info(const tm_graph* g, tm_graph_info* info) {
    if (!g || !info) { tmo::set_error("NULL argument"); return TM_EINVAL; }
    std::memset(info, 0, sizeof(*info));
    info->m = g->m;
    info->n_nodes = g->n;
    info->n_pairs = g->P;
    info->t_min = g->t_min;
    info->t_max = g->t_max;
    info->device_bytes = g->bytes;
    return TM_OK;
}

}  // extern "C"

namespace tmo {
TM_DEFINE_CHECK_WORD(check_word_graph)
}  // namespace tmo
