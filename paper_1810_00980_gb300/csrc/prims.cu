// Device primitives: exclusive scans into int64 (reduce-then-scan over tiles, where no block waits
// on another; up to 1,024 tiles in one launch, where a tile waits, with a limit, for the sums of
// earlier tiles) and a stable LSD radix sort of 32-bit keys with up to 12 bytes of payload (a tile
// waits, with a limit, for the counts of earlier tiles).
#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

#include "tm_internal.cuh"

namespace tmo {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;   // 2048

__device__ __forceinline__ int64_t warp_incl_scan(int64_t v) {
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t u = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// block-wide exclusive scan of one value per thread; returns the block total in *total
__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t* smem, int64_t* total) {
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int64_t inc = warp_incl_scan(v);
    if (lane == 31) smem[w] = inc;
    __syncthreads();
    if (w == 0) {
        int nw = blockDim.x >> 5;
        int64_t s = lane < nw ? smem[lane] : 0;
        int64_t si = warp_incl_scan(s);
        if (lane < nw) smem[lane] = si - s;
        if (lane == nw - 1) smem[32] = si;
    }
    __syncthreads();
    int64_t r = inc - v + smem[w];
    *total = smem[32];
    __syncthreads();
    return r;
}

// Each block scans one tile (exclusive), writes the tile total to sums[tile].
// (in may equal out: every thread reads its items before any thread writes)
__global__ void k_scan_tiles(const int64_t* in, int64_t* out, int64_t n, int64_t* __restrict__ sums) {
    // the tile passes through shared memory (padded: no bank conflicts) so that loads and
    // stores are coalesced
    __shared__ int64_t smem[33];
    __shared__ int64_t tile[kScanTile + kScanTile / 16];
    int64_t t0 = (int64_t)blockIdx.x * kScanTile;
    for (int i = threadIdx.x; i < kScanTile; i += blockDim.x) {
        int64_t idx = t0 + i;
        tile[i + (i >> 4)] = idx < n ? in[idx] : 0;
    }
    __syncthreads();
    int b = threadIdx.x * kScanItems;
    int64_t v[kScanItems];
    int64_t loc = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        v[i] = tile[b + i + ((b + i) >> 4)];
        loc += v[i];
    }
    int64_t total;
    int64_t run = block_excl_scan(loc, smem, &total);
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        tile[b + i + ((b + i) >> 4)] = run;
        run += v[i];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kScanTile; i += blockDim.x) {
        int64_t idx = t0 + i;
        if (idx < n) out[idx] = tile[i + (i >> 4)];
    }
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// 32-bit lengths -> 64-bit exclusive offsets, reduce-then-scan (each length read twice, each
// offset written once): per-tile sums first (tiles at or past the count, read on the device
// when d_n is given, sum to 0) ...
__global__ void k_len_reduce(const int32_t* __restrict__ in, int64_t n_max, const int64_t* __restrict__ d_n,
                             int64_t* __restrict__ sums) {
    __shared__ int64_t smem[33];
    int64_t n = d_n ? min(*d_n, n_max) : n_max;
    int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t loc = 0;
    for (int i = threadIdx.x; i < kScanTile; i += blockDim.x) {
        int64_t idx = base + i;
        if (idx < n) loc += in[idx];
    }
    int64_t total;
    block_excl_scan(loc, smem, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// Item starts: cf[i] = the element whose range holds item i * grain.  Each thread notes its own
// elements' (those of a range past kBigRange are left to the whole block: noted by one thread, the
// range of a hub's burst would be a long serial run of stores).
constexpr int64_t kBigRange = 2048;
struct BigRanges {
    int n;
    int64_t e[32], from[32], len[32];
};
__device__ __forceinline__ void note_items(BigRanges& B, int64_t* cf, int64_t ncf, int grain, int64_t e, int64_t from,
                                           int64_t len) {
    if (len > kBigRange) {
        const int k = atomicAdd(&B.n, 1);
        if (k < 32) {
            B.e[k] = e; B.from[k] = from; B.len[k] = len;
            return;
        }
    }
    for (int64_t i = (from + grain - 1) / grain; i * grain < from + len && i < ncf; i++) cf[TM_CHK_IDX(i, ncf, kChkSort)] = e;
}
__device__ __forceinline__ void note_big(const BigRanges& B, int64_t* cf, int64_t ncf, int grain) {
    for (int k = 0; k < min(B.n, 32); k++)
        for (int64_t i = (B.from[k] + grain - 1) / grain + threadIdx.x;
             i * grain < B.from[k] + B.len[k] && i < ncf; i += blockDim.x)
            cf[TM_CHK_IDX(i, ncf, kChkSort)] = B.e[k];
}

// ... then each tile's exclusive scan plus the tile's offset; the tile passes through shared
// memory so that both the 32-bit loads and the 64-bit stores are coalesced.  cf: as k_scan_once
__global__ void k_len_scan(const int32_t* __restrict__ in, int64_t* __restrict__ out, int64_t n_max,
                           const int64_t* __restrict__ d_n, const int64_t* __restrict__ offs,
                           int64_t* __restrict__ cf, int64_t ncf) {
    __shared__ int64_t smem[33];
    __shared__ int64_t tile[kScanTile + kScanTile / 16];   // one pad word per 16: no bank conflicts
    __shared__ BigRanges big;
    const int grain = item_grain(n_max);
    if (threadIdx.x == 0) big.n = 0;
    int64_t n = d_n ? min(*d_n, n_max) : n_max;
    int64_t t0 = (int64_t)blockIdx.x * kScanTile;
    if (t0 >= n) return;
    for (int i = threadIdx.x; i < kScanTile; i += blockDim.x) {
        int64_t idx = t0 + i;
        tile[i + (i >> 4)] = idx < n ? (int64_t)in[idx] : 0;
    }
    __syncthreads();
    int b = threadIdx.x * kScanItems;
    int64_t v[kScanItems];
    int64_t loc = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        v[i] = tile[b + i + ((b + i) >> 4)];
        loc += v[i];
    }
    int64_t total;
    int64_t run = block_excl_scan(loc, smem, &total) + offs[blockIdx.x];
    if (threadIdx.x == 0 && t0 + kScanTile >= n) {
        const int64_t end = (run + total + grain - 1) / grain;
        if (end < ncf) cf[TM_CHK_IDX(end, ncf, kChkSort)] = n - 1;
    }
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        note_items(big, cf, ncf, grain, t0 + b + i, run, v[i]);
        tile[b + i + ((b + i) >> 4)] = run;
        run += v[i];
    }
    __syncthreads();
    note_big(big, cf, ncf, grain);
    for (int i = threadIdx.x; i < kScanTile; i += blockDim.x) {
        int64_t idx = t0 + i;
        if (idx < n) out[idx] = tile[i + (i >> 4)];
    }
}

__global__ void k_scan_add(int64_t* __restrict__ out, int64_t n, const int64_t* __restrict__ offs) {
    int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t add = offs[blockIdx.x];
    for (int i = threadIdx.x; i < kScanTile; i += blockDim.x) {
        int64_t idx = base + i;
        if (idx < n) out[idx] += add;
    }
}

__global__ void k_scan_small(const int64_t* in, int64_t* out, int64_t n, int64_t* __restrict__ d_total) {
    // single block, n <= kScanTile
    __shared__ int64_t smem[33];
    int64_t base = (int64_t)threadIdx.x * kScanItems;
    int64_t v[kScanItems];
    int64_t loc = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        int64_t idx = base + i;
        v[i] = idx < n ? in[idx] : 0;
        loc += v[i];
    }
    int64_t total;
    int64_t run = block_excl_scan(loc, smem, &total);
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        int64_t idx = base + i;
        if (idx < n) out[idx] = run;
        run += v[i];
    }
    if (threadIdx.x == 0 && d_total) *d_total = total;
}

__global__ void k_set_i64(int64_t* p, int64_t v) { *p = v; }

// Exclusive scan of lengths (TI = int32_t or int64_t) into 64-bit offsets in one launch: a tile's
// sum, then its prefix, go through one word (top two bits: 1 sum known, 2 prefix known; sums below
// 2^62), and a warp looks back over 32 tiles at a time.  Prefixes travel 32 tiles per memory
// latency, so beyond kOnePassTiles tiles the two-pass form is as quick; below, one launch takes
// the place of three to five (a 20,000-edge count spent 22 of its 118 us on them).
// *d_total is zero before and, when a wait expires, below zero afterwards.
// CF also notes the first edge of every grain-th item (cf[i]: the element whose range holds item
// i * grain, grain = item_grain(n_max); past the last, n - 1), as far as cf's ncf entries go.
constexpr int kOneThreads = 256;
constexpr int kOneItems = 16;
constexpr int kOneTile = kOneThreads * kOneItems;

__device__ __forceinline__ unsigned long long ld_tile64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_tile64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

template <typename TI, bool CF>
__global__ void __launch_bounds__(kOneThreads) k_scan_once(const TI* __restrict__ in, int64_t* __restrict__ out, int64_t n_max,
                            const int64_t* __restrict__ d_n, int64_t* __restrict__ d_total, unsigned long long* words,
                            uint32_t* err, int limit, int64_t* __restrict__ cf, int64_t ncf) {
    __shared__ int64_t smem[33];
    __shared__ int64_t tile[kOneTile + kOneTile / 16];   // one pad word per 16: no bank conflicts
    __shared__ int64_t s_before;
    __shared__ uint32_t s_tile;
    __shared__ BigRanges big;
    const int grain = item_grain(n_max);
    if (CF && threadIdx.x == 0) big.n = 0;
    grid_wait();
    const int64_t n = d_n ? min(*d_n, n_max) : n_max;
    if (threadIdx.x == 0) s_tile = gridDim.x == 1 ? 0u : (uint32_t)atomicAdd(words, 1ull);
    __syncthreads();
    const int64_t t = s_tile, t0 = t * kOneTile;
    words += 8;
    if (t0 >= n) return;   // (no elements, or their number is not known: the total stays at zero)
    for (int i = threadIdx.x; i < kOneTile; i += kOneThreads) {
        const int64_t idx = t0 + i;
        tile[i + (i >> 4)] = idx < n ? (int64_t)in[idx] : 0;
    }
    __syncthreads();
    const int b = threadIdx.x * kOneItems;
    int64_t loc = 0;
#pragma unroll
    for (int i = 0; i < kOneItems; i++) loc += tile[b + i + ((b + i) >> 4)];
    int64_t total;
    const int64_t off = block_excl_scan(loc, smem, &total);
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int64_t before = 0;
        bool lost = false;
        if (t > 0) {
            if (lane == 0) st_tile64(words + t, (1ull << 62) | (unsigned long long)total);
            int64_t at = t - 1;
            int spins = 0;
            while (at >= 0) {
                const unsigned long long v = at - lane >= 0 ? ld_tile64(words + (at - lane)) : 2ull << 62;
                const unsigned pre = __ballot_sync(kFull, (v >> 62) == 2), gap = __ballot_sync(kFull, v == 0);
                const int first_gap = gap ? __ffs(gap) - 1 : 32, first_pre = pre ? __ffs(pre) - 1 : 32;
                int64_t x = lane < first_gap && lane <= first_pre ? (int64_t)(v & ((1ull << 62) - 1)) : 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
                before += x;
                if (first_pre < first_gap) break;
                at -= first_gap;
                if (first_gap > 0) {
                    spins = 0;
                } else if (++spins > limit) {
                    if (lane == 0) atomicOr(err, 1u);
                    lost = true;
                } else if ((spins & 63) == 0) {
                    lost = __any_sync(kFull, ld_tile((const uint32_t*)err) != 0);
                }
                if (lost) break;
            }
        }
        if (lost) {
            // no item may be taken from offsets that were not written: whichever comes first, the
            // last tile's total or this, what stays is below zero
            if (lane == 0) {
                atomicMin((long long*)d_total, -1ll);
                s_before = -1;
            }
        } else if (lane == 0) {
            if (gridDim.x > 1) st_tile64(words + t, (2ull << 62) | (unsigned long long)(before + total));
            s_before = before;
            if (t0 + kOneTile >= n) {
                atomicCAS((unsigned long long*)d_total, 0ull, (unsigned long long)(before + total));
                if (CF) {
                    const int64_t end = (before + total + grain - 1) / grain;
                    if (end < ncf) cf[TM_CHK_IDX(end, ncf, kChkSort)] = n - 1;
                }
            }
        }
    }
    __syncthreads();
    if (s_before < 0) return;   // the wait expired
    int64_t run = s_before + off;
#pragma unroll
    for (int i = 0; i < kOneItems; i++) {
        const int64_t v = tile[b + i + ((b + i) >> 4)];
        if (CF) note_items(big, cf, ncf, grain, t0 + b + i, run, v);
        tile[b + i + ((b + i) >> 4)] = run;
        run += v;
    }
    __syncthreads();
    if (CF) note_big(big, cf, ncf, grain);
    for (int i = threadIdx.x; i < kOneTile; i += kOneThreads) {
        const int64_t idx = t0 + i;
        if (idx < n) out[idx] = tile[i + (i >> 4)];
    }
}

// ------------------------------------------------------------------ radix sort
// Stable LSD radix sort of (key, a[, t]) triples, one kernel per digit.  The counts of the whole
// input, for every digit, come from one earlier read (count_digits, inside the kernel that
// produces the keys, or k_digit_count); a pass then finds each tile's place in every digit's run
// from the tiles before it (decoupled look-back: Merrill and Garland, "Single-pass parallel
// prefix scan with decoupled look-back", 2016; used for radix sorting by Adinets and Merrill,
// "Onesweep", 2022), so it reads and writes each triple once and nothing else of size n.  The
// passes it replaces read every key a second time for a histogram per tile and scanned
// 2^bits x tiles counters with three more kernels.
//
// A tile is 4096 keys, all of its loads in flight at once, so that three tiles per SM cover the
// memory's latency; each digit's run of the tile leaves shared memory as neighbouring
// addresses.  A pass moves 2.3 to 3.0 TB/s of its 2 x 12 bytes per key (1e7 keys, nine-bit
// digits: 93 to 106 us, 159 to 176 for both views at once; histogram, scan and scatter took 140
// to 180 per sort): 58 % of the LSU's wavefronts, for stores that reach four to eight runs each,
// and 55 % of the ALU, for a ballot per digit bit, are what bounds it.
constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 16;                       // per thread
constexpr int kSortTile = kSortThreads * kSortItems; // 4096

// lanes of `act` holding the same DB-bit digit: one ballot per bit (independent of one another,
// unlike the compare-and-vote loop behind __match_any_sync)
template <int DB>
__device__ __forceinline__ unsigned same_digit(uint32_t d, unsigned act) {
    unsigned m = act;
#pragma unroll
    for (int b = 0; b < DB; b++) {
        const bool bit = (d >> b) & 1u;
        const unsigned v = __ballot_sync(kFull, bit);
        m &= bit ? v : ~v;
    }
    return m;
}

// exclusive scan over the block of one value per thread (sm: one word per warp)
__device__ __forceinline__ uint32_t block_excl_scan_u32(uint32_t v, uint32_t* sm) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) sm[w] = inc;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int i = 0; i < kSortWarps; i++) before += i < w ? sm[i] : 0;
    return before + inc - v;
}

template <int TB> struct SortTime { using type = uint64_t; };
template <> struct SortTime<4> { using type = uint32_t; };

template <int TB, int DB>
constexpr size_t sort_smem_bytes() {
    constexpr size_t cnt = (size_t)2 * kSortWarps << DB, keys = (size_t)4 * kSortTile;
    return (size_t)kSortTile * (TB + 4 + 2) + (cnt > keys ? cnt : keys) + ((size_t)8 << DB);
}

// `bytes` bytes from src to the tile's place in shared memory without going through registers:
// 16 at a time where src allows it, else word by word
__device__ __forceinline__ void stage_tile(void* dst, const void* src, uint32_t bytes) {
    const uint32_t to = (uint32_t)__cvta_generic_to_shared(dst);
    const char* from = (const char*)src;
    if (((uintptr_t)from & 15) == 0) {
        for (uint32_t o = threadIdx.x * 16; o < bytes; o += kSortThreads * 16) {
            const uint32_t left = bytes - o < 16 ? bytes - o : 16;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to + o), "l"(from + o), "r"(left) : "memory");
        }
    } else {
        for (uint32_t o = threadIdx.x * 4; o < bytes; o += kSortThreads * 4)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to + o), "l"(from + o) : "memory");
    }
}

// One pass of one or two independent sorts (block b works on sort b mod J.jobs): warp w of a tile
// owns its items [512 w, 512 w + 512), 32 at a time in index order; ranks among equal digits are
// the lane order inside a ballot and the warp's running counters, then warps are offset by the
// counts of lower warps.  The payload waits in shared memory in input order while the keys are
// ranked (held in registers it spilled); the tile is put in digit order as (key, input slot).
template <int TB, int DB>
__global__ void __launch_bounds__(kSortThreads, TB == 8 ? 2 : 3) k_sort_pass(SortJobs J, int64_t n, int shift) {
    using T = typename SortTime<TB>::type;
    constexpr int ND = 1 << DB;
    constexpr int PER = ND > kSortThreads ? ND / kSortThreads : 1;   // digits per thread
    static_assert(ND <= kSortThreads || ND % kSortThreads == 0, "a thread's digits must not pass the last");
    extern __shared__ __align__(16) unsigned char sm_sort[];
    T* st = (T*)sm_sort;                                            // [TB ? tile : 0] input order
    uint32_t* sa = (uint32_t*)(sm_sort + (size_t)TB * kSortTile);   // [tile] input order
    uint32_t* gbase = sa + kSortTile;                        // [ND] output index of tile slot 0 of the digit
    uint32_t* tds = gbase + ND;                              // [ND] tile start of the digit
    uint16_t* slot = (uint16_t*)(tds + ND);                  // [tile] digit order -> input order
    uint32_t* sk = (uint32_t*)(slot + kSortTile);            // [tile] keys in digit order, once the
    uint16_t* cnt = (uint16_t*)sk;                           // [warps][ND] counters are done with
    __shared__ uint32_t s_tile, red[kSortWarps];
    const SortJob job = (J.jobs == 2 && (blockIdx.x & 1)) ? J.job[1] : J.job[0];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        const uint32_t ticket = atomicAdd(job.ticket, 1u);
        s_tile = gave_up(J.err) ? 0xffffffffu : ticket;
    }
    for (int i = threadIdx.x; i < kSortWarps * ND / 2; i += kSortThreads) ((uint32_t*)cnt)[i] = 0;
    __syncthreads();
    const int64_t tile = s_tile;
    const int64_t tbase = tile * kSortTile;
    if (tbase >= n) return;   // (also after an expired wait: an earlier pass may have left its lists unwritten)
    const int tn = (int)min((int64_t)kSortTile, n - tbase);
    const int wbase = w * (kSortItems * 32) + lane;
    uint32_t key[kSortItems], rank[kSortItems];
#pragma unroll
    for (int r = 0; r < kSortItems; r++) key[r] = wbase + r * 32 < tn ? __ldg(job.key_in + tbase + wbase + r * 32) : 0u;
    stage_tile(sa, job.a_in + tbase, 4u * (uint32_t)tn);
    if constexpr (TB != 0) stage_tile(st, (const T*)job.t_in + tbase, (uint32_t)TB * (uint32_t)tn);
    uint16_t* wc = cnt + w * ND;
#pragma unroll
    for (int r = 0; r < kSortItems; r++) {
        const bool ok = wbase + r * 32 < tn;
        const uint32_t d = (key[r] >> shift) & (ND - 1);
        const unsigned peers = same_digit<DB>(d, __ballot_sync(kFull, ok));
        const uint32_t c0 = wc[d];
        rank[r] = c0 + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
        if (ok && (peers >> lane) == 1u) wc[d] = (uint16_t)(c0 + __popc(peers));   // the highest peer
        __syncwarp();
    }
    __syncthreads();
    // per digit: the warps' offsets inside it and the tile's count, told to the tiles behind
    uint32_t tot[PER], sum = 0;
    uint32_t* words = job.words + tile * ND;
    const int d0 = threadIdx.x * PER;
    if (d0 < ND) {
#pragma unroll
        for (int x = 0; x < PER; x++) {
            uint32_t run = 0;
#pragma unroll
            for (int i = 0; i < kSortWarps; i++) {
                const uint32_t c = cnt[i * ND + d0 + x];
                cnt[i * ND + d0 + x] = (uint16_t)run;
                run += c;
            }
            tot[x] = run;
            sum += run;
            st_tile(words + d0 + x, tile == 0 ? (kTilePrefix | run) : run + 1);
        }
    }
    uint32_t at = block_excl_scan_u32(sum, red);
    if (d0 < ND) {
#pragma unroll
        for (int x = 0; x < PER; x++) {
            tds[d0 + x] = at;
            at += tot[x];
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; r++) {
        const uint32_t d = (key[r] >> shift) & (ND - 1);
        rank[r] += tds[d] + wc[d];
    }
    __syncthreads();   // the counters give way to the keys
#pragma unroll
    for (int r = 0; r < kSortItems; r++) {
        if (wbase + r * 32 < tn) {
            sk[rank[r]] = key[r];
            slot[rank[r]] = (uint16_t)(wbase + r * 32);
        }
    }
    // each digit's place in the output
    bool lost = false;
    if (d0 < ND) {
#pragma unroll
        for (int x = 0; x < PER; x++) {
            uint32_t before = 0;
            if (tile > 0) {
                if (!look_back(job.words + d0 + x, tile, ND, J.err, J.limit, before)) {
                    lost = true;
                    break;
                }
                st_tile(words + d0 + x, kTilePrefix | (before + tot[x]));
            }
            gbase[d0 + x] = job.base[d0 + x] + before - tds[d0 + x];
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (__syncthreads_or(lost)) return;   // a place is not known: the tile stays unwritten
    for (int i = threadIdx.x; i < tn; i += kSortThreads) {
        const uint32_t k = sk[i], o = slot[i];
        const int64_t pos = TM_CHK_IDX((int64_t)(uint32_t)(gbase[(k >> shift) & (ND - 1)] + (uint32_t)i), n, kChkSort);
        if (job.key_out) job.key_out[pos] = k;
        job.a_out[pos] = sa[o];
        if constexpr (TB != 0) ((T*)job.t_out)[pos] = st[o];
    }
}

// counts of every digit of every pass of `keys` (counts[pass][digit], zeroed before)
__global__ void k_digit_count(const uint32_t* __restrict__ keys, int64_t n, SortDigits D, uint32_t* __restrict__ counts) {
    extern __shared__ uint32_t sm_digits[];
    const int words = D.passes << D.db;
    for (int i = threadIdx.x; i < words; i += blockDim.x) sm_digits[i] = 0;
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        count_digits(sm_digits, D, keys[i]);
    __syncthreads();
    for (int i = threadIdx.x; i < words; i += blockDim.x)
        if (sm_digits[i]) atomicAdd(counts + i, sm_digits[i]);
}

// counts of each (sort, pass) -> the start of each digit's run, in place (one block each)
__global__ void __launch_bounds__(kSortThreads) k_digit_base(uint32_t* __restrict__ counts, int db) {
    __shared__ uint32_t red[kSortWarps];
    uint32_t* c = counts + ((size_t)blockIdx.x << db);
    const int per = max(1, (1 << db) / kSortThreads), d0 = threadIdx.x * per;
    uint32_t sum = 0;
    for (int x = 0; x < per; x++) sum += d0 + x < (1 << db) ? c[d0 + x] : 0;
    uint32_t at = block_excl_scan_u32(sum, red);
    for (int x = 0; x < per; x++)
        if (d0 + x < (1 << db)) {
            const uint32_t v = c[d0 + x];
            c[d0 + x] = at;
            at += v;
        }
}

// Polls after which a wait of the next launch expires; `ticket` numbers its tiles, zeroed before.
// The checked build can be told to leave tile 0 of a launch of several to nobody (check_expire): the
// tickets then start at one, the block with the last one finds no tile, and the others wait for a
// word that never comes.
#ifdef TM_CHECKED
std::atomic<int> g_expire{0};
int wait_limit(void* ticket, int64_t tiles, cudaStream_t st) {
    if (tiles < 2 || g_expire.load() <= 0 || g_expire.fetch_sub(1) != 1) return kSpinLimit;
    return cudaMemsetAsync(ticket, 1, 1, st) == cudaSuccess ? 1 << 10 : kSpinLimit;
}
#else
int wait_limit(void*, int64_t, cudaStream_t) { return kSpinLimit; }
#endif

template <int TB, int DB>
int sort_pass(SortJobs& J, int64_t n, int shift, cudaStream_t st) {
    {
        // the tile's shared memory exceeds the 48 KB default: allowed once per device
        static std::mutex mu;
        static bool done[64] = {};
        int dev = 0;
        TM_CUDA(cudaGetDevice(&dev));
        std::lock_guard<std::mutex> lk(mu);
        if (dev < 0 || dev >= 64 || !done[dev]) {
            TM_CUDA(cudaFuncSetAttribute(k_sort_pass<TB, DB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sort_smem_bytes<TB, DB>()));
            if (dev >= 0 && dev < 64) done[dev] = true;
        }
    }
    const int64_t tiles = (n + kSortTile - 1) / kSortTile, blocks = J.jobs * tiles;
    J.limit = wait_limit(J.job[0].ticket, tiles, st);
    k_sort_pass<TB, DB><<<(unsigned)blocks, kSortThreads, sort_smem_bytes<TB, DB>(), st>>>(J, n, shift);
    count_launch();
    TM_CUDA(cudaGetLastError());
    return TM_OK;
}

template <int TB>
int sort_pass_db(SortJobs& J, int64_t n, int shift, int db, cudaStream_t st) {
    switch (db) {
        case 5: return sort_pass<TB, 5>(J, n, shift, st);
        case 6: return sort_pass<TB, 6>(J, n, shift, st);
        case 7: return sort_pass<TB, 7>(J, n, shift, st);
        case 8: return sort_pass<TB, 8>(J, n, shift, st);
        case 9: return sort_pass<TB, 9>(J, n, shift, st);
        default: return sort_pass<TB, 10>(J, n, shift, st);
    }
}

}  // namespace

#ifdef TM_CHECKED
int check_expire(int nth) { return g_expire.exchange(nth); }
#endif

int scan_exclusive_i64(const int64_t* in, int64_t* out, int64_t n, int64_t* d_total,
                       cudaStream_t st) {
    if (n <= 0) {
        if (d_total) {
            k_set_i64<<<1, 1, 0, st>>>(d_total, 0); count_launch();
            TM_CUDA(cudaGetLastError());
        }
        return TM_OK;
    }
    if (n <= kScanTile) {
        k_scan_small<<<1, kScanThreads, 0, st>>>(in, out, n, d_total); count_launch();
        TM_CUDA(cudaGetLastError());
        return TM_OK;
    }
    int64_t ntiles = (n + kScanTile - 1) / kScanTile;
    int64_t* sums = nullptr;
    TM_CUDA(cudaMallocAsync((void**)&sums, sizeof(int64_t) * (size_t)ntiles * 2, st));
    int64_t* soffs = sums + ntiles;
    k_scan_tiles<<<(unsigned)ntiles, kScanThreads, 0, st>>>(in, out, n, sums); count_launch();
    int s1 = cudaGetLastError() == cudaSuccess ? TM_OK : TM_ECUDA;
    if (s1 == TM_OK) s1 = scan_exclusive_i64(sums, soffs, ntiles, d_total, st);
    if (s1 == TM_OK) {
        k_scan_add<<<(unsigned)ntiles, kScanThreads, 0, st>>>(out, n, soffs); count_launch();
        if (cudaGetLastError() != cudaSuccess) s1 = TM_ECUDA;
    }
    cudaFreeAsync(sums, st);
    if (s1 != TM_OK) set_error("scan launch failed");
    return s1;
}

int scan_exclusive_i64_ws(const int64_t* in, int64_t* out, int64_t n, int64_t* d_total,
                          int64_t* ws, int64_t ws_elems, cudaStream_t st) {
    // Same result as scan_exclusive_i64, with the per-tile sums in the
    // caller's workspace `ws` instead of a stream-ordered allocation.
    if (n <= 0) {
        if (d_total) {
            k_set_i64<<<1, 1, 0, st>>>(d_total, 0); count_launch();
            TM_CUDA(cudaGetLastError());
        }
        return TM_OK;
    }
    if (n <= kScanTile) {
        k_scan_small<<<1, kScanThreads, 0, st>>>(in, out, n, d_total); count_launch();
        TM_CUDA(cudaGetLastError());
        return TM_OK;
    }
    int64_t ntiles = (n + kScanTile - 1) / kScanTile;
    if (ntiles > kScanTile || 2 * ntiles > ws_elems) return TM_EINVAL;
    int64_t* sums = ws;
    int64_t* soffs = ws + ntiles;
    k_scan_tiles<<<(unsigned)ntiles, kScanThreads, 0, st>>>(in, out, n, sums); count_launch();
    k_scan_small<<<1, kScanThreads, 0, st>>>(sums, soffs, ntiles, d_total); count_launch();
    k_scan_add<<<(unsigned)ntiles, kScanThreads, 0, st>>>(out, n, soffs); count_launch();
    TM_CUDA(cudaGetLastError());
    return TM_OK;
}

int scan_lengths(const int32_t* in, int64_t* out, int64_t n_max, const int64_t* d_n, int64_t* d_total,
                 int64_t* cf, int64_t ncf, unsigned long long* words, uint32_t* err, int64_t* ws, int64_t ws_elems,
                 cudaStream_t st) {
    if (n_max <= 0) {
        k_set_i64<<<1, 1, 0, st>>>(d_total, 0); count_launch();
        TM_CUDA(cudaGetLastError());
        return TM_OK;
    }
    if (scan_once_words(n_max)) {
        const int64_t tiles = (n_max + kOneTile - 1) / kOneTile;
        const int limit = wait_limit(words, tiles, st);
        count_launch();
        TM_CUDA(launch_after(k_scan_once<int32_t, true>, dim3((unsigned)tiles), kOneThreads, 0, st,
                             in, out, n_max, d_n, d_total, words, err, limit, cf, ncf));
        return TM_OK;
    }
    int64_t ntiles = (n_max + kScanTile - 1) / kScanTile;
    int64_t need = 2 * ntiles + 2 * ((ntiles + kScanTile - 1) / kScanTile) + 2;
    int64_t* own = nullptr;
    if (!ws) {
        TM_CUDA(cudaMallocAsync((void**)&own, sizeof(int64_t) * (size_t)need, st));
        ws = own;
        ws_elems = need;
    }
    int rc = TM_OK;
    if (ws_elems < need || ntiles > (int64_t)kScanTile * kScanTile) rc = TM_EINVAL;   // caller's workspace too small
    if (rc == TM_OK) {
        int64_t* sums = ws;
        int64_t* soffs = ws + ntiles;
        k_len_reduce<<<(unsigned)ntiles, kScanThreads, 0, st>>>(in, n_max, d_n, sums); count_launch();
        if (cudaGetLastError() != cudaSuccess) rc = TM_ECUDA;
        if (rc == TM_OK) rc = scan_exclusive_i64_ws(sums, soffs, ntiles, d_total, ws + 2 * ntiles, need - 2 * ntiles, st);
        if (rc == TM_OK) {
            k_len_scan<<<(unsigned)ntiles, kScanThreads, 0, st>>>(in, out, n_max, d_n, soffs, cf, ncf); count_launch();
            if (cudaGetLastError() != cudaSuccess) rc = TM_ECUDA;
        }
    }
    if (own) cudaFreeAsync(own, st);
    if (rc != TM_OK) set_error("length scan failed");
    return rc;
}

int64_t scan_dn_ws_elems(int64_t n_max) {
    if (n_max <= kScanTile) return 0;
    int64_t ntiles = (n_max + kScanTile - 1) / kScanTile;
    return 2 * ntiles + 2 * ((ntiles + kScanTile - 1) / kScanTile) + 2;
}

size_t scan_once_words(int64_t n_max) {
    const int64_t tiles = (n_max + kOneTile - 1) / kOneTile;
    return n_max > 0 && tiles <= kOnePassTiles ? 8 + (size_t)tiles : 0;
}

int scan_once_i64(const int64_t* in, int64_t* out, int64_t n, int64_t* d_total, unsigned long long* words, uint32_t* err,
                  cudaStream_t st) {
    if (!scan_once_words(n)) return scan_exclusive_i64(in, out, n, d_total, st);
    const int64_t tiles = (n + kOneTile - 1) / kOneTile;
    const int limit = wait_limit(words, tiles, st);
    count_launch();
    TM_CUDA(launch_after(k_scan_once<int64_t, false>, dim3((unsigned)tiles), kOneThreads, 0, st,
                         in, out, n, nullptr, d_total, words, err, limit, nullptr, 0));
    return TM_OK;
}

// Digits of at most nine bits (ten when one pass then does): a tile's run of a digit is four keys
// at ten bits, 16 bytes in each array, 32 at seven, and the stores bound the pass.  Build of 1e8
// edges between 1e6 nodes (20 bits): two passes of ten 11.0 ms, three of seven 9.0, four of five
// 9.8; of 1e7 between 1e5 (17 bits): two of nine 0.90 ms, three of six 0.91.
SortDigits sort_digits(int bits) {
    SortDigits D;
    D.bits = std::max(bits, 1);
    D.passes = D.bits <= 10 ? 1 : (D.bits + 8) / 9;
    D.db = std::max(5, (D.bits + D.passes - 1) / D.passes);
    return D;
}

// words of one sort's scratch: tickets and tile words of every pass (zeroed by sort_clear)
static size_t sort_pass_words(int64_t n, const SortDigits& D) {
    const size_t ntiles = (size_t)((n + kSortTile - 1) / kSortTile);
    return ((ntiles << D.db) + 63) / 64 * 64 + 64;
}
size_t sort_ws_bytes(int64_t n, const SortDigits& D, int sorts, int counted) {
    return 4 * ((size_t)sorts * D.passes * sort_pass_words(n, D) + ((size_t)counted * D.passes << D.db) + 64);
}

SortWs sort_ws(void* mem, int64_t n, const SortDigits& D, int sorts, int counted) {
    SortWs W;
    W.D = D;
    W.n = n;
    W.err = (uint32_t*)mem;
    W.counts = W.err + 64;
    W.words = W.counts + ((size_t)counted * D.passes << D.db);
    W.counted = counted;
    W.bytes = sort_ws_bytes(n, D, sorts, counted);
    return W;
}

int sort_clear(const SortWs& W, cudaStream_t st) {
    TM_CUDA(cudaMemsetAsync(W.err, 0, W.bytes, st));
    return TM_OK;
}

int sort_bases(const SortWs& W, cudaStream_t st) {
    k_digit_base<<<(unsigned)(W.counted * W.D.passes), kSortThreads, 0, st>>>(W.counts, W.D.db);
    count_launch();
    TM_CUDA(cudaGetLastError());
    return TM_OK;
}

int sort_run(const SortWs& W, const SortIo* io, int sorts, int first, int tbytes, cudaStream_t st) {
    const size_t pw = sort_pass_words(W.n, W.D);
    for (int p = 0; p < W.D.passes; p++) {
        SortJobs J;
        J.jobs = sorts;
        J.err = W.err;
        for (int s = 0; s < sorts; s++) {
            const SortIo& x = io[s];
            // an odd number of passes still to come writes the final arrays, an even one the others
            const bool from_final = (W.D.passes - p) % 2 == 0, last = p + 1 == W.D.passes;
            SortJob& j = J.job[s];
            j.key_in = p == 0 ? x.key_in : from_final ? x.key_out : x.key_tmp;
            j.a_in = p == 0 ? x.a_in : from_final ? x.a_out : x.a_tmp;
            j.t_in = p == 0 ? x.t_in : from_final ? x.t_out : x.t_tmp;
            j.key_out = last && !x.keep_key ? nullptr : from_final ? x.key_tmp : x.key_out;
            j.a_out = from_final ? x.a_tmp : x.a_out;
            j.t_out = from_final ? x.t_tmp : x.t_out;
            uint32_t* w = W.words + pw * ((size_t)(first + s) * W.D.passes + p);
            j.ticket = w;
            j.words = w + 64;
            j.base = W.counts + (((size_t)x.counts * W.D.passes + p) << W.D.db);
        }
        const int shift = p * W.D.db;
        int rc;
        if (tbytes == 8) rc = sort_pass_db<8>(J, W.n, shift, W.D.db, st);
        else if (tbytes == 4) rc = sort_pass_db<4>(J, W.n, shift, W.D.db, st);
        else rc = sort_pass_db<0>(J, W.n, shift, W.D.db, st);
        if (rc != TM_OK) return rc;
    }
    return TM_OK;
}

int radix_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* keys_tmp, uint32_t* vals_tmp,
                     int64_t n, int bits, uint32_t* d_err, cudaStream_t st) {
    // Sorts (keys, vals) stably by the low `bits` bits of keys; the result ends
    // in keys/vals.  bits <= 32.
    if (n <= 1 || bits <= 0) return TM_OK;
    const SortDigits D = sort_digits(bits);
    void* mem = nullptr;
    TM_CUDA(cudaMallocAsync(&mem, sort_ws_bytes(n, D, 1, 1), st));
    SortWs W = sort_ws(mem, n, D, 1, 1);
    int rc = sort_clear(W, st);
    W.err = d_err;
    if (rc == TM_OK) {
        k_digit_count<<<(unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)sm_count() * 8), 256,
                        (size_t)4 * D.passes << D.db, st>>>(keys, n, D, W.counts);
        count_launch();
        if (cudaGetLastError() != cudaSuccess) rc = TM_ECUDA;
    }
    if (rc == TM_OK) rc = sort_bases(W, st);
    SortIo io;
    io.key_in = keys; io.a_in = vals; io.t_in = nullptr;
    // an even number of passes ends where it began, an odd one in the other arrays
    const bool even = D.passes % 2 == 0;
    io.key_out = even ? keys : keys_tmp; io.a_out = even ? vals : vals_tmp; io.t_out = nullptr;
    io.key_tmp = even ? keys_tmp : keys; io.a_tmp = even ? vals_tmp : vals; io.t_tmp = nullptr;
    io.counts = 0;
    io.keep_key = true;
    if (rc == TM_OK) rc = sort_run(W, &io, 1, 0, 0, st);
    if (rc == TM_OK && !even) {
        cudaError_t e = cudaMemcpyAsync(keys, keys_tmp, sizeof(uint32_t) * (size_t)n, cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(vals, vals_tmp, sizeof(uint32_t) * (size_t)n, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) rc = TM_ECUDA;
    }
    cudaFreeAsync(mem, st);
    if (rc != TM_OK) set_error("radix sort launch failed");
    return rc;
}

namespace {
std::mutex g_pool_mu;
bool g_pool_ready[64] = {};
cudaStream_t g_free_stream[64] = {};
}  // namespace

int pool_prepare(int dev) {
    if (dev < 0 || dev >= 64) return TM_OK;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (g_pool_ready[dev]) return TM_OK;
    // keep freed blocks of the device's default pool mapped, so that graphs and
    // batch scratch that come and go reuse memory instead of remapping it
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
        uint64_t keep = UINT64_MAX;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    }
    cudaStreamCreateWithFlags(&g_free_stream[dev], cudaStreamNonBlocking);
    cudaGetLastError();
    g_pool_ready[dev] = true;
    return TM_OK;
}

void pool_free(void* p, int dev) {
    if (!p) return;
    cudaStream_t s = (dev >= 0 && dev < 64) ? g_free_stream[dev] : nullptr;
    if (s) cudaFreeAsync(p, s);
    else cudaFree(p);
}

// Scratch arenas.  A large request to the stream-ordered pool costs about 0.3 ms of host
// time even when the pool keeps its memory (the device idles meanwhile), so the scratch
// of graph builds and batches comes from a few grow-only buffers per device instead.  A
// buffer is leased to one call at a time; the stream of the next lease waits on the event
// that the last holder recorded on its own stream at release.  A request that finds no
// free buffer is served by the pool.
namespace {
constexpr int kArenas = 4;
struct Arena {
    void* p = nullptr;
    size_t cap = 0;
    bool held = false;
    cudaEvent_t ev = nullptr;
    bool ev_set = false;
};
Arena g_arena[64][kArenas];
}  // namespace

int scratch_acquire(size_t bytes, cudaStream_t st, ScratchLease& L) {
    L = ScratchLease();
    int dev = 0;
    TM_CUDA(cudaGetDevice(&dev));
    L.dev = dev;
    if (dev >= 0 && dev < 64) {
        std::lock_guard<std::mutex> lk(g_pool_mu);
        int fit = -1, grow = -1;
        for (int i = 0; i < kArenas; i++) {
            const Arena& A = g_arena[dev][i];
            if (A.held) continue;
            if (A.cap >= bytes && (fit < 0 || A.cap < g_arena[dev][fit].cap)) fit = i;
            if (grow < 0 || A.cap > g_arena[dev][grow].cap) grow = i;
        }
        int i = fit >= 0 ? fit : grow;
        if (i >= 0) {
            Arena& A = g_arena[dev][i];
            cudaError_t e = cudaSuccess;
            if (!A.ev) e = cudaEventCreateWithFlags(&A.ev, cudaEventDisableTiming);
            if (e == cudaSuccess && A.ev_set) e = cudaStreamWaitEvent(st, A.ev, 0);
            if (e == cudaSuccess && A.cap < bytes) {
                if (A.p) cudaFreeAsync(A.p, st);
                A.p = nullptr;
                A.cap = 0;
                e = cudaMallocAsync(&A.p, bytes, st);
                if (e == cudaSuccess) A.cap = bytes;
                else A.p = nullptr;
            }
            if (e == cudaSuccess) {
                A.held = true;
                L.p = A.p;
                L.slot = i;
                return TM_OK;
            }
            cudaGetLastError();   // fall through to a pool block
        }
    }
    TM_CUDA(cudaMallocAsync(&L.p, bytes, st));
    return TM_OK;
}

void scratch_release(ScratchLease& L, cudaStream_t st) {
    if (!L.p) return;
    if (L.slot < 0) {
        cudaFreeAsync(L.p, st);
    } else {
        std::lock_guard<std::mutex> lk(g_pool_mu);
        Arena& A = g_arena[L.dev][L.slot];
        A.ev_set = cudaEventRecord(A.ev, st) == cudaSuccess;
        if (!A.ev_set) cudaGetLastError();
        A.held = false;
    }
    L = ScratchLease();
}

int pool_trim() {
    int dev = 0;
    TM_CUDA(cudaGetDevice(&dev));
    TM_CUDA(cudaDeviceSynchronize());
    if (dev >= 0 && dev < 64) {
        std::lock_guard<std::mutex> lk(g_pool_mu);
        for (int i = 0; i < kArenas; i++) {
            Arena& A = g_arena[dev][i];
            if (A.held || !A.p) continue;
            TM_CUDA(cudaFree(A.p));
            A.p = nullptr;
            A.cap = 0;
            A.ev_set = false;
        }
    }
    cudaMemPool_t pool;
    TM_CUDA(cudaDeviceGetDefaultMemPool(&pool, dev));
    TM_CUDA(cudaMemPoolTrimTo(pool, 0));
    return TM_OK;
}

int sm_count() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

}  // namespace tmo

namespace tmo {
TM_DEFINE_CHECK_WORD(check_word_prims)
}  // namespace tmo
