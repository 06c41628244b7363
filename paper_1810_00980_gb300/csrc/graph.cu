// Graph ingest and adjacency build (temporal graph T and its static graph G,
// Section 2).  Everything after the input copy runs on the device: validation,
// normalisation t' = t - t_min (Algorithm 1 assumes times start at 0), three
// stable radix sorts that leave every adjacency segment in time order, and
// segment offsets found from the sorted keys.
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
// view's, row 1 the in view's
__global__ void k_offsets(const uint32_t* __restrict__ out_keys, const uint32_t* __restrict__ in_keys, int64_t m,
                          int32_t n, int64_t* __restrict__ out_off, int64_t* __restrict__ in_off) {
    const uint32_t* keys = blockIdx.y ? in_keys : out_keys;
    int64_t* off = blockIdx.y ? in_off : out_off;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= m;
         i += (int64_t)gridDim.x * blockDim.x) {
        int64_t prev = i == 0 ? -1 : (int64_t)keys[i - 1];
        int64_t cur = i == m ? (int64_t)n : (int64_t)keys[i];
        for (int64_t v = prev + 1; v <= cur; v++) off[TM_CHK_IDX(v, (int64_t)n + 1, kChkNode)] = i;
    }
}

// Pair index of every pair-view position and the start of every pair, in one pass: a pair starts
// where (source, destination) changes; ballots number the starts inside a warp's 512 positions, a
// block scan and the look-back over earlier tiles number them across the graph.  8 bytes read
// and 4 (8 more per pair) written per edge; it replaces a flag array of 8 bytes per edge, its
// three-kernel scan and two passes over both.
constexpr int kPairItems = 16;
constexpr int kPairTile = kThreads * kPairItems;
__global__ void __launch_bounds__(kThreads) k_pairs(const uint32_t* __restrict__ src, const uint32_t* __restrict__ dst, int64_t m,
                        int32_t* __restrict__ pair_pid, int64_t* __restrict__ pair_off, uint32_t* ticket,
                        uint32_t* words, uint32_t* err, int64_t* __restrict__ P) {
    __shared__ uint32_t s_tile, s_warp[kThreads / 32];
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
    __syncthreads();
    const int64_t tile = s_tile, tbase = tile * kPairTile;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t base = tbase + (int64_t)w * (kPairItems * 32) + lane;
    uint32_t s[kPairItems], d[kPairItems], heads[kPairItems];
#pragma unroll
    for (int r = 0; r < kPairItems; r++) {
        const int64_t i = base + r * 32;
        s[r] = i < m ? src[i] : 0;
        d[r] = i < m ? dst[i] : 0;
    }
    // the position before the warp's first; every other one is a neighbouring lane's or round's
    uint32_t ls = 0, ld = 0;
    if (lane == 0 && base > 0 && base < m) {
        ls = src[base - 1];
        ld = dst[base - 1];
    }
    uint32_t mine = 0;
#pragma unroll
    for (int r = 0; r < kPairItems; r++) {
        const int64_t i = base + r * 32;
        uint32_t ps = __shfl_up_sync(kFull, s[r], 1), pd = __shfl_up_sync(kFull, d[r], 1);
        if (lane == 0) {
            ps = ls;
            pd = ld;
        }
        heads[r] = __ballot_sync(kFull, i < m && (i == 0 || s[r] != ps || d[r] != pd));
        mine += __popc(heads[r]);
        ls = __shfl_sync(kFull, s[r], 31);
        ld = __shfl_sync(kFull, d[r], 31);
    }
    if (lane == 0) s_warp[w] = mine;
    __syncthreads();
    uint32_t total = 0, below = 0;
#pragma unroll
    for (int i = 0; i < kThreads / 32; i++) {
        below += i < w ? s_warp[i] : 0;
        total += s_warp[i];
    }
    if (threadIdx.x == 0) st_tile(words + tile, tile == 0 ? (kTilePrefix | total) : total + 1);
    const uint32_t before = look_back_block(words, tile, err);
    if (threadIdx.x == 0) {
        if (tile > 0) st_tile(words + tile, kTilePrefix | (before + total));
        if (tbase + kPairTile >= m) {   // the last tile knows how many pairs there are
            *P = (int64_t)before + total;
            pair_off[(int64_t)before + total] = m;
        }
    }
    uint32_t run = before + below;   // starts before this round's 32 positions
#pragma unroll
    for (int r = 0; r < kPairItems; r++) {
        const int64_t i = base + r * 32;
        const uint32_t pid = run + __popc(heads[r] & (0xffffffffu >> (31 - lane))) - 1;
        if (i < m) {
            pair_pid[i] = (int32_t)pid;
            if ((heads[r] >> lane) & 1u) pair_off[TM_CHK_IDX(pid, m, kChkSort)] = i;
        }
        run += __popc(heads[r]);
    }
}

// Open-addressing hash of the static edges: key (src << 32 | dst) -> the pair's
// time-sorted segment of pair_t, stored in the slot as (begin, length) so that a
// lookup is one 16-byte load.  Capacity is a power of two >= 2 P, so every probe
// chain ends at an empty slot.
__global__ void k_hash_insert(const int32_t* __restrict__ out_src, const int32_t* __restrict__ pair_dst,
                              const int64_t* __restrict__ pair_off, int64_t P,
                              unsigned long long* __restrict__ slots, unsigned long long mask,
                              uint32_t* __restrict__ filt, unsigned long long fmask) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < P;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t at = pair_off[p];   // (the out view and the pair view hold a source at the same positions)
        unsigned long long key = ((unsigned long long)(uint32_t)out_src[at] << 32) | (uint32_t)pair_dst[at];
        unsigned long long seg = ((unsigned long long)(uint32_t)(pair_off[p + 1] - at) << 32) | (uint32_t)at;
        unsigned long long h0 = sm64_mix(key);
        atomicOr(filt + ((h0 >> 32) & fmask), (1u << (h0 & 31)) | (1u << ((h0 >> 5) & 31)));
        unsigned long long h = h0 & mask;
        for (unsigned long long it = 0; it <= mask; it++) {
            unsigned long long prev = atomicCAS(&slots[2 * h], kHashEmpty, key);
            if (prev == kHashEmpty) {
                slots[2 * h + 1] = seg;
                break;
            }
            h = (h + 1) & mask;
        }
    }
}

int bits_for(int32_t n) {
    int b = 0;
    while (b < 31 && ((int64_t)1 << b) < (int64_t)n) b++;
    return b;
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
                 + 2 * sz_i32m + align256(8 * (M + 1)) + sz_tm;   // pair view (P <= m)
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
    int32_t* pair_pid = (int32_t*)take(sz_i32m);
    int64_t* pair_off = (int64_t*)take(align256(8 * (M + 1)));
    void* pair_t = take(sz_tm);

    GraphDev& G = g->dev;
    G.m = m; G.n = n; G.tbytes = tb; G.loops = 0;
    G.src = gs; G.dst = gd; G.t = gt;
    G.out_off = out_off; G.out_nbr = out_nbr; G.out_t = out_t;
    G.in_off = in_off; G.in_nbr = in_nbr; G.in_t = in_t;
    G.pair_dst = pair_dst; G.pair_off = pair_off; G.pair_t = pair_t;
    G.out_src = out_src; G.in_dst = in_dst; G.pair_pid = pair_pid;
    G.hslots = nullptr; G.hmask = 0;
    G.pfilt = nullptr; G.pfmask = 0;
    g->hash_block = nullptr;
    g->ex_own_block = nullptr;
    g->ex_rev_block = nullptr;

    int rc = TM_OK;
    if (m == 0) {
        TM_CUDA(cudaMemsetAsync(out_off, 0, 8 * nN, st));
        TM_CUDA(cudaMemsetAsync(in_off, 0, 8 * nN, st));
        TM_CUDA(cudaMemsetAsync(pair_off, 0, 8, st));
        TM_CUDA(cudaStreamSynchronize(st));
        g->P = 0;
        G.P = 0;
        *out = g;
        return TM_OK;
    }

    // ---- scratch: the lists between the passes of two sorts, the sorts' counts and tile words,
    // and the pair index's tile words.  The sorts' spare words hold the flags and the pair count.
    const SortDigits D = sort_digits(bits_for(n));
    const size_t set = 2 * sz_i32m + sz_tm, ws_bytes = align256(sort_ws_bytes(m, D, 3, 2));
    const size_t pair_tiles = (size_t)((m + kPairTile - 1) / kPairTile), pair_ws = align256(4 * (pair_tiles + 64));
    ScratchLease lease;
    int lrc = scratch_acquire(2 * set + ws_bytes + pair_ws, st, lease);
    if (lrc != TM_OK) {
        cudaStreamSynchronize(st);
        pool_free(g->block, dev);
        delete g;
        return lrc;
    }
    char* q = (char*)lease.p;
    const SortWs W = sort_ws(q, m, D, 3, 2);
    uint32_t* flags = W.err + 8;
    int64_t* dP = (int64_t*)(W.err + 16);
    uint32_t* pw = (uint32_t*)(q + ws_bytes);
    q += ws_bytes + pair_ws;
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
    if (rc == TM_OK && cudaMemsetAsync(pw, 0, pair_ws, st) != cudaSuccess) rc = TM_ECUDA;
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
        k_offsets<<<dim3(grid_for(m + 1), 2), kThreads, 0, st>>>((const uint32_t*)out_src, (const uint32_t*)in_dst, m, n, out_off, in_off);
        launched();
    }
    if (rc == TM_OK) {
        k_pairs<<<(unsigned)pair_tiles, kThreads, 0, st>>>((const uint32_t*)out_src, (const uint32_t*)pair_dst, m, pair_pid,
                                                           pair_off, pw, pw + 64, W.err, dP);
        launched();
    }
    int64_t P = 0;
    if (rc == TM_OK) {
        uint32_t h[24];   // error word, flags, pair count
        e = cudaMemcpyAsync(h, W.err, sizeof(h), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) rc = cuda_status(e, "graph build", __FILE__, __LINE__);
        else if (h[8]) { set_error("timestamps are not sorted non-decreasingly"); rc = TM_EUNSORTED; }
        else if (h[9]) { set_error("node id outside [0, n_nodes)"); rc = TM_ERANGE; }
        else if (h[0]) { set_error("graph build: a wait for an earlier tile expired"); rc = TM_ECUDA; }
        else {
            G.loops = h[11] ? 1 : 0;
            std::memcpy(&P, h + 16, 8);
        }
    }
    // pair hash: capacity the next power of two >= 2 P; then the pair filter: 8 bits per pair
    // (a power of two of 32-bit words), at most 32 MB so that it stays in L2
    if (rc == TM_OK) {
        unsigned long long cap = 2;
        while (cap < 2ull * (unsigned long long)P) cap <<= 1;
        unsigned long long fw = 1;
        while (fw < ((unsigned long long)P + 3) / 4 && fw < (1ull << 23)) fw <<= 1;
        e = cudaMallocAsync(&g->hash_block, 16 * cap + 4 * fw, st);
        if (e != cudaSuccess) rc = cuda_status(e, "cudaMalloc(pair hash)", __FILE__, __LINE__);
        if (rc == TM_OK) {
            g->bytes += (int64_t)(16 * cap + 4 * fw);
            G.hslots = (const unsigned long long*)g->hash_block;
            G.hmask = cap - 1;
            uint32_t* filt = (uint32_t*)((char*)g->hash_block + 16 * cap);
            G.pfilt = filt;
            G.pfmask = fw - 1;
            e = cudaMemsetAsync(g->hash_block, 0xff, 16 * cap, st);
            if (e == cudaSuccess) e = cudaMemsetAsync(filt, 0, 4 * fw, st);
            if (e == cudaSuccess) {
                k_hash_insert<<<grid_for(P), kThreads, 0, st>>>(out_src, pair_dst, pair_off, P,
                                                               (unsigned long long*)g->hash_block, cap - 1,
                                                               filt, fw - 1);
                count_launch();
                e = cudaGetLastError();
            }
            int ev1 = pe.mark(st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) rc = cuda_status(e, "pair hash build", __FILE__, __LINE__);
            if (rc == TM_OK && pe.on) store_profile_graph(pe.ms(ev0, ev1));
        }
    }
    scratch_release(lease, st);
    if (rc != TM_OK) {
        cudaStreamSynchronize(st);
        pool_free(g->block, dev);
        pool_free(g->hash_block, dev);
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
        int32_t pid = G.pair_pid[e];
        int64_t te = (int64_t)G.pair_t[e];
        if (!reverse) {
            int64_t pa = G.pair_off[pid];
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
