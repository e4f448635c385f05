// collect.cu -- the per-node search-and-collect of Alg. 2 (Section 3.5 iii): one
// warp per node searches the kNN graph, and a block per node selects its C
// nearest of the keys measured.
#include "search_kern.cuh"

namespace nsg {

struct CollectArgs {
    ExactRows rows;
    const int *knn;
    int K, W, nav, L, C, H, hshift, max_steps;
    int64_t v0, nv;
    int *cand_ids;
    float *cand_d2;
    int *cand_count, *status;
    uint64_t *log;  // [nv][log_cap] measured keys, cand_count their numbers
    int log_cap;
    int *seen;    // longest log (one that filled counts as twice what it holds), logs that filled
    int sel_cap;  // keys the selection has room for: no log is longer
    bool left;    // merged lists only for the nodes whose logs filled (cand_count -1)
};

// v's nearest neighbours in the kNN graph that its search has not seen (Alg.
// 2): their keys in s.keys, their count returned.
template <class D>
__device__ __forceinline__ int knn_row_keys(const CollectArgs &a, const D &dist, WarpSmem &s, int v) {
    const unsigned lane = lane_id();
    const int *row = a.knn + (int64_t)v * a.K;
    int m = 0;
    for (int b = 0; b < a.K; b += 32) {
        int slot = b + (int)lane;
        int w = slot < a.K ? __ldg(row + slot) : -1;
        bool fresh = w >= 0 && visit(s.hash, (uint32_t)a.H - 1, a.hshift, w);
        unsigned bal = __ballot_sync(NSG_FULL, fresh);
        if (fresh) s.ids[m + __popc(bal & lanemask_lt())] = w;
        m += __popc(bal);
    }
    __syncwarp();
    if (m > 0) dist(s.ids, m, s.keys);
    return m;
}

// Search-and-collect with the collect list kept sorted as the search goes: for
// searches that measure more keys than a log holds.
template <int G, int V, int U>
__device__ __forceinline__ void collect_body(const CollectArgs &a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const unsigned lane = lane_id();
    WarpSmem s = carve_warp_smem(smem + warp * warp_smem_bytes(a.L, a.W, a.C, a.H), a.L, a.W, a.C, a.H);
    const int64_t stride = (int64_t)gridDim.x * wpb;
    const uint32_t hmask = (uint32_t)a.H - 1;
    for (int64_t j = (int64_t)blockIdx.x * wpb + warp; j < a.nv; j += stride) {
        if (a.left && a.cand_count[j] >= 0) continue;
        const int v = (int)(a.v0 + j);
        DistF32<G, V, U> dist{{}, a.rows.base4, a.rows.dp4};
        dist.Q.load_row(a.rows.base4 + (int64_t)v * a.rows.dp4, a.rows.dp4);
        int csize = 0;
        SearchOut o = warp_alg1<KEYS_MERGE>(dist, GraphRef{a.knn, a.K}, a.nav, a.L, s, hmask, a.hshift,
                                             a.max_steps, v, a.C, csize);
        // Alg. 2: v's nearest neighbours in G join the candidates
        const int m = knn_row_keys(a, dist, s, v);
        if (m > 0) collect_merge(s, m, v, a.C, csize);
        // Alg. 2: sorted candidates, cut to C
        for (int t = lane; t < a.C; t += 32) {
            uint64_t e = t < csize ? s.clist[t] : KEY_INF;
            a.cand_ids[j * a.C + t] = t < csize ? kid(e) : -1;
            a.cand_d2[j * a.C + t] = t < csize ? kd2(e) : __int_as_float(0x7f800000);
        }
        if (lane == 0) {
            a.cand_count[j] = csize;
            if (a.status) a.status[j] = o.capped ? -4 : 0;
        }
        __syncwarp();
    }
}

// 20 warps per SM by the lists' shared memory: rows of up to 512 values on 80
// registers without spills (the compiler's own choice is 64 with some: 612 -> 705
// ms for 1,000,000 uniform rows of 128 values, K = 100, L = 60).  Wider rows: 5
// blocks of 128 threads up to 1,024 values (20,000 x 960, K = 40, L = 40, C = 200:
// 12.6 ms on the compiler's own budget, 11.0), 4 above (20,000 x 1,500: 24.1 free,
// with 12 warps on 160 registers; 21.9).
template <int G, int V, int U>
__global__ void __launch_bounds__(256, 3) collect_kernel(CollectArgs a) {
    collect_body<G, V, U>(a);
}
template <int G, int V, int U>
__global__ void __launch_bounds__(128, V > 8 ? 4 : 5) collect_wide_kernel(CollectArgs a) {
    collect_body<G, V, U>(a);
}
template <int G, int V, int U>
void (*collect_entry())(CollectArgs) {
    if constexpr (V > 4) return collect_wide_kernel<G, V, U>;
    else return collect_kernel<G, V, U>;
}

// Search-and-collect, first half: the keys are only appended to the node's log
// in global memory.  Merging every expansion's keys into a sorted list of C in
// shared memory was most of a search's instructions (moving up to C keys each
// time) and its list a third of the shared memory: 20 warps per SM, 24 to 32
// with the log.  Both halves together, FP32 rows: 100,000 SIFT-shaped rows (K =
// 100, L = 40, C = 500) 18.6 -> 14.0 ms, 150,000 DEEP-shaped (64, 60, 500)
// 7.2 -> 6.2 ms, 10,000 x 32 (20, 40, 200) 0.57 -> 0.41 ms.  Integer rows go
// through their exact 8-bit copy, a quarter of the bytes gathered and of the
// instructions per row: 14.0 -> 9.0 ms, 0.41 -> 0.37 ms.
template <int G, int V, int U, bool U8>
__device__ __forceinline__ void collect_log_body(const CollectArgs &a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const unsigned lane = lane_id();
    WarpSmem s = carve_warp_smem(smem + warp * warp_smem_bytes(a.L, a.W, 0, a.H, true), a.L, a.W, 0, a.H, true);
    const int64_t stride = (int64_t)gridDim.x * wpb;
    int longest = 0, filled = 0;
    for (int64_t j = (int64_t)blockIdx.x * wpb + warp; j < a.nv; j += stride) {
        const int v = (int)(a.v0 + j);
        KeyLog lg{a.log + j * a.log_cap, a.log_cap, 0, false};
        bool capped = false;
        with_row_dist<G, V, U, U8>(a.rows, v, [&](const auto &dist) {
            int none = 0;
            capped = warp_alg1<KEYS_LOG>(dist, GraphRef{a.knn, a.K}, a.nav, a.L, s, (uint32_t)a.H - 1, a.hshift,
                                         a.max_steps, v, 0, none, nullptr, 0, nullptr, nullptr, nullptr, &lg)
                         .capped;
            const int m = lg.full ? 0 : knn_row_keys(a, dist, s, v);
            if (m > 0) log_append(lg, s.keys, m, v);
        });
        longest = max(longest, lg.full ? 2 * a.log_cap : lg.count);
        filled += lg.full;
        if (lane == 0) {
            a.cand_count[j] = lg.full ? -1 : lg.count;
            if (a.status) a.status[j] = capped ? -4 : 0;
        }
        __syncwarp();
    }
    if (lane == 0 && longest > 0) {
        atomicMax(a.seen, longest);
        if (filled) atomicAdd(a.seen + 1, filled);
    }
}

// As for the searches: rows of up to 512 values at 64 registers and 32 warps
// per SM; wider ones as above.
template <int G, int V, int U, bool U8>
__global__ void __launch_bounds__(256, 4) collect_log_kernel(CollectArgs a) {
    collect_log_body<G, V, U, U8>(a);
}
template <int G, int V, int U, bool U8>
__global__ void __launch_bounds__(128, V > 8 ? 4 : 5) collect_log_wide_kernel(CollectArgs a) {
    collect_log_body<G, V, U, U8>(a);
}
template <int G, int V, int U>
void (*collect_log_entry(bool u8))(CollectArgs) {
    if constexpr (V > 4) return collect_log_wide_kernel<G, V, U, false>;  // no 8-bit copy at these widths
    else return u8 ? collect_log_kernel<G, V, U, true> : collect_log_kernel<G, V, U, false>;
}

// Search-and-collect, second half: one block per node cuts its log to the C
// smallest distinct keys, sorted; nodes whose logs filled are left alone.  Duplicates (nodes the visited set forgot)
// go through an exact hash of the ids; two 1024-bin passes over the distance
// bits (their order is the distances' order) find a bound that lets through
// the C smallest and hardly more; those are sorted in shared memory by a bitonic
// network whose first step of each merge pairs mirrored positions, so that
// every comparison puts the smaller key first and positions past the end need
// no padding.  Bound by the shared-memory passes of the hash and
// the sort; the log itself is read up to four times, from L2 after the first.
// Each thread owns at most 32 log entries, whose
// first-copy flags are one register.
constexpr int SEL_BINS = 1024;
constexpr int LOG_CAP_MAX = 16384;
constexpr int LOG_LONG = 12;  // run_collect_log

template <int NT>
struct SelectShared {
    int hist[SEL_BINS];
    unsigned part[3][NT / 32];
    int bin, before, count;
};

// Bin that holds the rank-th smallest (rank >= 1) of the histogram's entries,
// and how many lie in the bins before it, in sh.bin and sh.before.
template <int NT>
__device__ __forceinline__ void select_bin(SelectShared<NT> &sh, int rank) {
    constexpr int PER = SEL_BINS / NT;
    const int t = threadIdx.x, lane = t & 31;
    int h[PER], sum = 0;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
        h[e] = sh.hist[t * PER + e];
        sum += h[e];
    }
    int inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(NSG_FULL, inc, o);
        if (lane >= o) inc += x;
    }
    if (lane == 31) sh.part[0][t >> 5] = (unsigned)inc;
    __syncthreads();
    int before = inc - sum;
    for (int w = 0; w < (t >> 5); ++w) before += (int)sh.part[0][w];
#pragma unroll
    for (int e = 0; e < PER; ++e) {
        if (before < rank && rank <= before + h[e]) {
            sh.bin = t * PER + e;
            sh.before = before;
        }
        before += h[e];
    }
    __syncthreads();
}

// Sorts a[0..n) in shared memory.  A warp's 32 comparisons of one step cover
// 64 neighbouring positions while the pairs lie within 64, so only the longer
// steps need the block's barrier.
template <int NT>
__device__ __forceinline__ void block_sort(uint64_t *a, int n) {
    for (int k = 2; k < 2 * n; k <<= 1) {
        for (int h = k >> 1; h > 0; h >>= 1) {
            const bool flip = h == k >> 1;
            if (h > 32 || (h == 32 && !flip)) __syncthreads();
            else __syncwarp();
            for (int p = threadIdx.x;; p += NT) {
                const int t = p & (h - 1), i = 2 * (p - t) + t;
                if (i >= n) break;
                const int j = flip ? 2 * (p - t) + 2 * h - 1 - t : i + h;
                if (j < n) {
                    const uint64_t x = a[i], y = a[j];
                    if (y < x) {
                        a[i] = y;
                        a[j] = x;
                    }
                }
            }
        }
    }
    __syncthreads();
}

template <int NT>
__global__ void __launch_bounds__(NT) collect_select_kernel(CollectArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ SelectShared<NT> sh;
    uint32_t *hash = reinterpret_cast<uint32_t *>(smem);  // then the keys to sort
    uint64_t *keys = reinterpret_cast<uint64_t *>(smem);  // [sel_cap]
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t j = blockIdx.x;
    const uint64_t *log = a.log + j * a.log_cap;
    const int n = a.cand_count[j];
    if (n < 0) return;
    // table of more than n slots: the largest power of two that the keys' space
    // holds is more than sel_cap
    int hb = 6;
    while ((1 << hb) < 2 * n && (2 << hb) <= 2 * a.sel_cap) ++hb;
    const uint32_t hmask = (1u << hb) - 1;
    for (int i = t; i <= (int)hmask; i += NT) hash[i] = HASH_EMPTY;
    for (int i = t; i < SEL_BINS; i += NT) sh.hist[i] = 0;
    if (t == 0) sh.count = 0;
    __syncthreads();
    unsigned first = 0, lo = 0xffffffffu, hi = 0, fresh = 0;
    for (int e = 0, i = t; i < n; ++e, i += NT) {
        const uint64_t k = log[i];
        const uint32_t id = (uint32_t)k, b = (uint32_t)(k >> 32);
        uint32_t p = (id * 2654435761u) >> (32 - hb), old;
        while ((old = atomicCAS(hash + p, HASH_EMPTY, id)) != HASH_EMPTY && old != id) p = (p + 1) & hmask;
        if (old == HASH_EMPTY) {
            first |= 1u << e;
            ++fresh;
            lo = min(lo, b);
            hi = max(hi, b);
        }
    }
    lo = __reduce_min_sync(NSG_FULL, lo);
    hi = __reduce_max_sync(NSG_FULL, hi);
    fresh = __reduce_add_sync(NSG_FULL, fresh);
    if (lane == 0) {
        sh.part[0][warp] = lo;
        sh.part[1][warp] = hi;
        sh.part[2][warp] = fresh;
    }
    __syncthreads();
    fresh = 0;
    for (int w = 0; w < NT / 32; ++w) {
        lo = min(lo, sh.part[0][w]);
        hi = max(hi, sh.part[1][w]);
        fresh += sh.part[2][w];
    }
    __syncthreads();  // part is used again
    uint32_t lim = 0xffffffffu;  // distance bits up to which keys are sorted
    if ((int)fresh > a.C) {
        int rank = a.C;
        uint32_t from = lo, to = hi;
        for (int pass = 0; pass < 2; ++pass) {
            const int sft = max(0, 32 - __clz(to - from) - 10);  // (to - from) >> sft < SEL_BINS
            if (pass) {
                for (int i = t; i < SEL_BINS; i += NT) sh.hist[i] = 0;
                __syncthreads();
            }
            for (int e = 0, i = t; i < n; ++e, i += NT)
                if (first >> e & 1) {
                    const uint32_t b = (uint32_t)(log[i] >> 32);
                    if (b >= from && b <= to) atomicAdd(&sh.hist[(b - from) >> sft], 1);
                }
            __syncthreads();
            select_bin(sh, rank);
            const uint32_t base = from + ((uint32_t)sh.bin << sft), width = (1u << sft) - 1;
            lim = to - base < width ? to : base + width;
            rank -= sh.before;
            const int in_bin = sh.hist[sh.bin];
            // bins that split no further, or hold little past the rank
            if (sft == 0 || in_bin - rank <= 8) break;
            from = base;
            to = lim;
            __syncthreads();  // sh.hist, sh.bin read above
        }
    }
    for (int e = 0, i = t; i < n; ++e, i += NT)
        if (first >> e & 1) {
            const uint64_t k = log[i];
            if ((uint32_t)(k >> 32) <= lim) keys[atomicAdd(&sh.count, 1)] = k;
        }
    __syncthreads();
    block_sort<NT>(keys, sh.count);
    const int cnt = min(sh.count, a.C);
    for (int i = t; i < a.C; i += NT) {
        const uint64_t k = i < cnt ? keys[i] : KEY_INF;
        a.cand_ids[j * a.C + i] = i < cnt ? kid(k) : -1;
        a.cand_d2[j * a.C + i] = i < cnt ? kd2(k) : __int_as_float(0x7f800000);
    }
    if (t == 0) a.cand_count[j] = cnt;
}

// Whether logs are tried, and the keys a log is given before any was seen: a
// search of pool L measured 0.03 to 2.1 times L K keys.
static bool log_form(int L, int K) { return (int64_t)L * K <= 2 * LOG_CAP_MAX; }
static int first_log_cap(int L, int K) {
    return (int)std::min<int64_t>(std::max<int64_t>(3 * (int64_t)L * K, 1024), LOG_CAP_MAX);
}
// Nodes searched before the logs' length is known: a wave.
static int64_t first_nodes() { return (int64_t)sm_count() * 32; }

// The keys of a log for the search of nv nodes, 0: no log form.  512 MiB at
// most: allocating and freeing costs 0.8 us per MiB.
int64_t collect_log_keys(int L, int K, int64_t nv) {
    if (!log_form(L, K) || nv < 1) return 0;
    const int64_t budget = (int64_t)((size_t(512) << 20) / 8);
    const int64_t first = std::min(nv, first_nodes()) * first_log_cap(L, K);
    const int64_t rest = nv * std::max<int64_t>((int64_t)L * K / 2, 1024);
    return std::min(budget, std::max(first, rest));
}

template <int NT>
static cudaError_t launch_select_nt(const CollectArgs &a, cudaStream_t st) {
    const size_t smem = 8 * (size_t)a.sel_cap;
    cudaError_t e = cudaFuncSetAttribute(collect_select_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    collect_select_kernel<NT><<<(unsigned)a.nv, NT, smem, st>>>(a);
    return cudaGetLastError();
}

// `longest`: of the logs.  The keys' space is also the hash table's: half of
// the power of two that leaves the table at most 70 % full.
static cudaError_t launch_select(CollectArgs a, int longest, cudaStream_t st) {
    int half = 32;
    while (2 * half * 7 < longest * 10) half *= 2;
    a.sel_cap = std::min(std::max((longest + 31) & ~31, half), LOG_CAP_MAX);
    return a.sel_cap <= 32 * 128   ? launch_select_nt<128>(a, st)
           : a.sel_cap <= 32 * 256 ? launch_select_nt<256>(a, st)
                                   : launch_select_nt<512>(a, st);
}

static CollectArgs collect_args(const CollectLaunch &l) {
    CollectArgs a;
    a.rows = ExactRows{reinterpret_cast<const float4 *>(l.base), l.dp / 4, reinterpret_cast<const uint4 *>(l.u8.rows),
                       l.u8.chunks, l.u8.d, l.u8.lo};
    a.knn = l.knn;
    a.K = l.K;
    a.W = round32(l.K);
    a.nav = l.nav;
    a.L = l.L;
    a.C = l.C;
    a.H = l.hash_slots;
    a.hshift = 32 - log2i((unsigned)l.hash_slots);
    a.max_steps = l.max_steps;
    a.v0 = l.v0;
    a.nv = l.nv;
    a.cand_ids = l.cand_ids;
    a.cand_d2 = l.cand_d2;
    a.cand_count = l.cand_count;
    a.status = l.status;
    a.log = nullptr;
    a.log_cap = a.sel_cap = 0;
    a.seen = nullptr;
    a.left = false;
    return a;
}

static cudaError_t launch_merge(const CollectLaunch &l, bool left, cudaStream_t st) {
    if (l.nv <= 0) return cudaSuccess;
    CollectArgs a = collect_args(l);
    a.left = left;
    const size_t per_warp = warp_smem_bytes(a.L, a.W, a.C, a.H);
    cudaError_t err = cudaSuccess;
    NSG_DISPATCH_DP4(a.rows.dp4, {
        auto kern = collect_entry<G_, V_, U_>();
        int grid, wpb;
        size_t smem;
        err = config(kern, per_warp, 4, l.nv, &grid, &wpb, &smem);
        if (err == cudaSuccess) {
            kern<<<grid, wpb * 32, smem, st>>>(a);
            err = cudaGetLastError();
        }
    });
    return err;
}

cudaError_t launch_collect(const CollectLaunch &l, cudaStream_t st) { return launch_merge(l, false, st); }

// The nodes j0 .. j0 + nv - 1 of a launch.
static CollectLaunch part_of(const CollectLaunch &l, int64_t j0, int64_t nv) {
    CollectLaunch p = l;
    p.v0 = l.v0 + j0;
    p.nv = nv;
    p.cand_ids = l.cand_ids + j0 * l.C;
    p.cand_d2 = l.cand_d2 + j0 * l.C;
    p.cand_count = l.cand_count + j0;
    p.status = l.status != nullptr ? l.status + j0 : nullptr;
    return p;
}

// How many keys a search measures depends on the rows and their number (0.04 L K
// for 100,000 DEEP-shaped rows, K = 64, L = 60, 0.24 for a million; 0.26 and
// 0.73 for as many SIFT-shaped, 100 and 40; 1.2 for uniform ones) and hardly on
// the node.  So every slice of nodes is given logs by the longest of the slice
// before it (a quarter more), the first, a part of a wave, long ones; and the
// selection gets the shared memory that the slice's longest log needs.  The
// host reads that number between the two: ~15 us a slice.  A node whose log
// fills is searched again with a merged list.  What a log costs grows with every
// key, a merged list's cost only with the keys that enter, which C bounds: FP32
// searches that pass LOG_LONG C keys are merged (uniform rows of 128 values, K =
// 100, L = 60, C = 500, 1,000,000: 1,105 ms logged, 612 merged; 30,000, 6,600
// keys: equal; 20,000 x 960, K = L = 40, C = 200: 13.4 and 11.4), 8-bit ones
// as long as logs hold them are not (300,000 such rows: 103 ms logged, 156
// merged on FP32 rows).  Merged lists alone -> logs: 1,000,000 SIFT-shaped rows
// 295 -> 138 ms, 10,000,000 DEEP-shaped 2,614 -> 2,040 (with logs of L K / 2 that
// were compacted when full: 293 and 3,220).
cudaError_t run_collect_log(const CollectLaunch &l, CollectLog &log, cudaStream_t st) {
    CollectArgs a = collect_args(l);
    a.log = log.keys;
    a.seen = log.seen;
    // the visited set takes 1024 slots while 24 warps per SM still fit: the
    // 512 that fit 32 warps beside rows of 100 neighbours measure 62 % more
    // nodes (100,000 SIFT-shaped rows: 1,460 keys per node, collect 8.7 ms;
    // 1024 slots 900 keys, 7.3 ms; 2048 on 20 warps 7.3, on 16 8.3 ms; a
    // million: 256, 174 and 162 ms; 10 million DEEP-shaped 2,810 and 2,160)
    if (a.H < 1024 && 6 * (4 * warp_smem_bytes(a.L, a.W, 0, 1024, true) + 1024) <= smem_per_sm()) a.H = 1024;
    a.hshift = 32 - log2i((unsigned)a.H);
    const size_t per_warp = warp_smem_bytes(a.L, a.W, 0, a.H, true);
    cudaError_t err = cudaSuccess;
    for (int64_t j0 = 0; j0 < l.nv;) {
        a.log_cap = log.cap > 0 ? log.cap : log.first_cap > 0 ? log.first_cap : first_log_cap(l.L, l.K);
        a.log_cap = std::min(a.log_cap, LOG_CAP_MAX);
        // a few waves at most: one slice, with the logs there is room for
        const bool one = log.cap == 0 && log.first_cap == 0 && l.nv <= first_nodes() * 5 / 2 && log.size >= 1024 * l.nv;
        if (one) a.log_cap = (int)std::min<int64_t>(a.log_cap, log.size / l.nv);
        int64_t nodes = std::min(l.nv - j0, log.size / a.log_cap);
        if (log.cap == 0 && !one) nodes = std::min(nodes, first_nodes());
        if (log.merge || nodes < 1) return launch_merge(part_of(l, j0, l.nv - j0), false, st);
        const CollectLaunch slice = part_of(l, j0, nodes);
        a.v0 = slice.v0;
        a.nv = slice.nv;
        a.cand_ids = slice.cand_ids;
        a.cand_d2 = slice.cand_d2;
        a.cand_count = slice.cand_count;
        a.status = slice.status;
        if ((err = cudaMemsetAsync(a.seen, 0, 2 * sizeof(int), st)) != cudaSuccess) return err;
        NSG_DISPATCH_DP4(a.rows.dp4, {
            auto kern = collect_log_entry<G_, V_, U_>(a.rows.u8 != nullptr);
            int grid, wpb;
            size_t smem;
            err = config(kern, per_warp, 4, a.nv, &grid, &wpb, &smem);
            if (err == cudaSuccess) {
                kern<<<grid, wpb * 32, smem, st>>>(a);
                err = cudaGetLastError();
            }
        });
        int seen[2] = {0, 0};
        if (err == cudaSuccess) err = cudaMemcpyAsync(seen, a.seen, sizeof(seen), cudaMemcpyDeviceToHost, st);
        if (err == cudaSuccess) err = cudaStreamSynchronize(st);
        if (err == cudaSuccess) err = launch_select(a, std::min(seen[0], a.log_cap), st);
        if (err == cudaSuccess && seen[1] > 0) err = launch_merge(slice, true, st);
        if (err != cudaSuccess) return err;
        log.merge = (seen[1] == 0 || a.log_cap == LOG_CAP_MAX) &&
                    seen[0] > (a.rows.u8 != nullptr ? LOG_CAP_MAX : LOG_LONG * l.C);
        log.cap = std::min(std::max((seen[0] + seen[0] / 4 + l.K + 31) & ~31, 1024), LOG_CAP_MAX);
        j0 += nodes;
    }
    return err;
}

}  // namespace nsg
