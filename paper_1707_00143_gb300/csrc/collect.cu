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

// Search-and-collect with the collect list kept sorted as the search goes: the
// general form, for searches that measure more keys than a log holds.
template <int G, int V, int U>
__global__ void __launch_bounds__(256) collect_kernel(CollectArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const unsigned lane = lane_id();
    WarpSmem s = carve_warp_smem(smem + warp * warp_smem_bytes(a.L, a.W, a.C, a.H), a.L, a.W, a.C, a.H);
    const int64_t stride = (int64_t)gridDim.x * wpb;
    const uint32_t hmask = (uint32_t)a.H - 1;
    for (int64_t j = (int64_t)blockIdx.x * wpb + warp; j < a.nv; j += stride) {
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

// Search-and-collect, first half: the keys are only appended to the node's log
// in global memory.  Merging every expansion's keys into a sorted list of C in
// shared memory was most of a search's instructions (moving up to C keys each
// time) and its list a third of the shared memory: 20 warps per SM, 32 with
// the log.  Both halves together, FP32 rows: 100,000 SIFT-shaped rows (K =
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
    for (int64_t j = (int64_t)blockIdx.x * wpb + warp; j < a.nv; j += stride) {
        const int v = (int)(a.v0 + j);
        KeyLog lg{a.log + j * a.log_cap, a.log_cap, a.C, 0, ~0ull};
        bool capped = false;
        with_row_dist<G, V, U, U8>(a.rows, v, [&](const auto &dist) {
            int none = 0;
            capped = warp_alg1<KEYS_LOG>(dist, GraphRef{a.knn, a.K}, a.nav, a.L, s, (uint32_t)a.H - 1, a.hshift,
                                         a.max_steps, v, 0, none, nullptr, 0, nullptr, nullptr, nullptr, &lg)
                         .capped;
            const int m = knn_row_keys(a, dist, s, v);
            if (m > 0) log_append(lg, s.keys, m, v);
        });
        if (lane == 0) {
            a.cand_count[j] = lg.count;
            if (a.status) a.status[j] = capped ? -4 : 0;
        }
        __syncwarp();
    }
}

// As for the searches: rows of up to 512 values at 64 registers and 32 warps
// per SM, wider ones on the compiler's own budget.
template <int G, int V, int U, bool U8>
__global__ void __launch_bounds__(256, 4) collect_log_kernel(CollectArgs a) {
    collect_log_body<G, V, U, U8>(a);
}
template <int G, int V, int U, bool U8>
__global__ void __launch_bounds__(256) collect_log_wide_kernel(CollectArgs a) {
    collect_log_body<G, V, U, U8>(a);
}
template <int G, int V, int U>
void (*collect_log_entry(bool u8))(CollectArgs) {
    if constexpr (V > 4) return collect_log_wide_kernel<G, V, U, false>;  // no 8-bit copy at these widths
    else return u8 ? collect_log_kernel<G, V, U, true> : collect_log_kernel<G, V, U, false>;
}

// Search-and-collect, second half: one block per node cuts its log to the C
// smallest distinct keys, sorted.  Duplicates (nodes the visited set forgot)
// go through an exact hash of the ids; two 1024-bin passes over the distance
// bits (their order is the distances' order) find a bound that lets through
// the C smallest and hardly more; those are sorted in shared memory by the
// network of log_compact.  Bound by the shared-memory passes of the hash and
// the sort; the log itself is read up to four times, from L2 after the first.
// Each thread owns at most 32 log entries, whose
// first-copy flags are one register.
constexpr int SEL_BINS = 1024;
constexpr int LOG_CAP_MAX = 16384;

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
    uint64_t *keys = reinterpret_cast<uint64_t *>(smem);  // [log_cap]
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t j = blockIdx.x;
    const uint64_t *log = a.log + j * a.log_cap;
    const int n = a.cand_count[j];
    // table of more than n slots: the largest power of two that the keys' space
    // holds is more than log_cap
    int hb = 6;
    while ((1 << hb) < 2 * n && (2 << hb) <= 2 * a.log_cap) ++hb;
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

// Log entries per node.  A search of pool L expands little more than L nodes
// and finds less than half of their K neighbours new (512 visited slots, most
// of any node: 1,643 keys of L K = 4,000 on 100,000 SIFT-shaped rows, 288 of
// 3,840 DEEP-shaped, 376 of 800 on 10,000 x 32); a log that fills all the same
// is compacted in place, so it holds two lists and a row.
// 0: such a log would pass the selection's limit, the lists are merged instead.
int collect_log_cap(int L, int K, int C) {
    const int64_t cap = std::max<int64_t>(std::max<int64_t>((int64_t)L * K / 2, 2 * (int64_t)C + K), 1024);
    return cap <= LOG_CAP_MAX ? (int)((cap + 31) & ~31) : 0;
}

template <int NT>
static cudaError_t launch_select_nt(const CollectArgs &a, cudaStream_t st) {
    const size_t smem = 8 * (size_t)a.log_cap;
    cudaError_t e = cudaFuncSetAttribute(collect_select_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    collect_select_kernel<NT><<<(unsigned)a.nv, NT, smem, st>>>(a);
    return cudaGetLastError();
}

static cudaError_t launch_select(const CollectArgs &a, cudaStream_t st) {
    return a.log_cap <= 32 * 128   ? launch_select_nt<128>(a, st)
           : a.log_cap <= 32 * 256 ? launch_select_nt<256>(a, st)
                                   : launch_select_nt<512>(a, st);
}

cudaError_t launch_collect(const CollectLaunch &l, cudaStream_t st) {
    if (l.nv <= 0) return cudaSuccess;
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
    cudaError_t err = cudaSuccess;
    a.log = l.log;
    a.log_cap = collect_log_cap(l.L, l.K, l.C);
    if (a.log != nullptr && a.log_cap > 0 && l.log_nodes > 0) {
        // the visited set takes 1024 slots while 24 warps per SM still fit: the
        // 512 that fit 32 warps beside rows of 100 neighbours measure 62 % more
        // nodes (100,000 SIFT-shaped rows: 1,460 keys per node, collect 8.7 ms;
        // 1024 slots 900 keys, 7.3 ms; 2048 on 20 warps 7.3, on 16 8.3 ms)
        if (a.H < 1024 && 6 * (4 * warp_smem_bytes(a.L, a.W, 0, 1024, true) + 1024) <= smem_per_sm()) a.H = 1024;
        a.hshift = 32 - log2i((unsigned)a.H);
        const size_t per_warp = warp_smem_bytes(a.L, a.W, 0, a.H, true);
        for (int64_t j0 = 0; j0 < l.nv && err == cudaSuccess; j0 += l.log_nodes) {
            a.v0 = l.v0 + j0;
            a.nv = std::min<int64_t>(l.log_nodes, l.nv - j0);
            a.cand_ids = l.cand_ids + j0 * l.C;
            a.cand_d2 = l.cand_d2 + j0 * l.C;
            a.cand_count = l.cand_count + j0;
            a.status = l.status != nullptr ? l.status + j0 : nullptr;
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
            if (err == cudaSuccess) err = launch_select(a, st);
        }
        return err;
    }
    const size_t per_warp = warp_smem_bytes(a.L, a.W, a.C, a.H);
    NSG_DISPATCH_DP4(a.rows.dp4, {
        auto kern = collect_kernel<G_, V_, U_>;
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

}  // namespace nsg
