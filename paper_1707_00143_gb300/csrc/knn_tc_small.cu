// knn_tc_small.cu -- the tensor-core kNN of knn_tc.cu for few base tiles: the same
// answer by a CTA per 128 query rows whose four epilogue warps scan and merge
// by themselves.  With few tiles most columns are candidates, so merging is
// the work and there is little scan to hide it behind; the pre-pass, the rings
// and the splits' lists then cost more than they save.  The rule that
// chooses is in knn_rule.h, with both sides' times.
//
// CTA = 6 warps: warp 0 issues TMA (the 128 x d query tile once, then a ring
// of base tiles), warp 1 owns TMEM and issues the MMAs into two accumulator
// buffers, warps 2-5 are the epilogue: thread r holds query row r's running
// top-k.  A base column j enters row r's candidate buffer only when
// |x_j|^2 - 2 q.x_j < (current k-th distance) - |q|^2; the common case costs
// one FMA and one min per element (a group of 16 columns is tested through its
// minimum).  Columns arrive in increasing id, so a strict comparison on the
// distance alone implements the (distance, id) order.  Buffers of 48+ keys are
// merged warp-cooperatively into the row's sorted list, which lives in the
// output arrays.
#include <algorithm>

#include "common.cuh"
#include "knn_tc.cuh"
#include "tc_ptx.cuh"

namespace nsg {

namespace {

constexpr int TC_M = 128;       // query rows per CTA (TMEM lanes)
constexpr int TC_N = 128;       // base rows per tile (accumulator columns)
constexpr int TC_BOXK = 64;     // bf16 elements per 128-byte swizzle atom
constexpr int TC_BUF = 64;      // candidate buffer per row
constexpr int TC_MERGE_AT = 48; // merge when a buffer holds this many (+ 16 per test < 64)
constexpr int TC_THREADS = 192;
constexpr int TC_MAXK = 256;

struct TcArgs {
    const float *qn;  // [m] squared norms of the query rows
    const float *xn;  // [ntiles * 128] squared norms of the base rows
    int64_t m, n, q0;
    int self_join, KL;
    int t0, t1;       // base tiles [t0, t1) of this launch (one chunk of the base)
    int first, last;  // first chunk: lists start empty; last chunk: pad short lists
    int kb;  // 64-wide K chunks per row (streaming form)
    int *ids;
    float *d2;
    int *lsz;  // [m] list sizes carried between chunks
    int *err;
};

// DK = 64 or 128: the 128-row query tile stays in shared memory and a stage
// holds one base tile.  DK = 0: rows wider than 128 values; a stage holds one
// 64-wide K chunk of both the query tile and the base tile (16 KB each), and
// a tile takes dk/64 stages.
template <int DK>
struct TcCfg {
    static constexpr int KB = DK / TC_BOXK;                     // swizzle atoms along K (resident form)
    static constexpr int A_BYTES = TC_M * DK * 2;
    static constexpr int B_BYTES = DK ? TC_N * DK * 2 : 2 * TC_N * 128;  // one pipeline stage
    static constexpr int NS = DK == 64 ? 7 : (DK == 128 ? 3 : 4);       // stages
    static constexpr int OFF_B = A_BYTES;
    static constexpr int OFF_BUF = OFF_B + NS * B_BYTES;
    static constexpr int OFF_WARP = OFF_BUF + TC_M * TC_BUF * 8;
    // per epilogue warp: merge list, sorted buffer, base norms, k-th slot, and
    // 16 values per lane for the insertion path (column-major, conflict-free)
    static constexpr int WARP_BYTES = TC_MAXK * 8 + TC_BUF * 8 + TC_N * 4 + 16 + 16 * 32 * 4;
    static constexpr int OFF_BAR = OFF_WARP + 4 * WARP_BYTES;
    static constexpr int NBAR = 2 * NS + 6;  // a_full, b_full[NS], b_empty[NS], acc_full[2], acc_empty[2], drain
    static constexpr int SMEM = OFF_BAR + NBAR * 8 + 16 + 1024;  // + alignment slack
};

// Bitonic sort of 64 keys held two per lane (index lane and lane + 32), ascending.
__device__ __forceinline__ void bitonic64(uint64_t &a, uint64_t &b, unsigned lane) {
#pragma unroll
    for (int k = 2; k <= 64; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j == 32) {  // partner in the same lane: index lane vs lane + 32 (k = 64: ascending)
                const uint64_t mn = a < b ? a : b, mx = a < b ? b : a;
                a = mn;
                b = mx;
            } else {
                const uint64_t oa = __shfl_xor_sync(NSG_FULL, a, j), ob = __shfl_xor_sync(NSG_FULL, b, j);
                const bool lower = (lane & j) == 0;
                const bool up_a = (lane & k) == 0, up_b = ((lane + 32) & k) == 0;
                const uint64_t mna = oa < a ? oa : a, mxa = oa < a ? a : oa;
                const uint64_t mnb = ob < b ? ob : b, mxb = ob < b ? b : ob;
                a = (lower == up_a) ? mna : mxa;
                b = (lower == up_b) ? mnb : mxb;
            }
        }
    }
}

__device__ __forceinline__ int count_less(const uint64_t *a, int len, uint64_t key) {
    int lo = 0, hi = len;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (a[mid] < key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Merge row `src`'s buffer (c <= 63 keys) into its sorted list of s keys
// (output arrays, capacity KL), warp-cooperatively: the list is read once
// (all loads issued before use), the buffer sorted, and every key written to
// its rank in the union.
__device__ __noinline__ void merge_row(int src, int row_local, int64_t row_g, int &cnt, int &lsize,
                                       float &thrp, float qn_r, const uint64_t *bufs, uint64_t *ls,
                                       uint64_t *sb, uint64_t *thr_slot, int *ids, float *d2, int KL) {
    const unsigned lane = lane_id();
    const int c = __shfl_sync(NSG_FULL, cnt, src);
    const int s = __shfl_sync(NSG_FULL, lsize, src);
    const int rl = __shfl_sync(NSG_FULL, row_local, src);
    const int64_t rg = __shfl_sync(NSG_FULL, row_g, src);
    int *oid = ids + rg * KL;
    float *od = d2 + rg * KL;
    float lv[TC_MAXK / 32];
    int li[TC_MAXK / 32];
#pragma unroll
    for (int t = 0; t < TC_MAXK / 32; ++t) {
        const int i = t * 32 + (int)lane;
        if (i < s) {
            lv[t] = od[i];
            li[t] = oid[i];
        }
    }
    uint64_t a = (int)lane < c ? bufs[rl * TC_BUF + lane] : ~0ull;
    uint64_t b = (int)lane + 32 < c ? bufs[rl * TC_BUF + 32 + lane] : ~0ull;
    bitonic64(a, b, lane);
    sb[lane] = a;
    sb[lane + 32] = b;
#pragma unroll
    for (int t = 0; t < TC_MAXK / 32; ++t) {
        const int i = t * 32 + (int)lane;
        if (i < s) ls[i] = make_key(lv[t], li[t]);
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < TC_MAXK / 32; ++t) {
        const int i = t * 32 + (int)lane;
        if (i < s) {
            const uint64_t key = ls[i];
            const int p = i + count_less(sb, c, key);
            if (p < KL) {
                od[p] = kd2(key);
                oid[p] = kid(key);
                if (p == KL - 1) *thr_slot = key;
            }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = (int)lane + 32 * h;
        const uint64_t key = h ? b : a;
        if (j < c) {
            const int p = j + count_less(ls, s, key);
            if (p < KL) {
                od[p] = kd2(key);
                oid[p] = kid(key);
                if (p == KL - 1) *thr_slot = key;
            }
        }
    }
    __syncwarp();
    if ((int)lane == src) {
        cnt = 0;
        lsize = s + c < KL ? s + c : KL;
        if (lsize == KL) thrp = kd2(*thr_slot) - qn_r;
    }
    __syncwarp();
}

template <int DK>
__global__ void __launch_bounds__(TC_THREADS, 1)
    knn_tc_small_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, TcArgs a) {
    using Cfg = TcCfg<DK>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char *sA = smem;
    unsigned char *sB = smem + Cfg::OFF_B;
    uint64_t *bufs = reinterpret_cast<uint64_t *>(smem + Cfg::OFF_BUF);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + Cfg::OFF_BAR);
    uint64_t *a_full = bars;
    uint64_t *b_full = bars + 1;
    uint64_t *b_empty = bars + 1 + Cfg::NS;
    uint64_t *acc_full = bars + 1 + 2 * Cfg::NS;
    uint64_t *acc_empty = acc_full + 2;
    uint64_t *drain = acc_empty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + Cfg::NBAR);
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile int *gerr = a.err;

    const int warp = threadIdx.x >> 5;
    const unsigned lane = lane_id();
    const int64_t row0 = (int64_t)blockIdx.x * TC_M;

    if (threadIdx.x == 0) {
        tc::mbar_init(a_full, 1);
        for (int s = 0; s < Cfg::NS; ++s) {
            tc::mbar_init(b_full + s, 1);
            tc::mbar_init(b_empty + s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(acc_full + b, 1);
            tc::mbar_init(acc_empty + b, 4);
        }
        tc::mbar_init(drain, 1);
        *abort = *gerr ? 1 : 0;  // another CTA already failed: do nothing
        tc::fence_barrier_init();
        tc::prefetch_tmap(&tmA);
        tc::prefetch_tmap(&tmB);
    }
    if (warp == 1) {
        tc::tmem_alloc(tmem_slot, 2 * TC_N);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    const bool skip = *abort != 0;  // uniform: read after the barrier

    if (skip) {
        // nothing issued; fall through to TMEM release
    } else if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            if (DK) {
                tc::mbar_expect_tx(a_full, Cfg::A_BYTES);
                for (int kb = 0; kb < Cfg::KB; ++kb)
                    tc::tma_load_2d(sA + kb * (TC_M * 128), &tmA, a_full, kb * TC_BOXK, (int)row0);
            }
            const int per_tile = DK ? 1 : a.kb;  // stages per tile
            const int nt = a.t1 - a.t0;
            int issued = 0;
            for (int c = 0; c < nt * per_tile; ++c) {
                const int s = c % Cfg::NS, tl = c / per_tile, kc = c - tl * per_tile, t = a.t0 + tl;
                if (!tc::mbar_wait(b_empty + s, ((c / Cfg::NS) & 1) ^ 1, abort, gerr)) break;
                tc::mbar_expect_tx(b_full + s, Cfg::B_BYTES);
                unsigned char *dst = sB + s * Cfg::B_BYTES;
                if (DK) {
                    for (int kb = 0; kb < Cfg::KB; ++kb)
                        tc::tma_load_2d(dst + kb * (TC_N * 128), &tmB, b_full + s, kb * TC_BOXK, t * TC_N);
                } else {
                    tc::tma_load_2d(dst, &tmA, b_full + s, kc * TC_BOXK, (int)row0);
                    tc::tma_load_2d(dst + TC_M * 128, &tmB, b_full + s, kc * TC_BOXK, t * TC_N);
                }
                issued = c + 1;
            }
            if (*abort) {
                // drain: wait (bounded) for the copies still in flight
                volatile int local = 0;
                if (DK) tc::mbar_wait(a_full, 0, &local, nullptr);
                for (int c = issued - Cfg::NS < 0 ? 0 : issued - Cfg::NS; c < issued; ++c) {
                    local = 0;
                    tc::mbar_wait(b_full + c % Cfg::NS, (c / Cfg::NS) & 1, &local, nullptr);
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            constexpr uint32_t idesc = tc::idesc_bf16_f32(TC_M, TC_N);
            const uint32_t a_base = tc::smem_u32(sA), b_base = tc::smem_u32(sB);
            bool ok = DK ? tc::mbar_wait(a_full, 0, abort, gerr) : true;
            const int per_tile = DK ? 1 : a.kb;
            int c = 0;
            for (int t = 0; ok && t < a.t1 - a.t0; ++t) {  // local tile index
                const int buf = t & 1;
                if (!tc::mbar_wait(acc_empty + buf, ((t >> 1) & 1) ^ 1, abort, gerr)) break;
                tc::fence_after_sync();
                for (int kc = 0; ok && kc < per_tile; ++kc, ++c) {
                    const int s = c % Cfg::NS;
                    if (!tc::mbar_wait(b_full + s, (c / Cfg::NS) & 1, abort, gerr)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after_sync();
                    if (DK) {
#pragma unroll
                        for (int kk = 0; kk < (DK ? DK : 64) / 16; ++kk) {
                            const uint32_t koff = (kk >> 2) * (TC_M * 128) + (kk & 3) * 32;
                            const uint32_t boff = s * Cfg::B_BYTES + (kk >> 2) * (TC_N * 128) + (kk & 3) * 32;
                            tc::mma_bf16(tmem + buf * TC_N, tc::sdesc_sw128(a_base + koff),
                                         tc::sdesc_sw128(b_base + boff), idesc, kk > 0 ? 1u : 0u);
                        }
                    } else {
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            const uint32_t st = b_base + s * Cfg::B_BYTES + kk * 32;
                            tc::mma_bf16(tmem + buf * TC_N, tc::sdesc_sw128(st), tc::sdesc_sw128(st + TC_M * 128),
                                         idesc, (kc > 0 || kk > 0) ? 1u : 0u);
                        }
                    }
                    tc::mma_commit(b_empty + s);
                }
                if (!ok) break;
                tc::mma_commit(acc_full + buf);
            }
            // every MMA issued so far has completed before TMEM is released
            tc::mma_commit(drain);
            volatile int local = 0;
            tc::mbar_wait(drain, 0, &local, nullptr);
        }
    } else {
        // ---------------- epilogue: warps 2..5 ----------------
        const int q = warp & 3;  // TMEM lane quadrant of this warp
        const int ew = warp - 2;
        unsigned char *wsm = smem + Cfg::OFF_WARP + ew * Cfg::WARP_BYTES;
        uint64_t *ls = reinterpret_cast<uint64_t *>(wsm);
        uint64_t *sb = ls + TC_MAXK;
        float *xs = reinterpret_cast<float *>(sb + TC_BUF);
        uint64_t *thr_slot = reinterpret_cast<uint64_t *>(xs + TC_N);
        float *tvs = reinterpret_cast<float *>(thr_slot + 2);  // [16][32]
        const int row_local = q * 32 + lane;
        const int64_t row_g = row0 + row_local;
        const bool valid = row_g < a.m;
        const float qn_r = valid ? a.qn[row_g] : 0.0f;
        const int64_t self_id = a.self_join ? a.q0 + row_g : -1;
        uint64_t *mybuf = bufs + row_local * TC_BUF;
        // the row's list (size and k-th key) carried over from earlier chunks;
        // a row past the end takes nothing: its threshold is -inf
        int cnt = 0, lsize = valid && !a.first ? a.lsz[row_g] : 0;
        float thrp = __int_as_float(valid ? 0x7f800000 : 0xff800000);
        if (valid && lsize == a.KL) thrp = a.d2[row_g * a.KL + a.KL - 1] - qn_r;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
        bool ok = true;
        const float4 *xn4 = reinterpret_cast<const float4 *>(a.xn);
        float4 xnext = __ldg(xn4 + (int64_t)a.t0 * (TC_N / 4) + lane);  // norms one tile ahead
        for (int tl = 0; tl < a.t1 - a.t0; ++tl) {
            const int buf = tl & 1, t = a.t0 + tl;
            const int64_t col0 = (int64_t)t * TC_N;
            // columns jj < lim exist; jj == self_local is the row itself
            const int lim = a.n - col0 < TC_N ? (int)(a.n - col0) : TC_N;
            const int self_local = self_id >= col0 && self_id < col0 + TC_N ? (int)(self_id - col0) : -1;
            __syncwarp();
            reinterpret_cast<float4 *>(xs)[lane] = xnext;
            if (t + 1 < a.t1) xnext = __ldg(xn4 + (int64_t)(t + 1) * (TC_N / 4) + lane);
            __syncwarp();
            const bool got = tc::mbar_wait(acc_full + buf, (tl >> 1) & 1, abort, gerr);
            if (!__all_sync(NSG_FULL, got)) {  // warp-uniform before the .sync.aligned TMEM loads
                ok = false;
                break;
            }
            tc::fence_after_sync();
#pragma unroll 1
            for (int c = 0; c < TC_N / 32; ++c) {
                uint32_t v[32];
                tc::tmem_ld32_wait(tq + buf * TC_N + c * 32, v);
                if (c == TC_N / 32 - 1) {
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(acc_empty + buf);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // |x|^2 - 2 q.x for 16 columns and their minimum: one FMA
                    // and one min per element; the insertion path runs only
                    // when some column beats the row's current k-th distance
                    const int jb = c * 32 + h * 16;
                    const float4 *x4 = reinterpret_cast<const float4 *>(xs + jb);
                    float tv[16];
#pragma unroll
                    for (int j4 = 0; j4 < 4; ++j4) {
                        const float4 xv = x4[j4];
                        const float xa[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            tv[j4 * 4 + e] = fmaf(-2.0f, __uint_as_float(v[h * 16 + j4 * 4 + e]), xa[e]);
                    }
                    float m8[8];  // minimum as a tree (independent instructions)
#pragma unroll
                    for (int j = 0; j < 8; ++j) m8[j] = fminf(tv[2 * j], tv[2 * j + 1]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) m8[j] = fminf(m8[2 * j], m8[2 * j + 1]);
                    const float mn = fminf(fminf(m8[0], m8[1]), fminf(m8[2], m8[3]));
                    if (mn < thrp) {
                        // columns of this group that exist, are not the row itself, and
                        // beat the threshold: a bit mask, then one step per set bit
                        const int nv = lim - jb;
                        unsigned vm = nv >= 16 ? 0xffffu : (nv <= 0 ? 0u : (1u << nv) - 1u);
                        if ((unsigned)(self_local - jb) < 16u) vm &= ~(1u << (self_local - jb));
                        unsigned msk = 0;
#pragma unroll
                        for (int j = 0; j < 16; ++j) msk |= (tv[j] < thrp ? 1u : 0u) << j;
                        msk &= vm;
                        if (msk) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) tvs[j * 32 + lane] = tv[j];
                            while (msk) {
                                const int j = __ffs(msk) - 1;
                                msk &= msk - 1;
                                mybuf[cnt] = make_key(fmaxf(qn_r + tvs[j * 32 + lane], 0.0f), (int)(col0 + jb + j));
                                ++cnt;
                            }
                        }
                    }
                    unsigned need = __ballot_sync(NSG_FULL, cnt >= TC_MERGE_AT);
                    while (need) {
                        const int src = __ffs(need) - 1;
                        need &= need - 1;
                        merge_row(src, row_local, row_g, cnt, lsize, thrp, qn_r, bufs, ls, sb, thr_slot,
                                  a.ids, a.d2, a.KL);
                    }
                }
            }
        }
        if (ok) {
            unsigned need = __ballot_sync(NSG_FULL, cnt > 0);
            while (need) {
                const int src = __ffs(need) - 1;
                need &= need - 1;
                merge_row(src, row_local, row_g, cnt, lsize, thrp, qn_r, bufs, ls, sb, thr_slot, a.ids,
                          a.d2, a.KL);
            }
            if (!a.last) {  // carry the list size to the next chunk
                if (valid) a.lsz[row_g] = lsize;
            } else  // pad rows holding fewer than k candidates
            for (int src = 0; src < 32; ++src) {
                const int s = __shfl_sync(NSG_FULL, lsize, src);
                const int64_t rg = __shfl_sync(NSG_FULL, row_g, src);
                const bool v = __shfl_sync(NSG_FULL, valid ? 1 : 0, src);
                if (!v) continue;
                for (int i = s + lane; i < a.KL; i += 32) {
                    a.ids[rg * a.KL + i] = -1;
                    a.d2[rg * a.KL + i] = __int_as_float(0x7f800000);
                }
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (*abort && !skip && threadIdx.x == 0) atomicExch(a.err, 1);
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, 2 * TC_N);
    }
}

template <int DK>
cudaError_t launch(const CUtensorMap &mA, const CUtensorMap &mB, const TcArgs &a, cudaStream_t st) {
    auto kern = knn_tc_small_kernel<DK>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TcCfg<DK>::SMEM);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((a.m + TC_M - 1) / TC_M), TC_THREADS, TcCfg<DK>::SMEM, st>>>(mA, mB, a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t knn_select_small(const KnnLaunch &l, const KnnOperands &o, int *ids, float *d2, cudaStream_t st) {
    TcArgs a;
    a.qn = o.qn;
    a.xn = o.xn;
    a.m = l.nq;
    a.n = l.n;
    a.q0 = l.q0;
    a.self_join = l.self_join;
    a.KL = o.KL;
    a.kb = o.dk / TC_BOXK;
    a.ids = ids;
    a.d2 = d2;
    a.err = o.err;
    // rows see columns in increasing id across chunks, and their lists carry over
    // through the output arrays and lsz
    const int64_t chunk = knn_chunk_tiles(o.dk), nchunks = (o.ntiles + chunk - 1) / chunk;
    cudaError_t e;
    KnnScratch<int> lsz;
    if (nchunks > 1 && (e = lsz.alloc((size_t)l.nq)) != cudaSuccess) return e;
    a.lsz = lsz.p;
    for (int64_t c = 0; c < nchunks; ++c) {
        a.t0 = (int)(c * chunk);
        a.t1 = (int)std::min<int64_t>(o.ntiles, (c + 1) * chunk);
        a.first = c == 0;
        a.last = c == nchunks - 1;
        e = o.dk == 64 ? launch<64>(o.mq, o.mx, a, st)
            : o.dk == 128 ? launch<128>(o.mq, o.mx, a, st)
                          : launch<0>(o.mq, o.mx, a, st);
        if (e != cudaSuccess) return e;
    }
    return knn_finish(o, st);  // lsz is freed on return
}

}  // namespace nsg
