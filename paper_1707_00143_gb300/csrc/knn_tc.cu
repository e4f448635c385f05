// knn_tc.cu -- brute-force k nearest neighbours on the 5th-generation tensor
// cores (serial scan of Section 4.1.2; the kNN graph G of Alg. 2 and the
// ground truth of Eq. 1).
//
// d2(q, x) = |q|^2 + (|x|^2 - 2 q.x): the dot products are a BF16 GEMM with
// FP32 accumulation in TMEM (tcgen05.mma, operands staged by TMA with 128-byte
// swizzle).  On integer data in 0..255 with d <= 128 every product, partial
// sum, norm and the final combination is an integer below 2^24, so the
// distances are exact and the selection below equals the serial scan bit for
// bit; the launcher checks the data and reports "not applicable" otherwise.
//
// A work unit is 256 query rows (two 128-row groups, M = 128 each, sharing the
// staged base tiles of N = 128 rows) against a range of base tiles; one
// persistent CTA per SM.  Warp 0 issues TMA, warp 1 the MMAs into two
// accumulators per group (all 512 TMEM columns).  Each group has four scanning
// warps: thread r of a group looks through query row r's columns.  A base
// column j becomes a candidate of row r only when
// |x_j|^2 - 2 q.x_j < (k-th distance so far) - |q|^2.  Columns arrive in
// increasing id, so a strict comparison on the distance alone implements the
// (distance, id) order.  The 8-column groups holding candidates go to the
// row's ring in global memory; behind each scanning warp a merging warp takes
// rows with 28 or more groups in their rings, merges their candidates into
// the rows' sorted lists, which live in the output arrays, and publishes the
// new k-th distances.  A scan with an older bound only finds more candidates.
//
// Bound by latency: at 262,144 x 128 the tensor pipe is active 25 % of the cycles
// and issue 42 %; a scanning warp loads 32 columns, waits and tests them with
// nothing in flight behind (long scoreboard 3.8 per instruction), and the
// accumulator hand-over holds the MMAs to that pace.  A column costs half a packed
// FMA and half a 3-input min per row, and a candidate's group ~10 warp
// instructions whatever the other 31
// rows do.  What the structure is for:
//  (a) merging takes ~5,000 cycles of dependent loads and shuffles; done by
//      the scanning warps it held up the accumulators, and with them every
//      other warp of the CTA (the sum of all merges, not their average);
//  (b) a candidate's whole group is stored without looking for it in there
//      (the merge filters), which also keeps the loop small;
//  (c) a pre-pass over a sample of the tiles (a quarter of them at most)
//      bounds every row's k-th distance before the first candidate: of the
//      sample's 64-column minima the k-th smallest has k columns at or below
//      it.  That leaves ~k (1 + ln(n / sample)) candidates per row instead of
//      k (1 + ln(n / k)).
// Measured (before: four epilogue warps that also merged, one CTA per 128
// rows, no pre-pass -> now): 300,007 x 128 integer rows, K = 100, 121.9 ->
// 40.2 ms (575 TFLOP/s); 1,000 queries on 1,000,000 x 960 floats, k = 100,
// 47.3 -> 6.5 ms, most of it from the split; 100 queries on 10,000 x 32, k = 10,
// 0.77 -> 0.49 ms.  Without the merging warps the first took 55-72 ms.
// Few query rows are spread over the SMs by splitting the base tiles; the
// splits' lists are merged at the end.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "knn_rule.h"
#include "knn_tc.cuh"
#include "tc_ptx.cuh"

namespace nsg {

namespace {

constexpr int TC_M = 128;       // query rows per group (TMEM lanes)
constexpr int TC_G = 2;         // row groups per work unit
constexpr int TC_UNIT = TC_G * TC_M;
constexpr int TC_N = 128;       // base rows per tile (accumulator columns)
constexpr int TC_BOXK = 64;     // bf16 elements per 128-byte swizzle atom
constexpr int TC_BUF = 64;      // candidates merged at a time
constexpr int TC_MERGE = 28;    // 8-column groups in a row's ring before they are merged (~30 candidates)
constexpr int TC_RING = 64;     // ring size (a power of two; a tile adds up to 16)
constexpr int TC_SCAN = 4 * TC_G;  // scanning warps, and as many merging warps
constexpr int TC_THREADS = 32 * (2 + 2 * TC_SCAN);
constexpr int TC_MAXK = 256;

struct TcArgs {
    const float *qn;  // [m] squared norms of the query rows
    const float *xn;  // [ntiles * 128] squared norms of the base rows, +inf past the last row
    int64_t m, n, q0;
    int self_join, KL;
    int tile0, tile1;  // tiles of this launch (sample positions in the pre-pass)
    int stride;        // base tile of position i is i * stride (1 but for the pre-pass)
    int T, S;          // row units, splits of the tile range; work unit u: rows rt0 + u % T, split u / T
    int rt0;
    int first, last;   // first chunk: lists start empty; last chunk: pad short lists
    int kb;            // 64-wide K chunks per row (streaming form)
    int *ids;          // lists [m][S][KL]
    float *d2;
    int *lsz;          // [m] list sizes carried between chunks
    const float *thr0; // [m] pre-pass bounds on |x|^2 - 2 q.x (strict), or nullptr
    float *minima;     // pre-pass: [2 * tiles][mpad], rows from unit rt0
    int64_t mpad;
    float *vals;       // [grid][256][TC_RING][8] candidate groups: |x|^2 - 2 q.x
    int *cols;         // [grid][256][TC_RING] their first columns
    int *err;
};

// DK = 64 or 128: the unit's 256 query rows stay in shared memory and a stage
// holds one base tile.  DK = 0: rows wider than 128 values; a stage holds one
// 64-wide K chunk of the base tile and of the query groups (16 KB each), and
// a tile takes dk/64 stages.
template <int DK>
struct TcCfg {
    static constexpr int KB = DK / TC_BOXK;                                      // swizzle atoms along K (resident form)
    static constexpr int A_GROUP = TC_M * DK * 2;                                // bytes of one resident group
    static constexpr int A_BYTES = TC_G * A_GROUP;
    static constexpr int B_BYTES = DK ? TC_N * DK * 2 : (1 + TC_G) * TC_N * 128;  // one pipeline stage
    static constexpr int NS = DK == 64 ? 8 : 4;                                  // stages
    static constexpr int OFF_B = A_BYTES;
    static constexpr int OFF_SCAN = OFF_B + NS * B_BYTES;        // per scanning warp: base norms of a tile
    static constexpr int OFF_MERGE = OFF_SCAN + TC_SCAN * TC_N * 4;
    // per merging warp: candidates being merged, k-th slot, rank counts
    static constexpr int MERGE_BYTES = TC_BUF * 8 + 16 + (TC_BUF + 4) * 4;
    // per row: ring head, tail, head at the unit's end, bound; per scanning
    // warp: units scanned, units the merging warp has begun
    static constexpr int OFF_ROW = OFF_MERGE + TC_SCAN * MERGE_BYTES;
    static constexpr int OFF_BAR = OFF_ROW + TC_UNIT * 16 + TC_SCAN * 8;
    // a_full, a_empty, b_full[NS], b_empty[NS], acc_full[G][2], acc_empty[G][2], drain
    static constexpr int NBAR = 2 + 2 * NS + 4 * TC_G + 1;
    static constexpr int SMEM = OFF_BAR + NBAR * 8 + 16 + 1024;  // + alignment slack
};

__device__ __forceinline__ float min3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// A row's sorted list in registers (entry t * 32 + lane), all loads in flight
// at once: entries past the list's end read its first one.
struct RowList {
    float d2[TC_MAXK / 32];
    int id[TC_MAXK / 32];
    __device__ __forceinline__ void load(const int *oid, const float *od, int KL) {
#pragma unroll
        for (int t = 0; t < TC_MAXK / 32; ++t) {
            const int i = t * 32 + (int)lane_id(), j = i < KL ? i : 0;
            d2[t] = od[j];
            id[t] = oid[j];
        }
    }
};

// Number of the c <= 64 sorted keys at sb that are less than each of four keys
// (four searches in step).
__device__ __forceinline__ void count_less4(const uint64_t *sb, int c, const uint64_t (&k)[4], int (&r)[4]) {
#pragma unroll
    for (int t = 0; t < 4; ++t) r[t] = 0;
#pragma unroll
    for (int step = 64; step > 0; step >>= 1)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int m = r[t] + step;
            if (m <= c && sb[m - 1] < k[t]) r[t] = m;
        }
}

// The c <= 64 candidates in sb into the sorted list of s keys at oid / od.
// Every candidate finds its rank among the candidates (independent compares
// against broadcast reads, while the list's loads are in flight; a sorting
// network is a chain of shuffles); list keys
// find theirs by binary search; the counts of those ranks give the candidates'
// ranks in the list.  One copy of this code, not inlined: a merge runs straight
// through, so fetching instructions counts (nine inlined copies: 47.7 ms instead
// of 39.8 ms for the 300,007-row graph).
__device__ __noinline__ void merge_piece(int c, int &size, uint64_t *sb, int *hist, uint64_t *thr_slot, int *oid,
                                         float *od, int KL) {
    int s = size;
    RowList list;
    list.load(oid, od, KL);
    const unsigned lane = lane_id();
    const uint64_t a = (int)lane < c ? sb[lane] : ~0ull, b = (int)lane + 32 < c ? sb[lane + 32] : ~0ull;
    int ra = 0, rb = 0;
    if (c <= 32) {
#pragma unroll 8
        for (int j = 0; j < c; ++j) ra += sb[j] < a;
    } else {
#pragma unroll 8
        for (int j = 0; j < c; ++j) {
            const uint64_t o = sb[j];
            ra += o < a;
            rb += o < b;
        }
    }
    __syncwarp();
    if ((int)lane < c) sb[ra] = a;
    if ((int)lane + 32 < c) sb[rb] = b;
    hist[lane] = 0;
    hist[lane + 32] = 0;
    if (lane == 0) hist[64] = 0;
    __syncwarp();
#pragma unroll
    for (int t0 = 0; t0 < TC_MAXK / 32; t0 += 4) {
        if (t0 * 32 >= s) break;
        uint64_t key[4];
        int r[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) key[t] = make_key(list.d2[t0 + t], list.id[t0 + t]);
        count_less4(sb, c, key, r);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int i = (t0 + t) * 32 + (int)lane, p = i + r[t];
            if (i < s) {
                atomicAdd(hist + r[t], 1);
                if (r[t] > 0 && p < KL) {  // the others stay where they are
                    od[p] = kd2(key[t]);
                    oid[p] = kid(key[t]);
                }
                if (p == KL - 1) *thr_slot = key[t];
            }
        }
    }
    __syncwarp();
    // list keys below sorted candidate j: those whose rank is at most j
    int h0 = hist[lane], h1 = hist[lane + 32];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(NSG_FULL, h0, o), y = __shfl_up_sync(NSG_FULL, h1, o);
        if ((int)lane >= o) {
            h0 += x;
            h1 += y;
        }
    }
    h1 += __shfl_sync(NSG_FULL, h0, 31);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = (int)lane + 32 * h, p = j + (h ? h1 : h0);
        if (j < c && p < KL) {
            const uint64_t k = sb[j];
            od[p] = kd2(k);
            oid[p] = kid(k);
            if (p == KL - 1) *thr_slot = k;
        }
    }
    size = s + c < KL ? s + c : KL;
    __syncwarp();
}

// Merge the groups [tail, head) of a row's ring into its sorted list (at most
// KL keys at oid / od, s of them): the values still below the row's bound are
// collected (the row itself, in a self join, is dropped) and merged up to 64 at
// a time, usually all at once.  Warp-wide; returns the row's bound.
__device__ __forceinline__ float merge_row(const float *vals, const int *cols, int tail, int head, int own, float q2,
                                           float bar, int &s, uint64_t *sb, int *hist, uint64_t *thr_slot, int *oid,
                                           float *od, int KL) {
    const unsigned lane = lane_id();
    const int total = (head - tail) * 8, e8 = (int)(lane & 7);
    int c = 0;
#pragma unroll 1
    for (int e0 = 0; e0 < total; e0 += 128) {
        float tv[4];
        int col[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {  // all loads issued before the first use
            const int r = (tail + ((e0 + t * 32 + (int)lane) >> 3)) & (TC_RING - 1);
            tv[t] = __ldcg(vals + r * 8 + e8);
            col[t] = __ldcg(cols + r) + e8;
        }
        bool take[4];
        int add = 0;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            take[t] = e0 + t * 32 + (int)lane < total && tv[t] < bar && col[t] != own;
            add += __popc(__ballot_sync(NSG_FULL, take[t]));
        }
        if (c + add > TC_BUF) {  // make room (more than 64 at once, a row's first groups: below, 32 at a time)
            __syncwarp();
            if (c > 0) merge_piece(c, s, sb, hist, thr_slot, oid, od, KL);
            if (s == KL) bar = kd2(*thr_slot) - q2;
            c = 0;
            __syncwarp();
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const unsigned bal = __ballot_sync(NSG_FULL, take[t]);
            if (take[t]) sb[c + __popc(bal & lanemask_lt())] = make_key(fmaxf(q2 + tv[t], 0.0f), col[t]);
            c += __popc(bal);
            if (add > TC_BUF && (t & 1)) {
                __syncwarp();
                if (c > 0) merge_piece(c, s, sb, hist, thr_slot, oid, od, KL);
                c = 0;
                __syncwarp();
            }
        }
        if (add > TC_BUF && s == KL) bar = kd2(*thr_slot) - q2;
    }
    __syncwarp();
    if (c > 0) {
        merge_piece(c, s, sb, hist, thr_slot, oid, od, KL);
        if (s == KL) bar = kd2(*thr_slot) - q2;
        __syncwarp();
    }
    return bar;
}

// The tiles of work unit u.
__device__ __forceinline__ void unit_tiles(const TcArgs &a, int u, int *rt, int *i0, int *i1) {
    const int sp = u / a.T;
    *rt = a.rt0 + u - sp * a.T;
    const int64_t len = a.tile1 - a.tile0;
    *i0 = a.tile0 + (int)(len * sp / a.S);
    *i1 = a.tile0 + (int)(len * (sp + 1) / a.S);
}

// Two FMAs in one instruction (round to nearest each).
__device__ __forceinline__ void fma2(float &d0, float &d1, float a0, float a1, float b, float c0, float c1) {
    uint64_t d, x, y, z;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a0), "f"(a1));
    asm("mov.b64 %0, {%1, %1};" : "=l"(y) : "f"(b));
    asm("mov.b64 %0, {%1, %2};" : "=l"(z) : "f"(c0), "f"(c1));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(x), "l"(y), "l"(z));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d0), "=f"(d1) : "l"(d));
}

// Row groups of a unit that hold query rows.
__device__ __forceinline__ int unit_groups(const TcArgs &a, int rt) {
    const int64_t rows = a.m - (int64_t)rt * TC_UNIT;
    return rows >= TC_UNIT ? TC_G : (int)((rows + TC_M - 1) / TC_M);
}

// A row's bound on |x|^2 - 2 q.x and its list's size when a unit begins: the
// k-th key carried over from earlier chunks once the list holds k, before that
// the pre-pass's; a row past the end takes nothing.  Keys are rounded sums with
// |q|^2 and equal ones go by id, so the pre-pass's bound is widened by what that
// rounding can make equal, and a norm past FP32's range (every key infinite)
// leaves it out.
__device__ __forceinline__ float first_bound(const TcArgs &a, int64_t row, int64_t list, int *lsize) {
    *lsize = 0;
    const float inf = __int_as_float(0x7f800000);
    if (row >= a.m) return -inf;
    if (!a.first) *lsize = a.lsz[row];
    const float q2 = a.qn[row];
    if (*lsize == a.KL) return a.d2[list + a.KL - 1] - q2;
    if (a.thr0 == nullptr || !(q2 < inf)) return inf;
    const float t = a.thr0[row];
    return t + (q2 + fabsf(t)) * (1.0f / (1 << 22));
}

// MINS: the pre-pass (minima of every sample tile's two 64-column groups),
// else the selection.
template <int DK, bool MINS>
__global__ void __launch_bounds__(TC_THREADS, 1)
    knn_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const __grid_constant__ TcArgs a) {
    using Cfg = TcCfg<DK>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char *sA = smem;
    unsigned char *sB = smem + Cfg::OFF_B;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + Cfg::OFF_BAR);
    uint64_t *a_full = bars, *a_empty = bars + 1;
    uint64_t *b_full = bars + 2;
    uint64_t *b_empty = b_full + Cfg::NS;
    uint64_t *acc_full = b_empty + Cfg::NS;  // [group * 2 + buffer]
    uint64_t *acc_empty = acc_full + 2 * TC_G;
    uint64_t *drain = acc_empty + 2 * TC_G;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + Cfg::NBAR);
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile int *gerr = a.err;
    volatile int *r_head = reinterpret_cast<volatile int *>(smem + Cfg::OFF_ROW);  // [256] each
    volatile int *r_tail = r_head + TC_UNIT, *r_end = r_tail + TC_UNIT;
    volatile float *r_thr = reinterpret_cast<volatile float *>(r_end + TC_UNIT);
    volatile int *scanned = reinterpret_cast<volatile int *>(r_thr + TC_UNIT);  // [TC_SCAN]
    volatile int *begun = scanned + TC_SCAN;

    const int warp = threadIdx.x >> 5;
    const unsigned lane = lane_id();
    const int units = a.T * a.S;

    for (int t = threadIdx.x; t < TC_UNIT; t += TC_THREADS) r_head[t] = r_tail[t] = r_end[t] = 0;
    if (threadIdx.x < TC_SCAN) scanned[threadIdx.x] = begun[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        tc::mbar_init(a_full, 1);
        tc::mbar_init(a_empty, 1);
        for (int s = 0; s < Cfg::NS; ++s) {
            tc::mbar_init(b_full + s, 1);
            tc::mbar_init(b_empty + s, 1);
        }
        for (int b = 0; b < 2 * TC_G; ++b) {
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
        tc::tmem_alloc(tmem_slot, 2 * TC_G * TC_N);
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
            const int per_tile = DK ? 1 : a.kb;  // stages per tile
            int c = 0, nu = 0;                   // stages issued; units whose query rows were
            bool ok = true;
            for (int u = blockIdx.x; ok && u < units; u += gridDim.x) {
                int rt, i0, i1;
                unit_tiles(a, u, &rt, &i0, &i1);
                const int row0 = rt * TC_UNIT, groups = unit_groups(a, rt);
                if (DK) {
                    if (!tc::mbar_wait(a_empty, (nu & 1) ^ 1, abort, gerr)) break;
                    tc::mbar_expect_tx(a_full, groups * Cfg::A_GROUP);
                    for (int g = 0; g < groups; ++g)
                        for (int kb = 0; kb < Cfg::KB; ++kb)
                            tc::tma_load_2d(sA + g * Cfg::A_GROUP + kb * (TC_M * 128), &tmA, a_full, kb * TC_BOXK,
                                            row0 + g * TC_M);
                    ++nu;
                }
                for (int i = i0; ok && i < i1; ++i)
                    for (int kc = 0; kc < per_tile; ++kc, ++c) {
                        const int s = c % Cfg::NS;
                        if (!tc::mbar_wait(b_empty + s, ((c / Cfg::NS) & 1) ^ 1, abort, gerr)) {
                            ok = false;
                            break;
                        }
                        unsigned char *dst = sB + s * Cfg::B_BYTES;
                        const int y = i * a.stride * TC_N;
                        tc::mbar_expect_tx(b_full + s, DK ? Cfg::B_BYTES : (1 + groups) * TC_N * 128);
                        if (DK) {
                            for (int kb = 0; kb < Cfg::KB; ++kb)
                                tc::tma_load_2d(dst + kb * (TC_N * 128), &tmB, b_full + s, kb * TC_BOXK, y);
                        } else {
                            tc::tma_load_2d(dst, &tmB, b_full + s, kc * TC_BOXK, y);
                            for (int g = 0; g < groups; ++g)
                                tc::tma_load_2d(dst + (1 + g) * TC_N * 128, &tmA, b_full + s, kc * TC_BOXK,
                                                row0 + g * TC_M);
                        }
                    }
            }
            if (*abort) {
                // drain: wait (bounded) for the copies still in flight
                volatile int local = 0;
                if (nu > 0) tc::mbar_wait(a_full, (nu - 1) & 1, &local, nullptr);
                for (int x = c - Cfg::NS < 0 ? 0 : c - Cfg::NS; x < c; ++x) {
                    local = 0;
                    tc::mbar_wait(b_full + x % Cfg::NS, (x / Cfg::NS) & 1, &local, nullptr);
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            constexpr uint32_t idesc = tc::idesc_bf16_f32(TC_M, TC_N);
            const uint32_t a_base = tc::smem_u32(sA), b_base = tc::smem_u32(sB);
            const int per_tile = DK ? 1 : a.kb;
            int c = 0, nu = 0;      // stages, units
            int tg[TC_G] = {0, 0};  // tiles of each group so far
            bool ok = true;
            for (int u = blockIdx.x; ok && u < units; u += gridDim.x, ++nu) {
                int rt, i0, i1;
                unit_tiles(a, u, &rt, &i0, &i1);
                const int groups = unit_groups(a, rt);
                if (DK && !tc::mbar_wait(a_full, nu & 1, abort, gerr)) break;
                for (int i = i0; ok && i < i1; ++i) {
                    for (int kc = 0; ok && kc < per_tile; ++kc, ++c) {
                        const int s = c % Cfg::NS;
                        if (!tc::mbar_wait(b_full + s, (c / Cfg::NS) & 1, abort, gerr)) {
                            ok = false;
                            break;
                        }
                        const uint32_t st = b_base + s * Cfg::B_BYTES;
#pragma unroll
                        for (int g = 0; g < TC_G; ++g) {
                            if (g >= groups) break;
                            const int ab = g * 2 + (tg[g] & 1);  // the tile's accumulator
                            if (kc == 0 && !tc::mbar_wait(acc_empty + ab, ((tg[g] >> 1) & 1) ^ 1, abort, gerr)) {
                                ok = false;
                                break;
                            }
                            tc::fence_after_sync();
                            const uint32_t acc = tmem + ab * TC_N;
                            if (DK) {
#pragma unroll
                                for (int kk = 0; kk < (DK ? DK : 64) / 16; ++kk) {
                                    const uint32_t off = (kk >> 2) * (TC_M * 128) + (kk & 3) * 32;
                                    tc::mma_bf16(acc, tc::sdesc_sw128(a_base + g * Cfg::A_GROUP + off),
                                                 tc::sdesc_sw128(st + off), idesc, kk > 0 ? 1u : 0u);
                                }
                            } else {
#pragma unroll
                                for (int kk = 0; kk < 4; ++kk)
                                    tc::mma_bf16(acc, tc::sdesc_sw128(st + (1 + g) * TC_N * 128 + kk * 32),
                                                 tc::sdesc_sw128(st + kk * 32), idesc, (kc > 0 || kk > 0) ? 1u : 0u);
                            }
                            if (kc == per_tile - 1) {
                                tc::mma_commit(acc_full + ab);
                                ++tg[g];
                            }
                        }
                        tc::mma_commit(b_empty + s);
                    }
                }
                if (DK && ok) tc::mma_commit(a_empty);
            }
            // every MMA issued so far has completed before TMEM is released
            tc::mma_commit(drain);
            volatile int local = 0;
            tc::mbar_wait(drain, 0, &local, nullptr);
        }
    } else if (warp < 2 + TC_SCAN) {
        // ---------------- scan: warps 2 + 4g .. 5 + 4g for row group g ----------------
        const int q = warp & 3;  // TMEM lane quadrant of this warp
        const int w = warp - 2, g = w >> 2;
        float *xs = reinterpret_cast<float *>(smem + Cfg::OFF_SCAN) + w * TC_N;
        const int row_local = g * TC_M + q * 32 + (int)lane;
        const unsigned ring = ((unsigned)blockIdx.x * TC_UNIT + row_local) * TC_RING;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + g * 2 * TC_N;
        const float4 *xn4 = reinterpret_cast<const float4 *>(a.xn);
        int tcnt = 0, nu = 0;    // tiles and units of this group so far
        int head = 0, told = 0;  // groups put into the ring; the count last published
        bool ok = true;
        for (int u = blockIdx.x; ok && u < units; u += gridDim.x) {
            int rt, i0, i1;
            unit_tiles(a, u, &rt, &i0, &i1);
            if (g >= unit_groups(a, rt)) continue;
            ++nu;
            const int64_t row_g = (int64_t)rt * TC_UNIT + row_local;
            const bool valid = row_g < a.m;
            float thrp = 0.0f;
            if (!MINS) {
                int lsize;
                thrp = first_bound(a, row_g, (row_g * a.S + u / a.T) * a.KL, &lsize);
            }
            float4 xnext = i0 < i1 ? __ldg(xn4 + (int64_t)i0 * a.stride * (TC_N / 4) + lane)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);  // norms one tile ahead
            for (int i = i0; i < i1; ++i, ++tcnt) {
                const int buf = tcnt & 1, col0 = i * a.stride * TC_N;
                __syncwarp();
                reinterpret_cast<float4 *>(xs)[lane] = xnext;
                if (i + 1 < i1) xnext = __ldg(xn4 + (int64_t)(i + 1) * a.stride * (TC_N / 4) + lane);
                bool room = true;
                if (!MINS) {
                    // the merging warp's bound, once it is at this unit; room in the
                    // ring for all of a tile's groups
                    if (begun[w] == nu) thrp = r_thr[row_local];
                    if (!__all_sync(NSG_FULL, head + 16 - r_tail[row_local] <= TC_RING)) {
                        __threadfence_block();
                        r_head[row_local] = told = head;
                        const uint64_t t0 = tc::globaltimer();
                        while (room && !__all_sync(NSG_FULL, head + 16 - r_tail[row_local] <= TC_RING)) {
                            __nanosleep(100);
                            if (*abort || tc::globaltimer() - t0 > tc::WAIT_TIMEOUT_NS) room = false;
                            room = __all_sync(NSG_FULL, room);
                        }
                        if (!room) *abort = 1;
                        if (begun[w] == nu) thrp = r_thr[row_local];
                    }
                }
                __syncwarp();
                const bool got = room && tc::mbar_wait(acc_full + g * 2 + buf, (tcnt >> 1) & 1, abort, gerr);
                if (!__all_sync(NSG_FULL, got)) {  // warp-uniform before the .sync.aligned TMEM loads
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                float even = 0.0f;
#pragma unroll 1
                for (int c = 0; c < TC_N / 32; ++c) {
                    uint32_t v[32];
                    tc::tmem_ld32_wait(tq + buf * TC_N + c * 32, v);
                    if (c == TC_N / 32 - 1) {  // the tile's last columns are in registers
                        tc::fence_before_sync();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(acc_empty + g * 2 + buf);
                    }
                    // |x|^2 - 2 q.x, and the minima of 8-column groups
                    const float4 *x4 = reinterpret_cast<const float4 *>(xs + c * 32);
                    float tv[32], m8[4];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float4 xv = x4[j];
                        fma2(tv[4 * j], tv[4 * j + 1], __uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]), -2.0f,
                             xv.x, xv.y);
                        fma2(tv[4 * j + 2], tv[4 * j + 3], __uint_as_float(v[4 * j + 2]),
                             __uint_as_float(v[4 * j + 3]), -2.0f, xv.z, xv.w);
                    }
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const float p = min3(tv[h * 8], tv[h * 8 + 1], tv[h * 8 + 2]);
                        const float r = min3(tv[h * 8 + 3], tv[h * 8 + 4], tv[h * 8 + 5]);
                        m8[h] = fminf(min3(tv[h * 8 + 6], tv[h * 8 + 7], p), r);
                    }
                    const float mn = fminf(min3(m8[0], m8[1], m8[2]), m8[3]);
                    if (MINS) {
                        if ((c & 1) == 0) even = mn;
                        else if (valid)
                            a.minima[((int64_t)i * 2 + (c >> 1)) * a.mpad + (row_g - (int64_t)a.rt0 * TC_UNIT)] =
                                fminf(even, mn);
                    } else if (mn < thrp) {
#pragma unroll
                        for (int h = 0; h < 4; ++h)
                            if (m8[h] < thrp) {
                                const unsigned at = ring + (head & (TC_RING - 1));
                                float4 *dst = reinterpret_cast<float4 *>(a.vals) + (size_t)at * 2;
                                dst[0] = make_float4(tv[h * 8], tv[h * 8 + 1], tv[h * 8 + 2], tv[h * 8 + 3]);
                                dst[1] = make_float4(tv[h * 8 + 4], tv[h * 8 + 5], tv[h * 8 + 6], tv[h * 8 + 7]);
                                a.cols[at] = col0 + c * 32 + h * 8;
                                ++head;
                            }
                    }
                    __syncwarp();
                }
                if (!MINS && __any_sync(NSG_FULL, head - told >= TC_MERGE / 2)) {
                    __threadfence_block();
                    r_head[row_local] = told = head;
                }
            }
            if (!MINS && ok) {
                // at most one unit ahead of the merging warp
                const uint64_t t0 = tc::globaltimer();
                while (ok && begun[w] != nu) {
                    __nanosleep(200);
                    if (*abort || tc::globaltimer() - t0 > tc::WAIT_TIMEOUT_NS) ok = false;
                }
                ok = __all_sync(NSG_FULL, ok);
                if (!ok) *abort = 1;
                r_end[row_local] = r_head[row_local] = told = head;
                __threadfence_block();
                __syncwarp();
                if (lane == 0) scanned[w] = nu;
            }
        }
    } else if (!MINS) {
        // ---------------- merge: one warp behind each scanning warp ----------------
        const int w = warp - 2 - TC_SCAN, g = w >> 2, q = (w + 2) & 3;
        unsigned char *wsm = smem + Cfg::OFF_MERGE + w * Cfg::MERGE_BYTES;
        uint64_t *sb = reinterpret_cast<uint64_t *>(wsm);
        uint64_t *thr_slot = sb + TC_BUF;
        int *hist = reinterpret_cast<int *>(thr_slot + 2);
        const int row_local = g * TC_M + q * 32 + (int)lane;
        const size_t ring0 = ((size_t)blockIdx.x * TC_UNIT + g * TC_M + q * 32) * TC_RING;
        int nu = 0, tail = 0;
        bool ok = true;
        for (int u = blockIdx.x; ok && u < units; u += gridDim.x) {
            int rt, i0, i1;
            unit_tiles(a, u, &rt, &i0, &i1);
            if (g >= unit_groups(a, rt)) continue;
            ++nu;
            const int64_t row_g = (int64_t)rt * TC_UNIT + row_local;
            const bool valid = row_g < a.m;
            const int64_t list0 = (row_g * a.S + u / a.T) * a.KL;
            const int self = a.self_join ? (int)(a.q0 + row_g) : -1;
            const float qn_r = valid ? a.qn[row_g] : 0.0f;
            int lsize;
            float thrp = first_bound(a, row_g, list0, &lsize);
            r_thr[row_local] = thrp;
            __threadfence_block();
            __syncwarp();
            if (lane == 0) begun[w] = nu;
            uint64_t t0 = tc::globaltimer();
            for (;;) {
                // the head is read before the flag: a head past the unit's end is
                // published only after the flag
                int head = tc::lds_acquire(r_head + row_local);
                const bool fin = __shfl_sync(NSG_FULL, tc::lds_acquire(scanned + w), 0) >= nu;
                if (fin) head = r_end[row_local];
                unsigned need = __ballot_sync(NSG_FULL, head - tail >= (fin ? 1 : TC_MERGE));
                if (!need) {
                    if (fin) break;
                    __nanosleep(500);
                    const bool gone = *abort || tc::globaltimer() - t0 > tc::WAIT_TIMEOUT_NS;
                    if (__any_sync(NSG_FULL, gone)) {
                        *abort = 1;
                        ok = false;
                        break;
                    }
                    continue;
                }
                while (need) {
                    const int src = __ffs(need) - 1;
                    need &= need - 1;
                    const int rt0 = __shfl_sync(NSG_FULL, tail, src), rh = __shfl_sync(NSG_FULL, head, src);
                    const int own = __shfl_sync(NSG_FULL, self, src);
                    const float q2 = __shfl_sync(NSG_FULL, qn_r, src);
                    const int64_t lr = __shfl_sync(NSG_FULL, list0, src);
                    int s = __shfl_sync(NSG_FULL, lsize, src);
                    const float *vals = a.vals + (ring0 + (size_t)src * TC_RING) * 8;
                    const float bar = merge_row(vals, a.cols + ring0 + (size_t)src * TC_RING, rt0, rh, own, q2,
                                                __shfl_sync(NSG_FULL, thrp, src), s, sb, hist, thr_slot, a.ids + lr,
                                                a.d2 + lr, a.KL);
                    if ((int)lane == src) {
                        lsize = s;
                        thrp = bar;
                        tail = rh;
                        // (the ring's entries have been read: no fence, which would
                        // wait for the list's stores, thousands of cycles)
                        r_thr[row_local] = bar;
                        r_tail[row_local] = rh;
                    }
                    __syncwarp();
                }
                t0 = tc::globaltimer();
            }
            if (!ok) break;
            if (!a.last) {  // carry the list size to the next chunk
                if (valid) a.lsz[row_g] = lsize;
            } else  // pad rows holding fewer than k candidates
                for (int src = 0; src < 32; ++src) {
                    const int s = __shfl_sync(NSG_FULL, lsize, src);
                    const int64_t lr = __shfl_sync(NSG_FULL, list0, src);
                    const bool v = __shfl_sync(NSG_FULL, valid ? 1 : 0, src);
                    if (!v) continue;
                    for (int x = s + (int)lane; x < a.KL; x += 32) {
                        a.ids[lr + x] = -1;
                        a.d2[lr + x] = __int_as_float(0x7f800000);
                    }
                }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (*abort && !skip && threadIdx.x == 0) atomicExch(a.err, 1);
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, 2 * TC_G * TC_N);
    }
}

// A float's bits as an unsigned number of the same order, and back.
__device__ __forceinline__ unsigned order_bits(float f) {
    const unsigned u = __float_as_uint(f);
    return u & 0x80000000u ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float from_order_bits(unsigned u) {
    return __uint_as_float(u & 0x80000000u ? u & 0x7fffffffu : ~u);
}

// A strict bound just above the `rank`-th smallest of each row's `count`
// minima (to 2^-11 relative: the search over the order bits stops 12 bits
// early, rounding up).  One warp per row, at most KPL minima per lane.
template <int KPL>
__global__ void __launch_bounds__(256) knn_bound_kernel(const float *minima, int count, int64_t mpad, int64_t m,
                                                        int rank, float *thr) {
    const unsigned lane = lane_id();
    for (int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); r < m; r += (int64_t)gridDim.x * 8) {
        unsigned k[KPL];
#pragma unroll
        for (int t = 0; t < KPL; ++t) {
            const int i = t * 32 + (int)lane;
            k[t] = i < count ? order_bits(__ldg(minima + (int64_t)i * mpad + r)) : ~0u;
        }
        unsigned t0 = 0;  // fewer than `rank` keys are below t0
#pragma unroll 1
        for (int bit = 31; bit >= 12; --bit) {
            const unsigned c = t0 | (1u << bit);
            int below = 0;
#pragma unroll
            for (int t = 0; t < KPL; ++t) below += k[t] < c;
            if (__reduce_add_sync(NSG_FULL, below) < rank) t0 = c;
        }
        if (lane == 0) {
            const unsigned inf = 0xff800000u;  // order bits of +inf
            thr[r] = t0 >= inf || t0 + 0x1000u >= inf ? __int_as_float(0x7f800000) : from_order_bits(t0 + 0x1000u);
        }
    }
}

// The KL smallest keys of each row's S split lists [m][S][KL] (sorted, -1
// padded): one block per row, every warp merges its share of the lists, then
// one warp the eight results.
__global__ void __launch_bounds__(256) knn_merge_kernel(const int *ids_in, const float *d2_in, int64_t m, int S, int KL,
                                                        int *ids, float *d2) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int sizes[8];
    const int warp = threadIdx.x >> 5;
    const unsigned lane = lane_id();
    // per warp: list, candidates, ck, sk [KL] (u64); cp, sp [KL] (int)
    uint64_t *list = reinterpret_cast<uint64_t *>(smem) + (size_t)warp * 5 * KL;
    uint64_t *cand = list + KL, *ck = cand + KL, *sk = ck + KL;
    int *cp = reinterpret_cast<int *>(sk + KL), *sp = cp + KL;
    for (int64_t r = blockIdx.x; r < m; r += gridDim.x) {
        int size = 0;
        for (int p = warp; p < S; p += 8) {
            const int64_t at = (r * S + p) * KL;
            int c = 0;
            for (int b = 0; b < KL; b += 32) {
                const int j = b + (int)lane;
                const int id = j < KL ? ids_in[at + j] : -1;
                const unsigned bal = __ballot_sync(NSG_FULL, id >= 0);
                if (id >= 0) cand[c + __popc(bal & lanemask_lt())] = make_key(d2_in[at + j], id);
                c += __popc(bal);
            }
            __syncwarp();
            if (c > 0) warp_merge(list, KL, size, cand, c, ck, cp, sk, sp);
        }
        if (lane == 0) sizes[warp] = size;
        __syncthreads();
        if (warp == 0) {
            for (int w = 1; w < 8; ++w)
                if (sizes[w] > 0)
                    warp_merge(list, KL, size, reinterpret_cast<uint64_t *>(smem) + (size_t)w * 5 * KL, sizes[w], ck,
                               cp, sk, sp);
            for (int c = lane; c < KL; c += 32) {
                const bool has = c < size;
                ids[r * KL + c] = has ? kid(list[c]) : -1;
                d2[r * KL + c] = has ? kd2(list[c]) : __int_as_float(0x7f800000);
            }
        }
        __syncthreads();
    }
}

// Row-wise BF16 copy with K padded to DK, squared norms of the rounded values
// (+inf past the last row: such a column is never a candidate), and a flag
// raised when a value is not an integer in 0..255.  Bound by memory: a warp
// has four rows of 16-byte loads in flight.  The norms are summed lane by lane,
// value c in lane c % 32 (read again, from L1), as they have always been: where
// keys tie but for rounding (clusters far from the origin, whose rows round to few
// values) the order of the sum decides which candidates are kept.
__global__ void __launch_bounds__(256) bf16_rows_kernel(const float4 *__restrict__ src, int64_t rows, int dp4,
                                                        uint2 *dst, int dk4, float *norms, int64_t rows_pad,
                                                        int *nonint) {
    constexpr int RW = 4;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const unsigned lane = lane_id();
    const float *flat = reinterpret_cast<const float *>(src);
    bool bad = false;
    for (int64_t r0 = warp * RW; r0 < rows_pad; r0 += nw * RW) {
        float acc[RW] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int c0 = 0; c0 < dk4; c0 += 32) {
            const int c = c0 + (int)lane;
            float4 v[RW];
#pragma unroll
            for (int j = 0; j < RW; ++j)
                v[j] = r0 + j < rows && c < dp4 ? __ldg(src + (r0 + j) * dp4 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < RW; ++j) {
                const float f[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
                unsigned short h[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const __nv_bfloat16 b = __float2bfloat16_rn(f[e]);
                    bad |= !(f[e] >= 0.0f && f[e] <= 255.0f && f[e] == rintf(f[e]));
                    h[e] = __bfloat16_as_ushort(b);
                }
                if (r0 + j < rows && c < dk4)
                    dst[(r0 + j) * dk4 + c] =
                        make_uint2(h[0] | ((unsigned)h[1] << 16), h[2] | ((unsigned)h[3] << 16));
            }
            const int at = 4 * c0 + (int)lane;  // the chunk's values of this lane
#pragma unroll
            for (int j = 0; j < RW; ++j)
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int i = at + 32 * t;
                    const float f = r0 + j < rows && i < 4 * dp4 ? __ldg(flat + (r0 + j) * 4 * dp4 + i) : 0.0f;
                    const float hv = __bfloat162float(__float2bfloat16_rn(f));
                    acc[j] += hv * hv;
                }
        }
#pragma unroll
        for (int j = 0; j < RW; ++j) {
            const float s = group_sum<32>(acc[j]);
            if (lane == 0 && r0 + j < rows_pad) norms[r0 + j] = r0 + j < rows ? s : __int_as_float(0x7f800000);
        }
    }
    if (__any_sync(NSG_FULL, bad) && lane == 0) atomicOr(nonint, 1);
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// 2-D tensor map over a [rows][dk] bf16 matrix, box = 64 (K) x 128 rows, 128B swizzle.
bool make_map(CUtensorMap *map, const void *ptr, int64_t rows, int dk) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)dk, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)dk * 2};
    cuuint32_t box[2] = {(cuuint32_t)TC_BOXK, (cuuint32_t)TC_N};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Work split of one selection over `ntiles` base tiles: as few splits as
// finish the (row unit, split) pairs in about the least number of waves; a
// unit costs its tiles and, once, about 40 tiles' time to fill its lists.
int knn_splits(int T, int64_t ntiles, int64_t m, int KL) {
    const int sms = sm_count();
    double best = 0.0;
    int bs = 1;
    for (int S = 1; S <= 256 && S * 8 <= std::max<int64_t>(ntiles, 8); ++S) {
        if (S > 1 && (size_t)m * S * KL * 8 > (size_t(1) << 30)) break;
        const int64_t waves = ((int64_t)T * S + sms - 1) / sms;
        const double cost = (double)waves * ((double)ntiles / S + 40.0);
        if (S == 1 || cost < 0.9 * best) {
            best = cost;
            bs = S;
        }
    }
    return bs;
}

template <int DK, bool MINS>
cudaError_t launch_tc(const CUtensorMap &mA, const CUtensorMap &mB, const TcArgs &a, cudaStream_t st) {
    auto kern = knn_tc_kernel<DK, MINS>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TcCfg<DK>::SMEM);
    if (e != cudaSuccess) return e;
    const int64_t units = (int64_t)a.T * a.S;
    kern<<<(unsigned)std::min<int64_t>(units, sm_count()), TC_THREADS, TcCfg<DK>::SMEM, st>>>(mA, mB, a);
    return cudaGetLastError();
}

template <bool MINS>
cudaError_t launch_tc(int dk, const CUtensorMap &mA, const CUtensorMap &mB, const TcArgs &a, cudaStream_t st) {
    return dk == 64 ? launch_tc<64, MINS>(mA, mB, a, st)
           : dk == 128 ? launch_tc<128, MINS>(mA, mB, a, st)
                       : launch_tc<0, MINS>(mA, mB, a, st);
}

}  // namespace

// The KL best per query row into ids / d2 [nq][KL]: by work units of 256 rows.
static cudaError_t select_units(const KnnLaunch &l, const KnnOperands &o, int *idsout, float *d2out, cudaStream_t st) {
    const int KL = o.KL;
    const int64_t ntiles = o.ntiles;
    const int T = (int)((l.nq + TC_UNIT - 1) / TC_UNIT);
    const int S = knn_splits(T, ntiles, l.nq, KL);
    cudaError_t e;
    KnnScratch<float> d2p, vals;
    KnnScratch<int> ids_p, cols;
    if (S > 1) {
        if ((e = ids_p.alloc((size_t)l.nq * S * KL)) != cudaSuccess) return e;
        if ((e = d2p.alloc((size_t)l.nq * S * KL)) != cudaSuccess) return e;
    }
    const int64_t grid = std::min<int64_t>((int64_t)T * S, sm_count());
    if ((e = vals.alloc((size_t)grid * TC_UNIT * TC_RING * 8)) != cudaSuccess) return e;
    if ((e = cols.alloc((size_t)grid * TC_UNIT * TC_RING)) != cudaSuccess) return e;
    TcArgs a;
    a.qn = o.qn;
    a.xn = o.xn;
    a.m = l.nq;
    a.n = l.n;
    a.q0 = l.q0;
    a.self_join = l.self_join;
    a.KL = KL;
    a.kb = o.dk / TC_BOXK;
    a.ids = S > 1 ? ids_p.p : idsout;
    a.d2 = S > 1 ? d2p.p : d2out;
    a.err = o.err;
    a.vals = vals.p;
    a.cols = cols.p;
    a.T = T;
    a.thr0 = nullptr;
    a.minima = nullptr;
    a.mpad = 0;
    a.rt0 = 0;
    a.lsz = nullptr;
    a.first = a.last = 1;
    // Pre-pass: `rank` of the sample's 64-column minima have as many distinct
    // columns at or below them (one more where a row meets itself).
    const int rank = KL + (l.self_join ? 1 : 0);
    const int P = knn_sample_tiles(ntiles, rank);
    KnnScratch<float> minima, thr;
    if (P > 0) {
        // up to 1 GB of minima at a time: blocks of row units
        const int64_t fit = (int64_t(1) << 30) / ((int64_t)2 * P * TC_UNIT * 4);
        const int TB = (int)std::max<int64_t>(1, std::min<int64_t>(T, fit));
        TcArgs p = a;
        p.mpad = (int64_t)TB * TC_UNIT;
        if ((e = minima.alloc((size_t)2 * P * p.mpad)) != cudaSuccess) return e;
        if ((e = thr.alloc((size_t)l.nq)) != cudaSuccess) return e;
        p.minima = minima.p;
        p.tile0 = 0;
        p.tile1 = P;
        p.stride = (int)(ntiles / P);
        for (int t0 = 0; t0 < T; t0 += TB) {
            p.rt0 = t0;
            p.T = std::min(TB, T - t0);
            p.S = (int)std::max<int64_t>(1, std::min<int64_t>(P / 4, ((int64_t)sm_count() * 4 + p.T - 1) / p.T));
            if ((e = launch_tc<true>(o.dk, o.mq, o.mx, p, st)) != cudaSuccess) return e;
            const int64_t r0 = (int64_t)t0 * TC_UNIT, rows = std::min<int64_t>((int64_t)p.T * TC_UNIT, l.nq - r0);
            const int64_t blocks = std::min<int64_t>((rows + 7) / 8, (int64_t)sm_count() * 16);
            auto bound = 2 * P <= 512 ? knn_bound_kernel<16> : 2 * P <= 1024 ? knn_bound_kernel<32> : knn_bound_kernel<48>;
            bound<<<(unsigned)blocks, 256, 0, st>>>(minima.p, 2 * P, p.mpad, rows, rank, thr.p + r0);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        a.thr0 = thr.p;
    }
    // an unsplit base is taken in chunks: rows see columns in increasing id
    // across them, and their lists carry over through the output arrays and lsz
    const int64_t chunk = S > 1 ? ntiles : knn_chunk_tiles(o.dk), nchunks = (ntiles + chunk - 1) / chunk;
    KnnScratch<int> lsz;
    if (nchunks > 1 && (e = lsz.alloc((size_t)l.nq)) != cudaSuccess) return e;
    a.lsz = lsz.p;
    a.S = S;
    a.stride = 1;
    for (int64_t c = 0; c < nchunks; ++c) {
        a.tile0 = (int)(c * chunk);
        a.tile1 = (int)std::min<int64_t>(ntiles, (c + 1) * chunk);
        a.first = c == 0;
        a.last = c == nchunks - 1;
        if ((e = launch_tc<false>(o.dk, o.mq, o.mx, a, st)) != cudaSuccess) return e;
    }
    if (S > 1) {
        const size_t smem = (size_t)8 * 5 * KL * sizeof(uint64_t);
        if ((e = cudaFuncSetAttribute(knn_merge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
            cudaSuccess)
            return e;
        const int64_t blocks = std::min<int64_t>(l.nq, (int64_t)sm_count() * 16);
        knn_merge_kernel<<<(unsigned)blocks, 256, smem, st>>>(a.ids, a.d2, l.nq, S, KL, idsout, d2out);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return knn_finish(o, st);  // scratch is freed on return
}

cudaError_t knn_finish(const KnnOperands &o, cudaStream_t st) {
    int failed = 0;
    cudaError_t e = cudaMemcpyAsync(&failed, o.err, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e == cudaSuccess && failed ? cudaErrorLaunchTimeout : e;
}

int64_t knn_chunk_tiles(int dk) {
    if (const char *ct = getenv("NSG_KNN_CHUNK_TILES"))
        if (atoi(ct) > 0) return atoi(ct);
    return std::max<int64_t>(1, (int64_t(48) << 20) / ((int64_t)TC_N * dk * 2));
}

// Tensor-core kNN when the data allows an exact answer (integer 0..255,
// d <= 128, k <= 256); *used = 0 when it does not apply (nothing written).
cudaError_t launch_knn_tc(const KnnLaunch &l, int *used, cudaStream_t st) {
    *used = 0;
    if (l.nq <= 0 || l.k > TC_MAXK || l.dp > 1024 || !encode_fn()) return cudaSuccess;
    const int dk = l.dp <= 64 ? 64 : (l.dp <= 128 ? 128 : (l.dp + 63) / 64 * 64);
    const int64_t ntiles = (l.n + TC_N - 1) / TC_N;
    if (ntiles > INT32_MAX / TC_N) return cudaSuccess;
    const int64_t npad = ntiles * TC_N;
    KnnScratch<__nv_bfloat16> xb, qb;
    KnnScratch<float> xn, qn;
    KnnScratch<int> flag;
    cudaError_t e;
    if ((e = xb.alloc((size_t)l.n * dk)) != cudaSuccess) return e;
    if ((e = xn.alloc((size_t)npad)) != cudaSuccess) return e;
    if ((e = flag.alloc(2)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(flag.p, 0, 2 * sizeof(int), st)) != cudaSuccess) return e;
    const int grid_rows = sm_count() * 8;
    bf16_rows_kernel<<<grid_rows, 256, 0, st>>>(reinterpret_cast<const float4 *>(l.base), l.n, l.dp / 4,
                                                reinterpret_cast<uint2 *>(xb.p), dk / 4, xn.p, npad, flag.p);
    KnnOperands o;
    o.xn = xn.p;
    const __nv_bfloat16 *qsrc = xb.p + (l.self_join ? l.q0 * dk : 0);
    o.qn = xn.p + (l.self_join ? l.q0 : 0);
    o.dk = dk;
    o.ntiles = ntiles;
    o.err = flag.p + 1;
    if (!l.self_join) {
        if ((e = qb.alloc((size_t)l.nq * dk)) != cudaSuccess) return e;
        if ((e = qn.alloc((size_t)l.nq)) != cudaSuccess) return e;
        bf16_rows_kernel<<<grid_rows, 256, 0, st>>>(reinterpret_cast<const float4 *>(l.queries), l.nq, l.dp / 4,
                                                    reinterpret_cast<uint2 *>(qb.p), dk / 4, qn.p, l.nq, flag.p);
        qsrc = qb.p;
        o.qn = qn.p;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    int other = 0;
    if ((e = cudaMemcpyAsync(&other, flag.p, sizeof(int), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    // Integer data 0..255 with d <= 128: the GEMM-form distances are exact and
    // the k best lists are the answer.  Otherwise (float data, or wider rows
    // whose integer sums may pass 2^24) the GEMM keeps the KL = k + margin best
    // candidates by its BF16 distance and an exact FP32 re-rank picks the k.
    const bool exact = !other && dk <= 128;
    o.KL = exact ? l.k : std::min(l.k + std::max(l.k / 2, 32), TC_MAXK);
    if (!exact && o.KL < l.k + 16) return cudaSuccess;  // no room for a margin: exact scan instead
    if (!make_map(&o.mq, qsrc, l.self_join ? l.n - l.q0 : l.nq, dk) || !make_map(&o.mx, xb.p, l.n, dk))
        return cudaSuccess;
    // the rows' sorted lists live in the output arrays (exact) or in scratch
    // (candidates); distances are kept even when the caller asked for ids only
    KnnScratch<float> d2s;
    KnnScratch<int> ids_s;
    float *d2out = l.d2;
    int *idsout = l.ids;
    if (!exact) {
        if ((e = ids_s.alloc((size_t)l.nq * o.KL)) != cudaSuccess) return e;
        idsout = ids_s.p;
    }
    if (!exact || !d2out) {
        if ((e = d2s.alloc((size_t)l.nq * o.KL)) != cudaSuccess) return e;
        d2out = d2s.p;
    }
    const bool bounded = knn_sample_tiles(ntiles, o.KL + (l.self_join ? 1 : 0)) > 0;
    bool small = knn_small(l.n, l.nq, o.KL, bounded, sm_count());
    if (const char *env = getenv("NSG_KNN_ENGINE")) {  // one of the kernels (tests)
        if (strcmp(env, "small") == 0) small = true;
        else if (strcmp(env, "units") == 0) small = false;
    }
    if (!small) {
        e = select_units(l, o, idsout, d2out, st);
        if (e == cudaErrorMemoryAllocation) {  // up to 1 GB of minima, splits' lists, rings: do without
            cudaGetLastError();
            small = true;
        }
    }
    if (small) e = knn_select_small(l, o, idsout, d2out, st);
    if (e != cudaSuccess) return e;
    if (!exact) {
        if ((e = launch_knn_rerank(l, idsout, o.KL, st)) != cudaSuccess) return e;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;  // scratch is freed on return
    }
    *used = 1;
    return cudaSuccess;
}

}  // namespace nsg
