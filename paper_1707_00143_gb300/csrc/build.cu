// build.cu -- Alg. 2 kernels other than the per-node search: centroid,
// navigating node, MRNG edge selection, reachability BFS helpers of the
// connectivity pass (the pass itself is in connect.cu); plus the
// precision count (Eq. 1) and a row-padding copy.
#include <climits>

#include "kernels.h"
#include "lowp.cuh"

namespace nsg {

__host__ __device__ static inline int round32(int x) { return (x + 31) & ~31; }

template <typename T>
__device__ __forceinline__ T ld_volatile(const T *p) {
    return *reinterpret_cast<const volatile T *>(p);
}

// ---------------------------------------------------------------------------
// Centroid (Alg. 2, first step): block b sums rows [b*rows, (b+1)*rows) of every
// column in FP64 (row order), then one pass adds the block sums in block order
// and divides by n.  On integer data every partial sum is exact.
// ---------------------------------------------------------------------------
__global__ void centroid_partial_kernel(const float *__restrict__ base, int64_t n, int d,
                                        int64_t rows, double *__restrict__ partial) {
    const int64_t r0 = (int64_t)blockIdx.x * rows;
    const int64_t r1 = r0 + rows < n ? r0 + rows : n;
    for (int j = threadIdx.x; j < d; j += blockDim.x) {
        double s = 0.0;
        for (int64_t r = r0; r < r1; ++r) s = __dadd_rn(s, (double)__ldg(base + r * d + j));
        partial[(int64_t)blockIdx.x * d + j] = s;
    }
}

__global__ void centroid_final_kernel(const double *__restrict__ partial, int nb, int d, int64_t n,
                                      double *__restrict__ c) {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < d; j += gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int b = 0; b < nb; ++b) s = __dadd_rn(s, partial[(int64_t)b * d + j]);
        c[j] = __ddiv_rn(s, (double)n);
    }
}

cudaError_t launch_centroid(const float *base, int64_t n, int d, double *partial, int nblocks,
                            double *c, cudaStream_t st) {
    int64_t rows = (n + nblocks - 1) / nblocks;
    int nb = (int)((n + rows - 1) / rows);
    int threads = d < 256 ? round32(d) : 256;
    centroid_partial_kernel<<<nb, threads, 0, st>>>(base, n, d, rows, partial);
    centroid_final_kernel<<<(d + 255) / 256, 256, 0, st>>>(partial, nb, d, n, c);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Navigating node (Alg. 2; Section 3.5 ii): Alg. 1 on the kNN graph from `start`
// toward the centroid, one block.  Distances are FP64 sums over j in order with
// explicitly rounded operations (no FMA), so they do not depend on the
// compiler.
//
// One search is a chain of steps, so a step's latency is what counts.  Up to
// NAV_ROWS neighbours at a time, the block reads tiles of NAV_TILE values of
// all their rows (coalesced) and leaves the rounded squares in shared memory;
// the first warps add a row's squares in order, one row per thread, while the
// others fill the next tile; and the new keys enter the sorted pool by rank,
// from one buffer into the other.  Bound by the chain of steps (~60 of ~7 us)
// and the SM's few FP64 units.  One warp with a lane per row and lane 0
// inserting took 1.65 ms for 100,000 SIFT-shaped rows (K = 100, L = 40,
// centroid included; now 0.55), 0.86 ms for DEEP-shaped (now 0.35), 0.57 ms
// for 10,000 x 32 (now 0.26).
// ---------------------------------------------------------------------------
constexpr int NAV_THREADS = 512, NAV_ROWS = 128, NAV_TILE = 64, NAV_PITCH = NAV_TILE + 1;

__device__ __forceinline__ bool dkey_less(double da, int ia, double db, int ib) {
    return da < db || (da == db && ia < ib);
}
// the same order on the bits of distances >= +0 that are no NaN
__device__ __forceinline__ bool bkey_less(uint64_t a, int ia, uint64_t b, int ib) {
    return a < b || (a == b && ia < ib);
}

struct NavShared {
    int warp_new[NAV_ROWS / 32];
    int at, u;
    uint64_t ck[NAV_ROWS];  // the new nodes' distances (bits) and ids
    int ci[NAV_ROWS];
};

__host__ __device__ inline size_t nav_smem_bytes(int d, int L) {
    return 8ull * (d + 2 * NAV_ROWS * NAV_PITCH + 2 * (size_t)L) + 4ull * 2 * (size_t)L;
}

__global__ void __launch_bounds__(NAV_THREADS) navigate_kernel(const float *__restrict__ base, int d,
                                                               const int *__restrict__ knn, int K,
                                                               const double *__restrict__ cg, int start, int L,
                                                               uint32_t *visited, int max_steps, int *nav_out,
                                                               int *status) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ NavShared sh;
    double *c = reinterpret_cast<double *>(smem);
    double *tile = c + d;                                                             // two of NAV_ROWS rows
    uint64_t *pk = reinterpret_cast<uint64_t *>(tile + 2 * NAV_ROWS * NAV_PITCH);     // two pools of L
    int *pi = reinterpret_cast<int *>(pk + 2 * (size_t)L);                            // ids, bit 31 = checked
    const int t = threadIdx.x, lane = t & 31;
    const int tiles = (d + NAV_TILE - 1) / NAV_TILE;
    for (int j = t; j < d; j += NAV_THREADS) c[j] = cg[j];
    if (t == 0) {
        atomicOr(visited + (start >> 5), 1u << (start & 31));
        sh.ci[0] = start;
    }
    __syncthreads();
    // squares of tile i of the rows sh.ci[0..m) by threads f0..NAV_THREADS-1
    auto fill = [&](int i, int m, int f0) {
        double *out = tile + (i & 1) * NAV_ROWS * NAV_PITCH;
        const int j0 = i * NAV_TILE, w = min(NAV_TILE, d - j0);
#pragma unroll 4
        for (int e = t - f0; e < m * NAV_TILE; e += NAV_THREADS - f0) {
            const int r = e / NAV_TILE, jj = e % NAV_TILE;
            if (jj < w) {
                const double x = __dsub_rn((double)__ldg(base + (int64_t)sh.ci[r] * d + j0 + jj), c[j0 + jj]);
                out[r * NAV_PITCH + jj] = __dmul_rn(x, x);
            }
        }
    };
    // distances of the rows sh.ci[0..m) into sh.ck; whether one of them is a NaN
    auto measure = [&](int m) -> bool {
        double s = 0.0;
        fill(0, m, 0);
        __syncthreads();
        for (int i = 0; i < tiles; ++i) {
            if (t >= NAV_ROWS) {
                if (i + 1 < tiles) fill(i + 1, m, NAV_ROWS);
            } else if (t < m) {
                const double *row = tile + (i & 1) * NAV_ROWS * NAV_PITCH + t * NAV_PITCH;
                const int w = min(NAV_TILE, d - i * NAV_TILE);
#pragma unroll 8
                for (int jj = 0; jj < w; ++jj) s = __dadd_rn(s, row[jj]);
            }
            __syncthreads();
        }
        if (t < m) sh.ck[t] = (uint64_t)__double_as_longlong(s);
        return __syncthreads_or(t < m && s != s) != 0;
    };
    // NaN distances have no order: the pool is then kept by insertion, one node after the other
    bool serial = measure(1);
    if (t == 0) {
        pk[0] = sh.ck[0];
        pi[0] = start;
    }
    __syncthreads();
    int size = 1, cur = 0, steps = 0;
    bool capped = false;
    for (;;) {
        int *ids = pi + cur * L;
        if (t < 32) {  // the first unchecked entry
            int at = -1;
            for (int b = 0; b < size && at < 0; b += 32) {
                const unsigned bal = __ballot_sync(NSG_FULL, b + lane < size && ids[b + lane] >= 0);
                if (bal) at = b + __ffs(bal) - 1;
            }
            if (lane == 0) {
                sh.at = at;
                if (at >= 0) sh.u = ids[at];
            }
        }
        __syncthreads();
        const int at = sh.at, u = sh.u;
        if (at < 0) break;
        if (steps >= max_steps) {
            capped = true;
            break;
        }
        ++steps;
        if (t == 0) ids[at] |= INT_MIN;
        for (int b = 0; b < K; b += NAV_ROWS) {
            int w = -1, rank = 0;
            if (t < NAV_ROWS) {
                if (b + t < K) w = __ldg(knn + (int64_t)u * K + b + t);
                if (w >= 0) {
                    const uint32_t bit = 1u << (w & 31);
                    if (atomicOr(visited + (w >> 5), bit) & bit) w = -1;
                }
                const unsigned bal = __ballot_sync(NSG_FULL, w >= 0);
                rank = __popc(bal & lanemask_lt());
                if (lane == 0) sh.warp_new[t >> 5] = __popc(bal);
            }
            __syncthreads();
            int m = 0;
#pragma unroll
            for (int x = 0; x < NAV_ROWS / 32; ++x) {
                if (x < (t >> 5)) rank += sh.warp_new[x];
                m += sh.warp_new[x];
            }
            if (w >= 0) sh.ci[rank] = w;
            __syncthreads();
            if (m == 0) continue;
            if (measure(m)) serial = true;
            uint64_t *k0 = pk + cur * L;
            int *i0 = pi + cur * L;
            if (!serial) {
                uint64_t *k1 = pk + (cur ^ 1) * L;
                int *i1 = pi + (cur ^ 1) * L;
                for (int x = t; x < NAV_ROWS + size; x += NAV_THREADS) {
                    const bool fresh = x < NAV_ROWS;
                    if (fresh && x >= m) continue;
                    const uint64_t k = fresh ? sh.ck[x] : k0[x - NAV_ROWS];
                    const int tag = fresh ? sh.ci[x] : i0[x - NAV_ROWS], id = tag & INT_MAX;
                    int pos = x - NAV_ROWS;  // pool entries smaller than it
                    if (fresh) {
                        int lo = 0, hi = size;
                        while (lo < hi) {
                            const int mid = (lo + hi) >> 1;
                            if (bkey_less(k0[mid], i0[mid] & INT_MAX, k, id)) lo = mid + 1;
                            else hi = mid;
                        }
                        pos = lo;
                    }
                    for (int y = 0; y < m; ++y) pos += bkey_less(sh.ck[y], sh.ci[y], k, id);
                    if (pos < L) {
                        k1[pos] = k;
                        i1[pos] = tag;
                    }
                }
                cur ^= 1;
            } else if (t == 0) {
                int sz = size;
                for (int x = 0; x < m; ++x) {
                    const double dv = __longlong_as_double((long long)sh.ck[x]);
                    const int iv = sh.ci[x];
                    auto before = [&](int p) {
                        return dkey_less(dv, iv, __longlong_as_double((long long)k0[p]), i0[p] & INT_MAX);
                    };
                    if (sz == L && !before(L - 1)) continue;
                    int pos = sz < L ? sz : L - 1;
                    while (pos > 0 && before(pos - 1)) {
                        k0[pos] = k0[pos - 1];
                        i0[pos] = i0[pos - 1];
                        --pos;
                    }
                    k0[pos] = sh.ck[x];
                    i0[pos] = iv;
                    if (sz < L) ++sz;
                }
            }
            size = min(L, size + m);
            __syncthreads();
        }
    }
    if (t == 0) {
        *nav_out = pi[cur * L] & INT_MAX;
        *status = capped ? -4 : 0;
    }
}

cudaError_t launch_navigate(const float *base, int64_t n, int d, const int *knn, int K,
                            const double *c, int start, int L, uint32_t *visited_bits,
                            int max_steps, int *nav_out, int *status, cudaStream_t st) {
    (void)n;
    const size_t smem = nav_smem_bytes(d, L);
    cudaError_t e = cudaFuncSetAttribute(navigate_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    navigate_kernel<<<1, NAV_THREADS, smem, st>>>(base, d, knn, K, c, start, L, visited_bits, max_steps,
                                                  nav_out, status);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// MRNG edge selection (Alg. 2; Section 3.3), one warp per node.  Candidates are
// already sorted by key; the first is kept; a later candidate p is occluded
// when d2(p, r) < d2(p, v) for a kept r (r in the open lune of vp); stop at R.
//
// The warp takes the candidates in batches of NB = (32 / G) * B: each G-lane
// group holds B candidate rows in registers (batch position b * (32/G) + grp).
// The kept rows are read once per batch, U at a time, and every group measures
// them against its B candidates; the pass ends early once every candidate of
// the batch is occluded.  The survivors are then taken in candidate order:
// the first is kept, and the later survivors are measured against it (the
// kept set a sequential scan would have at their turn), and so on.  Results,
// and the count of candidates examined, equal the one-at-a-time scan.
// ---------------------------------------------------------------------------
struct PruneArgs {
    ExactRows rows;
    const int *cand_ids;
    const float *cand_d2;
    const int *cand_count;
    int C, R, Wr;
    int64_t v0, nv;
    int *adj, *deg;
    unsigned long long *examined;
};

// Batch positions (b * P + g) whose flag is set in group g's lane 0, as a mask.
template <int G, int B>
__device__ __forceinline__ unsigned batch_mask(const bool (&f)[B]) {
    constexpr int P = 32 / G;
    const bool lead = lane_id() % G == 0;
    unsigned m = 0;
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const unsigned bal = __ballot_sync(NSG_FULL, lead && f[b]);
#pragma unroll
        for (int g = 0; g < P; ++g) m |= ((bal >> (g * G)) & 1u) << (b * P + g);
    }
    return m;
}

// Rows as the selection holds them, a slice per lane of a G-lane group.
template <int G_, int V>
struct PruneF32 {
    static constexpr int G = G_;
    struct Reg {
        float4 v[V];
    };
    static __device__ __forceinline__ Reg load(const ExactRows &r, int64_t id, bool valid) {
        const float4 *row = r.base4 + id * r.dp4;
        Reg x;
#pragma unroll
        for (int w = 0; w < V; ++w) {
            const int k = w * G + (int)lane_id() % G;
            x.v[w] = (valid && k < r.dp4) ? __ldg(row + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        return x;
    }
    static __device__ __forceinline__ float dist(const Reg &x, const Reg &q) {
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < V; ++w) s += sq4(x.v[w], q.v[w]);
        return group_sum<G>(s);
    }
};

template <int G_, int VC>
struct PruneU8 {
    static constexpr int G = G_;
    struct Reg {
        uint4 v[VC];
    };
    static __device__ __forceinline__ Reg load(const ExactRows &r, int64_t id, bool valid) {
        const uint4 *row = r.u8 + id * r.dc;
        Reg x;
#pragma unroll
        for (int w = 0; w < VC; ++w) {
            const int k = w * G + (int)lane_id() % G;
            x.v[w] = (valid && k < r.dc) ? __ldg(row + k) : make_uint4(0, 0, 0, 0);
        }
        return x;
    }
    static __device__ __forceinline__ float dist(const Reg &x, const Reg &q) {
        unsigned s = 0;
#pragma unroll
        for (int w = 0; w < VC; ++w) {
            unsigned e = __vabsdiffu4(x.v[w].x, q.v[w].x);
            s = __dp4a(e, e, s);
            e = __vabsdiffu4(x.v[w].y, q.v[w].y);
            s = __dp4a(e, e, s);
            e = __vabsdiffu4(x.v[w].z, q.v[w].z);
            s = __dp4a(e, e, s);
            e = __vabsdiffu4(x.v[w].w, q.v[w].w);
            s = __dp4a(e, e, s);
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) s += __shfl_xor_sync(NSG_FULL, s, o, G);
        return (float)s;
    }
};

template <class Row, int U, int B>
__device__ __forceinline__ void prune_body(const PruneArgs &a) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int G = Row::G;
    constexpr int P = 32 / G, NB = P * B;
    static_assert(NB <= 32, "batch mask holds 32 positions");
    const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int lane = (int)lane_id(), grp = lane / G;
    int *kept = reinterpret_cast<int *>(smem) + (size_t)warp * a.Wr;
    const int64_t stride = (int64_t)gridDim.x * wpb;
    unsigned long long examined = 0;
    for (int64_t j = (int64_t)blockIdx.x * wpb + warp; j < a.nv; j += stride) {
        const int64_t v = a.v0 + j;
        const int *ci = a.cand_ids + j * a.C;
        const float *cd = a.cand_d2 + j * a.C;
        int cnt = a.cand_count != nullptr ? min(max(a.cand_count[j], 0), a.C) : a.C;
        if (cnt > 0 && ci[0] < 0) cnt = 0;  // a negative id ends the list
        int nk = 0, t = 0;                  // kept; candidates examined
        if (cnt > 0) {
            if (lane == 0) kept[0] = ci[0];
            nk = 1;
            t = 1;
        }
        __syncwarp();
        while (t < cnt && nk < a.R) {
            typename Row::Reg q[B];
            float pdv[B];
            bool occ[B];
            int id[B];
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int c = t + b * P + grp;
                id[b] = c < cnt ? ci[c] : 0;
                occ[b] = id[b] < 0;
            }
            const unsigned neg = batch_mask<G, B>(occ);
            if (neg) cnt = t + __ffs(neg) - 1;  // a negative id ends the list
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int c = t + b * P + grp;
                const bool valid = c < cnt;
                pdv[b] = valid ? cd[c] : 0.0f;
                occ[b] = !valid;
                q[b] = Row::load(a.rows, valid ? id[b] : 0, valid);
            }
            // against the kept set as it was before the batch
            for (int i0 = 0; i0 < nk; i0 += U) {
                bool all = true;
#pragma unroll
                for (int b = 0; b < B; ++b) all &= occ[b];
                if (__all_sync(NSG_FULL, all)) break;
                typename Row::Reg x[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = i0 + u;
                    x[u] = Row::load(a.rows, i < nk ? kept[i] : 0, i < nk);
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int b = 0; b < B; ++b) {
                        const float s = Row::dist(x[u], q[b]);
                        if (i0 + u < nk && s < pdv[b]) occ[b] = true;
                    }
            }
            // survivors in candidate order, each measured against the ones kept before it
            bool live_f[B];
#pragma unroll
            for (int b = 0; b < B; ++b) live_f[b] = !occ[b];
            unsigned live = batch_mask<G, B>(live_f);
            int stop = -1;
            while (live) {
                const int pos = __ffs(live) - 1;
                live &= live - 1u;
                const int pj = ci[t + pos];
                if (lane == 0) kept[nk] = pj;
                ++nk;
                if (nk == a.R) {
                    stop = pos;
                    break;
                }
                if (!live) break;
                const typename Row::Reg x = Row::load(a.rows, pj, true);
                bool hit[B];
#pragma unroll
                for (int b = 0; b < B; ++b) hit[b] = Row::dist(x, q[b]) < pdv[b];
                live &= ~batch_mask<G, B>(hit);
            }
            __syncwarp();
            t = stop >= 0 ? t + stop + 1 : min(t + NB, cnt);
        }
        examined += (unsigned long long)t;
        for (int e = lane; e < a.R; e += 32) a.adj[v * a.R + e] = e < nk ? kept[e] : -1;
        if (lane == 0) a.deg[v] = nk;
        __syncwarp();
    }
    if (a.examined != nullptr && lane == 0 && examined) atomicAdd(a.examined, examined);
}

// Rows of up to 4 float4s per lane run 3 blocks per SM (78 registers, no
// spills; 8 % faster than 2 blocks on 128-value rows); wider rows keep the
// compiler's own budget (at 3 blocks they spill and run 1.8x slower).
template <class Row, int U, int B>
__global__ void __launch_bounds__(256) prune_kernel(PruneArgs a) {
    prune_body<Row, U, B>(a);
}
template <class Row, int U, int B>
__global__ void __launch_bounds__(256, 3) prune_narrow_kernel(PruneArgs a) {
    prune_body<Row, U, B>(a);
}
template <class Row, int U, int B>
__global__ void __launch_bounds__(256, 3) prune_u8_kernel(PruneArgs a) {
    prune_body<Row, U, B>(a);
}

// Candidate rows held per lane group: two while they fit in 32 float4s.  8-bit
// rows take a quarter of the lanes, loads and arithmetic, so a batch is up to
// 32 candidates: four per group of four or more lanes.  100,000 SIFT-shaped
// rows (R = 50, C = 500): FP32 7.17 ms; 8-bit 3.48 ms with one, 2.85 with two,
// 2.61 with four (4 blocks per SM: 2.92 with two, 2.74 with four; 4 kept rows
// at a time instead of 2: 3.08).
template <int G, int V, int U>
void (*prune_entry(bool u8))(PruneArgs) {
    if constexpr (V > 4) {  // no 8-bit copy at these widths
        return prune_kernel<PruneF32<G, V>, U, V <= 8 ? 2 : 1>;
    } else {
        using S = Exact8Shape<G, V>;
        if (u8) return prune_u8_kernel<PruneU8<S::lanes, S::chunks>, U, S::lanes < 4 ? S::lanes : 4>;
        return prune_narrow_kernel<PruneF32<G, V>, U, 2>;
    }
}

cudaError_t launch_prune(const PruneLaunch &l, cudaStream_t st) {
    if (l.nv <= 0) return cudaSuccess;
    PruneArgs a;
    a.rows = ExactRows{reinterpret_cast<const float4 *>(l.base), l.dp / 4, reinterpret_cast<const uint4 *>(l.u8.rows),
                       l.u8.chunks, l.u8.d, l.u8.lo};
    a.cand_ids = l.cand_ids;
    a.cand_d2 = l.cand_d2;
    a.cand_count = l.cand_count;
    a.C = l.C;
    a.R = l.R;
    a.Wr = round32(l.R);
    a.v0 = l.v0;
    a.nv = l.nv;
    a.adj = l.adj;
    a.deg = l.deg;
    a.examined = l.examined;
    const int wpb = 8;
    size_t smem = (size_t)wpb * a.Wr * 4;
    cudaError_t err = cudaSuccess;
    NSG_DISPATCH_DP4(a.rows.dp4, {
        void (*kern)(PruneArgs) = prune_entry<G_, V_, U_>(a.rows.u8 != nullptr);
        err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (err == cudaSuccess) {
            int per_sm = 0;
            err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, wpb * 32, smem);
            if (err == cudaSuccess) {
                int64_t need = (l.nv + wpb - 1) / wpb;
                int64_t full = (int64_t)sm_count() * (per_sm > 0 ? per_sm : 1);
                int grid = (int)(need < full ? need : full);
                kern<<<grid, wpb * 32, smem, st>>>(a);
                err = cudaGetLastError();
            }
        }
    });
    return err;
}

// ---------------------------------------------------------------------------
// Reachability from the navigating node: level-synchronous BFS over the
// fixed-width graph (the reached set equals that of the paper's DFS tree).
// ---------------------------------------------------------------------------
__global__ void bfs_seed_kernel(uint32_t *reached, int root, int *frontier, int *count) {
    atomicOr(reached + (root >> 5), 1u << (root & 31));
    frontier[0] = root;
    *count = 1;
}

// One level: the frontier's size *nf is read on the device, so levels are
// enqueued back to back without the host in between.
__global__ void bfs_level_kernel(const int *__restrict__ adj, int R, const int *__restrict__ frontier,
                                 const int *nf, int *next, int *next_count, uint32_t *reached) {
    const int64_t total = (int64_t)*nf * R;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x) {
        int u = frontier[x / R];
        int v = adj[(int64_t)u * R + x % R];
        if (v < 0) continue;
        uint32_t bit = 1u << (v & 31);
        if (!(atomicOr(reached + (v >> 5), bit) & bit)) next[atomicAdd(next_count, 1)] = v;
    }
}

cudaError_t launch_bfs_seed(uint32_t *reached, int root, int *frontier, int *count, cudaStream_t st) {
    bfs_seed_kernel<<<1, 1, 0, st>>>(reached, root, frontier, count);
    return cudaGetLastError();
}

cudaError_t launch_bfs_level(const int *adj, int R, const int *frontier, const int *nf, int *next,
                             int *next_count, uint32_t *reached, cudaStream_t st) {
    bfs_level_kernel<<<sm_count() * 8, 256, 0, st>>>(adj, R, frontier, nf, next, next_count, reached);
    return cudaGetLastError();
}

__global__ void fill_kernel(int *p, int64_t n, int v) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x)
        p[x] = v;
}

cudaError_t launch_fill(int *p, int64_t n, int v, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const int64_t blocks = (n + 255) / 256, cap = (int64_t)sm_count() * 8;
    fill_kernel<<<(int)(blocks < cap ? blocks : cap), 256, 0, st>>>(p, n, v);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Precision (Eq. 1): per query, how many of the first k ids are among the
// first k ground-truth ids.
// ---------------------------------------------------------------------------
__global__ void recall_kernel(const int *__restrict__ ids, int ld_ids, const int *__restrict__ gt,
                              int ld_gt, int64_t nq, int k, int *hits) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nq;
         q += (int64_t)gridDim.x * blockDim.x) {
        int h = 0;
        for (int a = 0; a < k; ++a) {
            int id = ids[q * ld_ids + a];
            if (id < 0) continue;
            for (int b = 0; b < k; ++b)
                if (gt[q * ld_gt + b] == id) {
                    ++h;
                    break;
                }
        }
        hits[q] = h;
    }
}

cudaError_t launch_recall(const int *ids, int ld_ids, const int *gt, int ld_gt, int64_t nq, int k,
                          int *hits, cudaStream_t st) {
    if (nq <= 0) return cudaSuccess;
    int64_t blocks = (nq + 255) / 256;
    recall_kernel<<<(int)(blocks < 65535 ? blocks : 65535), 256, 0, st>>>(ids, ld_ids, gt, ld_gt, nq,
                                                                           k, hits);
    return cudaGetLastError();
}

__global__ void pad_rows_kernel(const float *__restrict__ src, int64_t n, int d, float *__restrict__ dst,
                                int dp) {
    const int64_t total = n * dp;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = x / dp;
        int c = (int)(x % dp);
        dst[x] = c < d ? src[r * d + c] : 0.0f;
    }
}

cudaError_t launch_pad_rows(const float *src, int64_t n, int d, float *dst, int dp, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    int64_t blocks = (n * dp + 255) / 256;
    int64_t cap = (int64_t)sm_count() * 16;
    pad_rows_kernel<<<(int)(blocks < cap ? blocks : cap), 256, 0, st>>>(src, n, d, dst, dp);
    return cudaGetLastError();
}

}  // namespace nsg
