// connect.cu -- the connectivity pass of Alg. 2 (Section 3.5 iv).
//
// Sequential definition (what the oracle computes): reach from the
// navigating node; while some node is unreached, u = the smallest unreached
// id, run Alg. 1 on the current graph from the navigating node toward x_u,
// give the first result with a free slot (else the smallest reached id with
// one) the edge s->u, and mark everything u reaches.
//
// GPU form, identical result, batch by batch:
//   list     the next B unreached ids in ascending order (one CTA);
//   label    every unreached node gets the smallest list position that reaches
//            it through unreached nodes (label-correcting BFS, a few levels over
//            the whole GPU, what is left by one CTA).  New edges start at reached nodes, so
//            nothing a batch adds changes this: listed id j is a fix-up exactly
//            when its label is j, and when the fix-ups before position j are
//            made, the nodes labelled below j are reached;
//   rounds   fix-up f's search depends on the edges s_i -> u_i proposed by the
//            fix-ups i < f.  Every round, one warp per fix-up runs Alg. 1 on the
//            graph with the proposals of earlier fix-ups (GraphView hides the
//            later ones) -- in the first round for all, then only where a changed
//            proposal could have changed it -- and picks its s with the degrees
//            that view gives; then one CTA finds sources for those whose pools
//            have no room, collects the proposals, sorts them by
//            (source, fix-up) and writes them past the rows' degrees.  Fix-up 0
//            depends on nothing, and once the fix-ups before f stand still, f is
//            final after one more round: whatever precedes the first proposal
//            that changed in a round is the sequential loop's choice;
//   commit   the final prefix (all of the batch, once a round changed nothing)
//            becomes part of the graph and the next list starts after it.
// A changed edge e->w can matter to f's search only if e was expanded and w
// entered (or could enter) the pool then: the pool was not yet full, or key(w)
// was below its L-th key at that expansion.  Once the pool is full its L-th
// key never rises, so a w that could not enter at e's expansion can never
// enter later either, and the pool is unchanged.  The search logs, per
// expansion, the node and that entry bar; the check uses a relative slack of
// 2^-10 on the distance, so summation-order rounding can only cause an extra
// search.
//
// Bound by latency: a search is a chain of ~60 dependent expansions, so what
// counts is how many fix-ups one chain's time serves.  Before, one CTA walked
// the batch in order with ~10 dependent round trips to memory per fix-up and
// repeated a stale search alone.  Measured (whole build, before -> after):
// 10,000 x 32 16.9 -> 5.4 ms, 100,000 x 128 115.6 -> 58.9 ms, 150,000 x 96 on
// an nn-descent graph 106.4 -> 51.8 ms (the pass itself 66 -> 4, 65 -> 5 and
// 68 -> 8 ms).  With the exact 8-bit copy of integer rows (one round of gathers
// per expansion instead of three or four) and the largest visited set that
// fits, the pass takes 2.8, 3.2 and 6.2 ms of 2.9, 3.9 and 6.4 before.
#include <climits>
#include <vector>

#include "kernels.h"
#include "lowp.cuh"

#ifndef NSG_CONNECT_U_WIDE8
#define NSG_CONNECT_U_WIDE8 4  // rows in flight per warp, 513..1024-value rows
#endif

namespace nsg {

namespace {

constexpr int CONNECT_FIRST_BATCH = 1024;
constexpr int CONNECT_MIN_BATCH = 64;
constexpr int CONNECT_MAX_BATCH = 4096;  // 2 sort entries per fix-up in 64 KB of shared memory
constexpr int CONNECT_ROUNDS = 8;        // rounds enqueued per batch (they end early when settled)
constexpr int LABEL_LEVELS = 10;         // label levels run by the whole GPU before one CTA finishes

__host__ __device__ inline int round32c(int x) { return (x + 31) & ~31; }
inline int log2c(unsigned x) {
    int r = 0;
    while ((1u << r) < x) ++r;
    return r;
}

template <typename T>
__device__ __forceinline__ T ldv(const T *p) {
    return *reinterpret_cast<const volatile T *>(p);
}

__device__ __forceinline__ bool bit_is_set(const uint32_t *bits, int64_t x) {
    return (ldv(bits + (x >> 5)) >> (x & 31)) & 1u;
}

// State of the pass on the device.
struct FixState {
    long long cursor;    // every id below it is reached
    int cnt, last;       // ids listed, the last one
    int F, touched;      // fix-ups among them, nodes labelled
    int nent;            // sorted edge entries of the last round
    int settled;         // the proposals stand still (up to jfirst / none)
    int jfirst, none;    // first fix-up whose proposal changed; first without one
    int added, status, capped, redone;  // totals of the pass
    int B;                              // ids the next list takes
    int stamp;                          // last label level run
    int room;                           // every id below it is full
    int lev[LABEL_LEVELS + 1];          // queue sizes of this batch's label levels
};

// Edge entries are sorted by (source, fix-up): source << 32 | fix-up << 2 | kind.
constexpr unsigned ENT_CUR = 1;  // a current proposal
constexpr unsigned ENT_CHG = 2;  // proposed or withdrawn in the last round
__device__ __forceinline__ int ent_fix(uint64_t e) { return (int)((uint32_t)e >> 2); }
__device__ __forceinline__ int ent_src(uint64_t e) { return (int)(e >> 32); }

// ids >= cursor that are not reached, ascending, at most B
// (one CTA), and the start of their labels.
__global__ void __launch_bounds__(1024) gather_unreached_kernel(const uint32_t *reached, int64_t n, int *list,
                                                                int *label, int *touched, int *queue, FixState *st) {
    __shared__ int warp_sum[32];
    __shared__ int sh_total;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t nwords = (n + 31) >> 5, cursor = st->cursor;
    const int B = st->B;
    if (tid == 0) sh_total = 0;
    __syncthreads();
    for (int64_t w0 = cursor >> 5; w0 < nwords; w0 += blockDim.x) {
        const int total = sh_total;
        if (total >= B) break;
        const int64_t w = w0 + tid;
        uint32_t miss = 0;
        if (w < nwords) {
            miss = ~ldv(reached + w);
            if (w == nwords - 1 && (n & 31)) miss &= (1u << (n & 31)) - 1u;
            if (w == (cursor >> 5)) miss &= ~((1u << (cursor & 31)) - 1u);
        }
        const int c = __popc(miss);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(NSG_FULL, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        int before = 0, block = 0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
            if (k < warp) before += warp_sum[k];
            block += warp_sum[k];
        }
        int j = total + before + incl - c;
        while (miss && j < B) {
            const int b = __ffs(miss) - 1;
            miss &= miss - 1u;
            list[j++] = (int)(w * 32 + b);
        }
        __syncthreads();
        if (tid == 0) sh_total = total + block;
        __syncthreads();
    }
    const int cnt = sh_total < B ? sh_total : B;
    for (int j = tid; j < cnt; j += blockDim.x) {
        const int u = list[j];
        label[u] = j;
        touched[j] = u;
        queue[j] = u;
    }
    if (tid <= LABEL_LEVELS) st->lev[tid] = tid == 0 ? cnt : 0;
    if (tid == 0) {
        st->cnt = cnt;
        st->last = cnt > 0 ? list[cnt - 1] : -1;
        st->touched = cnt;
    }
}

struct FixArgs {
    ExactRows rows;  // base4, dp4 and the exact 8-bit copy, if any
    const float4 *base4;
    int dp4;
    int64_t n;
    int *adj, *deg;
    int R, W, nav, L, H, hshift, max_steps;
    uint32_t *reached;
    int *label;               // [n] INT_MAX outside a batch
    int *stamp;               // [n] last label level that queued the node
    int bmax;
    int2 *head;               // [n] source -> (first entry, entries); {0, 0} outside a batch
    int *qa, *qb, *touched;   // [n] each
    FixState *st;
    int *list, *fix, *flab;   // [B] listed ids; the fix-ups and their labels
    uint64_t *pools, *xthr;   // [B][L] final pools; [B][xcap] entry bar at each expansion
    int *xlog, *xcnt, *psize; // [B][xcap] expanded nodes; expansions (INT_MAX: the search hit its cap)
    int xcap;
    int *snew, *scur;         // [B] proposed source (-1: nothing has room), this and the last round
    int *used;                // [n] proposals that take a source's slots, 0 between uses
    int *slot, *hold;         // [B] adjacency slot a proposal occupies (-1: none) and what it held
    uint64_t *ent;            // [2 * B]
};

// One node of a label level: its label offered to the unreached nodes it links
// to; a node whose label falls is queued once per level (its stamp).  Warp-wide.
__device__ __forceinline__ void label_node(const FixArgs &a, int node, int stamp, int *nxt, int *ncount) {
    const unsigned lane = lane_id();
    const int l = ldv(a.label + node);
    const int *row = a.adj + (int64_t)node * a.R;
    for (int b = 0; b < a.R; b += 32) {
        const int slot = b + (int)lane;
        const int v = slot < a.R ? row[slot] : -1;
        bool push = false, first = false;
        if (v >= 0 && !bit_is_set(a.reached, v) && ldv(a.label + v) > l) {
            const int old = atomicMin(a.label + v, l);
            first = old == INT_MAX;
            push = old > l && atomicExch(a.stamp + v, stamp) != stamp;
        }
        const unsigned bf = __ballot_sync(NSG_FULL, first), bp = __ballot_sync(NSG_FULL, push);
        int at = 0, an = 0;
        if (lane == 0 && bf) at = atomicAdd(&a.st->touched, __popc(bf));
        if (lane == 0 && bp) an = atomicAdd(ncount, __popc(bp));
        at = __shfl_sync(NSG_FULL, at, 0);
        an = __shfl_sync(NSG_FULL, an, 0);
        if (first) a.touched[at + __popc(bf & lanemask_lt())] = v;
        if (push) nxt[an + __popc(bp & lanemask_lt())] = v;
    }
}

__global__ void __launch_bounds__(256) label_level_kernel(FixArgs a, int level, const int *cur, int *nxt) {
    const int nc = a.st->lev[level], stamp = a.st->stamp + level + 1;
    const int warps = gridDim.x * (blockDim.x >> 5);
    for (int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < nc; i += warps)
        label_node(a, cur[i], stamp, nxt, &a.st->lev[level + 1]);
}

// The label levels that are left, and the list of fix-ups.  One CTA.
__global__ void __launch_bounds__(1024) label_kernel(FixArgs a, int *cur, int *nxt) {
    __shared__ int sh_next, sh_F;
    __shared__ int warp_sum[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x;
    FixState *st = a.st;
    const int cnt = st->cnt;
    int nc = st->lev[LABEL_LEVELS], stamp = st->stamp + LABEL_LEVELS;
    if (tid == 0) sh_F = 0;
    __syncthreads();
    while (nc > 0) {  // ends: every queued node's label fell since it was last queued
        ++stamp;
        if (tid == 0) sh_next = 0;
        __syncthreads();
        for (int i = warp; i < nc; i += nt >> 5) label_node(a, ldv(cur + i), stamp, nxt, &sh_next);
        __syncthreads();
        nc = sh_next;
        __syncthreads();
        int *t = cur;
        cur = nxt;
        nxt = t;
    }
    // fix-ups in list order
    for (int b = 0; b < cnt; b += nt) {
        const int j = b + tid;
        const int u = j < cnt ? a.list[j] : 0;
        const bool is = j < cnt && ldv(a.label + u) == j;
        const unsigned bal = __ballot_sync(NSG_FULL, is);
        if (lane == 0) warp_sum[warp] = __popc(bal);
        __syncthreads();
        int before = sh_F, all = 0;
        for (int k = 0; k < (nt >> 5); ++k) {
            if (k < warp) before += warp_sum[k];
            all += warp_sum[k];
        }
        if (is) {
            const int f = before + __popc(bal & lanemask_lt());
            a.fix[f] = u;
            a.flab[f] = j;
            a.scur[f] = -1;
            a.slot[f] = -1;
        }
        __syncthreads();
        if (tid == 0) sh_F += all;
        __syncthreads();
    }
    if (tid == 0) {
        st->F = sh_F;
        st->stamp = stamp;
        st->nent = 0;
        st->settled = 0;
        st->jfirst = 0;
        st->none = INT_MAX;
    }
}

// Whether a proposal that changed in the last round could have changed fix-up
// f's search.  Warp-wide: a lane per logged expansion walks the entries of its
// node; distances by the whole warp.
__device__ __forceinline__ bool fix_stale(const FixArgs &a, int f, int u) {
    const unsigned lane = lane_id();
    const int xc = a.xcnt[f];
    if (xc > a.xcap) return a.st->jfirst < f;
    const float4 *xu = a.base4 + (int64_t)u * a.dp4;
    for (int b = 0; b < xc; b += 32) {
        const int t = b + (int)lane;
        int p = 0, end = 0;
        float bar = 0.0f;
        bool open = false;  // the pool was not full: any new neighbour entered
        if (t < xc) {
            const int2 h = a.head[a.xlog[(int64_t)f * a.xcap + t]];
            p = h.x;
            end = h.x + h.y;
            if (h.y > 0) {
                const uint64_t thr = a.xthr[(int64_t)f * a.xcap + t];
                open = thr == KEY_INF;
                bar = kd2(thr) * (1.0f + 1.0f / 1024.0f);
            }
        }
        for (;;) {
            int i = -1;  // the lane's next changed edge of an earlier fix-up
            while (p < end && i < 0) {
                const uint64_t e = a.ent[p++];
                if ((e & ENT_CHG) && ent_fix(e) < f) i = ent_fix(e);
            }
            unsigned pend = __ballot_sync(NSG_FULL, i >= 0);
            if (!pend) break;
            if (__any_sync(NSG_FULL, i >= 0 && open)) return true;
            while (pend) {
                const int src = __ffs(pend) - 1;
                pend &= pend - 1u;
                const float4 *xw = a.base4 + (int64_t)a.fix[__shfl_sync(NSG_FULL, i, src)] * a.dp4;
                const float lim = __shfl_sync(NSG_FULL, bar, src);
                float d2 = 0.0f;
                for (int c = (int)lane; c < a.dp4; c += 32) d2 += sq4(__ldg(xu + c), __ldg(xw + c));
                if (!(group_sum<32>(d2) > lim)) return true;  // a NaN on either side: searched again
            }
        }
    }
    return false;
}

// The first of `size` pool entries (key order) with room in fix-up f's view, -1
// if there is none.  Warp-wide.
__device__ __forceinline__ int fix_select(const FixArgs &a, int f, const uint64_t *pool, int size) {
    const unsigned lane = lane_id();
    for (int b = 0; b < size; b += 32) {
        const int t = b + (int)lane;
        int e = -1;
        bool room = false;
        if (t < size) {
            e = kid(pool[t]);
            int d = a.deg[e];
            if (d < a.R) {
                const int2 h = a.head[e];
                if (d + h.y >= a.R)
                    for (int p = h.x; p < h.x + h.y; ++p) {
                        const uint64_t x = a.ent[p];
                        d += (x & ENT_CUR) && ent_fix(x) < f;
                    }
                room = d < a.R;
            }
        }
        const unsigned bal = __ballot_sync(NSG_FULL, room);
        if (bal) return __shfl_sync(NSG_FULL, e, __ffs(bal) - 1);
    }
    return -1;
}

template <int G, int V, int U, bool U8>
__global__ void __launch_bounds__(256) fix_search_kernel(FixArgs a, int round) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const unsigned lane = lane_id();
    if (a.st->settled) return;
    WarpSmem s = carve_warp_smem(smem + warp * warp_smem_bytes(a.L, a.W, 0, a.H, true), a.L, a.W, 0, a.H, true);
    const int F = a.st->F;
    int csize = 0;
    for (int f = blockIdx.x * wpb + warp; f < F; f += gridDim.x * wpb) {
        const int u = a.fix[f];
        uint64_t *pool = a.pools + (int64_t)f * a.L;
        int size;
        if (round == 0 || fix_stale(a, f, u)) {
            SearchOut o;
            with_row_dist<G, V, U, U8>(a.rows, u, [&](const auto &dist) {
                o = warp_alg1<KEYS_POOL>(dist, GraphView{a.adj, a.R, a.deg, a.label, a.flab[f]}, a.nav, a.L, s,
                                         (uint32_t)a.H - 1, a.hshift, a.max_steps, -1, 0, csize,
                                         a.xlog + (int64_t)f * a.xcap, a.xcap, nullptr,
                                         a.xthr + (int64_t)f * a.xcap);
            });
            size = o.size;
            for (int t = lane; t < size; t += 32) pool[t] = s.pool[t];
            if (lane == 0) {
                a.psize[f] = size;
                a.xcnt[f] = o.capped ? INT_MAX : o.n_expand;
                if (round > 0) atomicAdd(&a.st->redone, 1);
            }
            __syncwarp();
            const int sel = fix_select(a, f, s.pool, size);
            if (lane == 0) a.snew[f] = sel;
        } else {
            const int sel = fix_select(a, f, pool, a.psize[f]);
            if (lane == 0) a.snew[f] = sel;
        }
        __syncwarp();
    }
}

// Takes the last round's proposals out of the graph.  Block-wide.
__device__ __forceinline__ void withdraw(const FixArgs &a, int F, int from, int nent) {
    for (int f = from + (int)threadIdx.x; f < F; f += blockDim.x)
        if (a.slot[f] >= 0) a.adj[(int64_t)a.scur[f] * a.R + a.slot[f]] = a.hold[f];
    for (int p = threadIdx.x; p < nent; p += blockDim.x) a.head[ent_src(a.ent[p])] = make_int2(0, 0);
}

// Sources for the fix-ups whose pools have no room: in order, the smallest id
// that is reached when the fix-ups before are made and has a slot that their
// proposals leave.  Block-wide; list [F] in shared memory.  Taken one per batch, at its
// end, they had cost a batch each (20,000 x 16 uniform rows, K = R = 5: the pass 132
// ms; 20,000 x 1,500, R = 24: 894 ms).
__device__ __forceinline__ void fix_fallback(const FixArgs &a, int F, int *list, int *warp_sum, int *found) {
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    int cnt = 0;
    for (int b = 0; b < F; b += nt) {
        const int f = b + tid;
        const bool is = f < F && a.snew[f] < 0;
        const unsigned bal = __ballot_sync(NSG_FULL, is);
        if (lane == 0) warp_sum[warp] = __popc(bal);
        __syncthreads();
        int before = cnt;
        for (int k = 0; k < (nt >> 5); ++k) {
            if (k < warp) before += warp_sum[k];
            cnt += warp_sum[k];
        }
        if (is) list[before + __popc(bal & lanemask_lt())] = f;
        __syncthreads();
    }
    if (cnt == 0) return;
    int prev = 0, room = a.st->room;
    for (int i = 0; i < cnt; ++i) {
        const int f = list[i], lim = a.flab[f];
        for (int g = prev + tid; g < f; g += nt)
            if (ldv(a.snew + g) >= 0) atomicAdd(a.used + ldv(a.snew + g), 1);
        prev = f;
        int sel = INT_MAX;
        bool full = true;  // every id so far
        for (int64_t w0 = room; w0 < a.n && sel == INT_MAX; w0 += nt) {
            if (tid == 0) found[0] = found[1] = INT_MAX;
            __syncthreads();
            const int64_t x = w0 + tid;
            if (x < a.n && a.deg[x] < a.R) {
                atomicMin(found, (int)x);
                if (a.deg[x] + ldv(a.used + x) < a.R && (bit_is_set(a.reached, x) || a.label[x] < lim))
                    atomicMin(found + 1, (int)x);
            }
            __syncthreads();
            const int first = found[0];
            sel = found[1];
            __syncthreads();
            if (full) room = first == INT_MAX ? (int)(w0 + nt < a.n ? w0 + nt : a.n) : first;
            full = full && first == INT_MAX;
        }
        if (sel == INT_MAX) break;  // no room anywhere: the batch ends here
        if (tid == 0) a.snew[f] = sel;
        __syncthreads();
    }
    __syncthreads();
    if (tid == 0) a.st->room = room;
    for (int f = tid; f < F; f += nt)
        if (ldv(a.snew + f) >= 0) a.used[ldv(a.snew + f)] = 0;
    __syncthreads();
}

// The round's proposals against the last round's: entries sorted by source,
// the current ones written past their sources' degrees in fix-up order (the
// slots the sequential loop would give them).  One CTA.
__global__ void __launch_bounds__(1024) fix_propose_kernel(FixArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *ent = reinterpret_cast<uint64_t *>(smem);
    __shared__ int sh_n, sh_first, sh_none, sh_found[2], sh_sum[32];
    FixState *st = a.st;
    const int tid = threadIdx.x, nt = blockDim.x;
    if (st->settled) return;
    const int F = st->F;
    if (tid == 0) {
        sh_n = 0;
        sh_first = INT_MAX;
        sh_none = INT_MAX;
    }
    withdraw(a, F, 0, st->nent);
    __syncthreads();
    fix_fallback(a, F, reinterpret_cast<int *>(smem), sh_sum, sh_found);
    __syncthreads();
    for (int f = tid; f < F; f += nt) {
        const int was = a.scur[f], now = a.snew[f];
        const unsigned chg = was != now ? ENT_CHG : 0u;
        if (now >= 0) ent[atomicAdd(&sh_n, 1)] = ((uint64_t)now << 32) | ((uint32_t)f << 2) | ENT_CUR | chg;
        else atomicMin(&sh_none, f);
        if (chg) {
            if (was >= 0) ent[atomicAdd(&sh_n, 1)] = ((uint64_t)was << 32) | ((uint32_t)f << 2) | ENT_CHG;
            atomicMin(&sh_first, f);
        }
        a.scur[f] = now;
    }
    __syncthreads();
    const int N = sh_n;
    int P2 = 2;
    while (P2 < N) P2 <<= 1;
    for (int p = N + tid; p < P2; p += nt) ent[p] = ~0ull;
    __syncthreads();
    for (int k = 2; k <= P2; k <<= 1)  // bitonic sort
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int x = tid; x < P2 / 2; x += nt) {
                const int lo = ((x & ~(j - 1)) << 1) | (x & (j - 1)), hi = lo | j;
                const uint64_t p = ent[lo], q = ent[hi];
                if ((p > q) == ((lo & k) == 0)) {
                    ent[lo] = q;
                    ent[hi] = p;
                }
            }
            __syncthreads();
        }
    for (int p = tid; p < N; p += nt) {
        const uint64_t e = ent[p];
        const int src = ent_src(e);
        a.ent[p] = e;
        if (p == 0 || ent_src(ent[p - 1]) != src) {
            int q = p + 1;
            while (q < N && ent_src(ent[q]) == src) ++q;
            a.head[src] = make_int2(p, q - p);
        }
        if (e & ENT_CUR) {
            const int f = ent_fix(e);
            int at = a.deg[src];
            for (int q = p - 1; q >= 0 && ent_src(ent[q]) == src; --q) at += (ent[q] & ENT_CUR) ? 1 : 0;
            int *cell = a.adj + (int64_t)src * a.R + at;
            if (at < a.R) {  // (a source more fix-ups want than it has room for takes the first ones)
                a.hold[f] = *cell;
                *cell = a.fix[f];
                a.slot[f] = at;
            } else {
                a.slot[f] = -1;
            }
        }
    }
    for (int f = tid; f < F; f += nt)
        if (a.scur[f] < 0) a.slot[f] = -1;
    if (tid == 0) {
        st->nent = N;
        st->jfirst = sh_first;
        st->none = sh_none;
        st->settled = sh_first == INT_MAX || sh_none < sh_first;
    }
}

// The final prefix of the batch enters the graph; a fix-up for which nothing had
// room is tried once more against the graph itself.  One CTA.
__global__ void __launch_bounds__(1024) fix_commit_kernel(FixArgs a) {
    __shared__ int sh_found;
    FixState *st = a.st;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int F = st->F, touched = st->touched, none = st->none, first = st->jfirst;
    const int nent = st->nent;
    if (st->cnt == 0) return;
    int done = min(F, min(none, first));
    withdraw(a, F, done, nent);
    for (int f = tid; f < done; f += nt) {
        atomicAdd(a.deg + a.scur[f], 1);
        if (a.xcnt[f] == INT_MAX) st->capped = 1;
    }
    __syncthreads();
    int limit = done < F ? a.flab[done] : INT_MAX;
    for (int t = tid; t < touched; t += nt) {
        const int v = a.touched[t];
        if (a.label[v] < limit) atomicOr(a.reached + (v >> 5), 1u << (v & 31));
    }
    if (none < F && none < first) {
        if (tid == 0) sh_found = INT_MAX;
        __syncthreads();
        for (int64_t x = tid; x < a.n; x += nt)
            if (bit_is_set(a.reached, x) && ldv(a.deg + x) < a.R) {
                atomicMin(&sh_found, (int)x);
                break;
            }
        __syncthreads();
        const int sel = sh_found;
        if (sel == INT_MAX) {
            if (tid == 0) st->status = -5;
        } else {
            if (tid == 0) {
                const int u = a.fix[done], dg = a.deg[sel];
                a.adj[(int64_t)sel * a.R + dg] = u;
                a.deg[sel] = dg + 1;
                if (a.xcnt[done] == INT_MAX) st->capped = 1;
            }
            ++done;
            const int lim2 = done < F ? a.flab[done] : INT_MAX;
            for (int t = tid; t < touched; t += nt) {
                const int v = a.touched[t], l = a.label[v];
                if (l >= limit && l < lim2) atomicOr(a.reached + (v >> 5), 1u << (v & 31));
            }
        }
    }
    __syncthreads();
    for (int t = tid; t < touched; t += nt) a.label[a.touched[t]] = INT_MAX;
    if (tid == 0) {
        st->cursor = done < F ? a.fix[done] : (long long)st->last + 1;
        st->added += done;
        // the batch follows how much of it settled (the result does not depend
        // on it): a larger one serves more fix-ups per search's latency, until
        // the chains of fix-ups that depend on one another outlast the rounds
        if (done * 10 >= F * 9) st->B = min(st->B * 2, a.bmax);
        else if (done * 2 < F) st->B = max(st->B / 2, CONNECT_MIN_BATCH);
    }
}

}  // namespace

cudaError_t run_connect(const ConnectLaunch &l, int out_host[4], cudaStream_t st) {
    const int64_t n = l.n;
    const int64_t nwords = (n + 31) / 32;
    const int xcap = 4 * l.L + 64;
    // fix-ups per batch: what fits 512 MB of pools and logs, at most the kernels' limit
    int BMAX = CONNECT_MAX_BATCH;
    while (BMAX > CONNECT_MIN_BATCH && (size_t)BMAX * (8 * (size_t)l.L + 12 * (size_t)xcap) > (size_t(512) << 20)) BMAX /= 2;
    // one allocation for the whole pass
    size_t need = 0;
    auto plan = [&](size_t bytes) {
        const size_t at = need;
        need += (bytes + 255) & ~size_t(255);
        return at;
    };
    const size_t o_reached = plan(4 * nwords), o_stamp = plan(4 * n), o_used = plan(4 * n), o_head = plan(8 * n),
                 o_st = plan(sizeof(FixState)), o_lev = plan(4 * (BFS_LEVELS + 1)), zeroed = need;
    const size_t o_label = plan(4 * n), o_qa = plan(4 * n), o_qb = plan(4 * n), o_touched = plan(4 * n),
                 o_list = plan(4 * BMAX), o_fix = plan(4 * BMAX), o_flab = plan(4 * BMAX), o_xcnt = plan(4 * BMAX),
                 o_psize = plan(4 * BMAX), o_snew = plan(4 * BMAX), o_scur = plan(4 * BMAX), o_slot = plan(4 * BMAX),
                 o_hold = plan(4 * BMAX), o_ent = plan(16 * BMAX), o_pools = plan(8 * (size_t)BMAX * l.L),
                 o_xthr = plan(8 * (size_t)BMAX * xcap), o_xlog = plan(4 * (size_t)BMAX * xcap);
    struct Slab {
        unsigned char *p = nullptr;
        ~Slab() {
            if (p) cudaFree(p);
        }
    } slab;
    cudaError_t e;
    if ((e = cudaMalloc(reinterpret_cast<void **>(&slab.p), need))) return e;
    auto at = [&](size_t o) { return slab.p + o; };
    FixArgs a;
    a.base4 = reinterpret_cast<const float4 *>(l.base);
    a.dp4 = l.dp / 4;
    a.rows = ExactRows{a.base4, a.dp4, reinterpret_cast<const uint4 *>(l.u8.rows), l.u8.chunks, l.u8.d, l.u8.lo};
    a.n = n;
    a.adj = l.adj;
    a.deg = l.deg;
    a.R = l.R;
    a.W = round32c(l.R);
    a.nav = l.nav;
    a.L = l.L;
    a.max_steps = l.max_steps;
    a.reached = reinterpret_cast<uint32_t *>(at(o_reached));
    a.stamp = reinterpret_cast<int *>(at(o_stamp));
    a.used = reinterpret_cast<int *>(at(o_used));
    a.bmax = BMAX;
    a.head = reinterpret_cast<int2 *>(at(o_head));
    a.st = reinterpret_cast<FixState *>(at(o_st));
    a.label = reinterpret_cast<int *>(at(o_label));
    a.qa = reinterpret_cast<int *>(at(o_qa));
    a.qb = reinterpret_cast<int *>(at(o_qb));
    a.touched = reinterpret_cast<int *>(at(o_touched));
    a.list = reinterpret_cast<int *>(at(o_list));
    a.fix = reinterpret_cast<int *>(at(o_fix));
    a.flab = reinterpret_cast<int *>(at(o_flab));
    a.xcnt = reinterpret_cast<int *>(at(o_xcnt));
    a.psize = reinterpret_cast<int *>(at(o_psize));
    a.snew = reinterpret_cast<int *>(at(o_snew));
    a.scur = reinterpret_cast<int *>(at(o_scur));
    a.slot = reinterpret_cast<int *>(at(o_slot));
    a.hold = reinterpret_cast<int *>(at(o_hold));
    a.ent = reinterpret_cast<uint64_t *>(at(o_ent));
    a.pools = reinterpret_cast<uint64_t *>(at(o_pools));
    a.xthr = reinterpret_cast<uint64_t *>(at(o_xthr));
    a.xlog = reinterpret_cast<int *>(at(o_xlog));
    a.xcap = xcap;
    int *lev = reinterpret_cast<int *>(at(o_lev));
    if ((e = cudaMemsetAsync(slab.p, 0, zeroed, st)) || (e = launch_fill(a.label, n, INT_MAX, st))) return e;
    // reach from the navigating node: level-synchronous BFS, BFS_LEVELS levels
    // between two looks from the host (levels past the end find no frontier)
    if ((e = launch_bfs_seed(a.reached, l.nav, a.qa, lev, st))) return e;
    FixState h{};
    h.B = CONNECT_FIRST_BATCH < BMAX ? CONNECT_FIRST_BATCH : BMAX;
    if ((e = cudaMemcpyAsync(a.st, &h, sizeof(h), cudaMemcpyHostToDevice, st))) return e;
    auto list_next = [&]() -> cudaError_t {  // the next batch's list, and the state after it to the host
        gather_unreached_kernel<<<1, 1024, 0, st>>>(a.reached, n, a.list, a.label, a.touched, a.qa, a.st);
        cudaError_t g = cudaGetLastError();
        if (!g) g = cudaMemcpyAsync(&h, a.st, sizeof(h), cudaMemcpyDeviceToHost, st);
        return g;
    };
    int *cur = a.qa, *nxt = a.qb;
    for (int64_t level = 0; level <= n; level += BFS_LEVELS) {
        for (int t = 0; t < BFS_LEVELS; ++t) {
            if ((e = launch_bfs_level(l.adj, l.R, cur, lev + t, nxt, lev + t + 1, a.reached, st))) return e;
            std::swap(cur, nxt);
        }
        int nf = 0;
        if ((e = cudaMemcpyAsync(&nf, lev + BFS_LEVELS, sizeof(int), cudaMemcpyDeviceToHost, st))) return e;
        if ((e = cudaStreamSynchronize(st))) return e;
        if (nf == 0) break;
        if ((e = cudaMemsetAsync(lev, 0, 4 * (BFS_LEVELS + 1), st))) return e;
        if ((e = cudaMemcpyAsync(lev, &nf, sizeof(int), cudaMemcpyHostToDevice, st))) return e;
    }
    const int wpb = 4;
    const size_t psmem = 16 * (size_t)BMAX;
    if ((e = cudaFuncSetAttribute(fix_propose_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psmem)) ||
        (e = list_next()) || (e = cudaStreamSynchronize(st)))
        return e;
    for (int64_t batch = 0; batch <= n && h.cnt > 0 && !h.status; ++batch) {
        int *cur = a.qa, *nxt = a.qb;
        for (int t = 0; t < LABEL_LEVELS; ++t) {
            label_level_kernel<<<sm_count() * 4, 256, 0, st>>>(a, t, cur, nxt);
            std::swap(cur, nxt);
        }
        label_kernel<<<1, 1024, 0, st>>>(a, cur, nxt);
        NSG_DISPATCH_DP4(a.dp4, {
            // a batch's searches leave the SMs nearly empty, so their latency,
            // not the occupancy, sets the time: 513..1024-value rows keep more
            // rows in flight than the search kernels do
            constexpr int UC = V_ == 8 ? NSG_CONNECT_U_WIDE8 : U_;
            void (*search)(FixArgs, int) = fix_search_kernel<G_, V_, UC, false>;
            if constexpr (V_ <= 4)
                if (a.rows.u8 != nullptr) search = fix_search_kernel<G_, V_, UC, true>;
            // a batch has few searches: the largest visited set (little measured
            // twice) that lets all of them run at once; with 512 slots the pass
            // takes 3.20 ms instead of 3.16 (SIFT-shaped 100,000), 6.37 instead of
            // 6.19 (DEEP-shaped 150,000)
            const int64_t blocks = ((h.cnt + wpb - 1) / wpb + sm_count() - 1) / sm_count();  // per SM
            a.H = l.hash_slots;
            for (int slots = 4096; slots > a.H; slots >>= 1)
                if (blocks * (wpb * warp_smem_bytes(l.L, a.W, 0, slots, true) + 1024) <= smem_per_sm() &&
                    wpb * warp_smem_bytes(l.L, a.W, 0, slots, true) <= smem_optin())
                    a.H = slots;
            a.hshift = 32 - log2c((unsigned)a.H);
            const size_t per_warp = warp_smem_bytes(l.L, a.W, 0, a.H, true);
            e = cudaFuncSetAttribute(search, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(per_warp * wpb));
            for (int r = 0; r < CONNECT_ROUNDS && !e; ++r) {
                search<<<(h.cnt + wpb - 1) / wpb, wpb * 32, per_warp * wpb, st>>>(a, r);
                fix_propose_kernel<<<1, 1024, psmem, st>>>(a);
                e = cudaGetLastError();
            }
        });
        if (e) return e;
        fix_commit_kernel<<<1, 1024, 0, st>>>(a);
        if ((e = cudaGetLastError()) || (e = list_next()) || (e = cudaStreamSynchronize(st))) return e;
    }
    out_host[0] = h.added;
    out_host[1] = h.status;
    out_host[2] = h.capped;
    out_host[3] = h.redone;
    return cudaSuccess;
}

}  // namespace nsg
