// search_int8.cu -- the plain search kernels on integer rows: the FP32 keys from
// an exact 8-bit copy, a quarter of the bytes gathered and of the instructions
// per row, for queries that the copy holds (no fraction, no value outside its
// 256); the others are searched on the FP32 rows.  10,000 queries on 300,000
// SIFT-shaped rows (k = 100, L = 150): 3.29 -> 1.86 ms; one query on 100,000
// (L = 100): 0.41 -> 0.34 ms.
#include "search_kern.cuh"

namespace nsg {

// Whether the 8-bit copy x - lo holds every query: whole numbers within its 256,
// whose distances are exact in both forms (else *left = 1).
__global__ void __launch_bounds__(256) queries_held_kernel(const float *queries, int64_t count, float lo, int *left) {
    bool held = true;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < count; i += (int64_t)gridDim.x * 256) {
        const float v = __ldg(queries + i), y = v - lo;
        held &= rintf(v) == v && rintf(y) == y && y >= 0.0f && y <= 255.0f;
    }
    if (!__all_sync(NSG_FULL, held) && lane_id() == 0) *left = 1;
}

// One kernel that has both paths, or a kernel each of which the batch as a
// whole takes one.  In one kernel warps on different paths evict each other's
// instructions once the SMs are full, the more so the longer the row's code (10,000
// queries on 50,000 x 200 rows, k = 10, L = 150: 2,435 us with fractions in every
// other query, 2,181 with fractions throughout, 1,502 with none, 2,107 on FP32 rows
// alone), and with pools in global memory it spills (50 queries, L = 1,500: 5 %
// slower than FP32 rows alone; apart 1 %).  Apart: 2,121, 2,096 and 1,442 us;
// but the two more launches cost ~15 us, 10 % of a single query's search (L = 30), 4 %
// of 2,500 queries', and rows of up to 64 values have little code to evict (10,000
// queries on 50,000 x 32: every other one a fraction 1,606 us apart, 1,539 in one).
template <bool GP>
static cudaError_t launch_apart(SearchArgs a, const SearchLaunch &l, size_t per_warp, int wpq, cudaStream_t st) {
    int *left = l.work + WORK_LEFT;
    const int64_t count = l.nq / a.parts * a.d;
    const int64_t blocks = std::min<int64_t>((count + 1023) / 1024, (int64_t)sm_count() * 8);
    queries_held_kernel<<<(unsigned)blocks, 256, 0, st>>>(l.queries, count, a.lo, left);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    a.left = left;
    e = launch_search_args<GP, false, PREC_F32_INT8>(a, l, per_warp, 0, false, wpq, st);
    if (e != cudaSuccess) return e;
    return launch_search_args<GP, false, PREC_F32_REST>(a, l, per_warp, 0, false, wpq, st);
}

cudaError_t launch_search_int8(const SearchArgs &a, const SearchLaunch &l, size_t per_warp, int wpq, cudaStream_t st) {
    if (a.gpool != nullptr) return launch_apart<true>(a, l, per_warp, wpq, st);
    if (l.nq >= 4096 && l.d > 64) return launch_apart<false>(a, l, per_warp, wpq, st);
    return launch_search_args<false, false, PREC_F32_EITHER>(a, l, per_warp, 0, false, wpq, st);
}

}  // namespace nsg
