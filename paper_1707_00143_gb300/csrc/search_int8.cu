// search_int8.cu -- the plain search kernels on integer rows: the FP32 keys from
// an exact 8-bit copy, a quarter of the bytes gathered and of the instructions
// per row.  A query that the copy does not hold (a fraction, a value outside
// its 256) is searched on the FP32 rows by the same warp.  10,000 queries on
// 300,000 SIFT-shaped rows (k = 100, L = 150): 3.29 -> 1.86 ms; one query on
// 100,000 (L = 100): 0.41 -> 0.34 ms.
#include "search_kern.cuh"

namespace nsg {

cudaError_t launch_search_int8(const SearchArgs &a, const SearchLaunch &l, size_t per_warp, int wpq, cudaStream_t st) {
    return a.gpool != nullptr ? launch_search_args<true, false, true>(a, l, per_warp, 0, false, wpq, st)
                              : launch_search_args<false, false, true>(a, l, per_warp, 0, false, wpq, st);
}

}  // namespace nsg
