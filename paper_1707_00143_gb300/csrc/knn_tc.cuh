// knn_tc.cuh -- what the two tensor-core kNN kernels share (knn_tc.cu converts the
// rows and chooses; knn_tc_small.cu).
#pragma once

#include <cuda.h>

#include "kernels.h"

namespace nsg {

// BF16 rows padded to dk values, their squared norms (base: +inf up to a whole
// tile), and the lists to keep.
struct KnnOperands {
    CUtensorMap mq, mx;  // boxes of 64 values by 128 rows, 128-byte swizzle
    const float *xn, *qn;
    int dk;
    int64_t ntiles;  // base tiles of 128 rows
    int KL;          // entries per row's list
    int *err;        // device flag: a bounded wait gave up
};

// Tiles of a chunk of the base: ~48 MB of BF16 rows, one launch per chunk over
// every query row, so a chunk stays in L2 while they pass over it (a single
// sweep per CTA would re-read a base larger than L2 from HBM once per wave of
// CTAs).  NSG_KNN_CHUNK_TILES: smaller chunks (tests).
int64_t knn_chunk_tiles(int dk);

template <typename T>
struct KnnScratch {
    T *p = nullptr;
    ~KnnScratch() {
        if (p) cudaFree(p);
    }
    cudaError_t alloc(size_t n) { return cudaMalloc(reinterpret_cast<void **>(&p), n * sizeof(T) + 16); }
};

// Waits for the stream; an error where a pipeline wait gave up.
cudaError_t knn_finish(const KnnOperands &o, cudaStream_t st);

// The KL best per query row into ids / d2 [nq][KL], by a CTA per 128 rows.
cudaError_t knn_select_small(const KnnLaunch &l, const KnnOperands &o, int *ids, float *d2, cudaStream_t st);

}  // namespace nsg
