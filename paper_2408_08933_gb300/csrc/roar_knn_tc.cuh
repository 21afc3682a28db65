// The tensor-core part of the kNN (roar_knn_tc.cu), as roar_knn.cu calls it.
#pragma once

#include <cuda_bf16.h>

#include "roar_internal.cuh"

namespace roar {

// How nt rows of T run against n rows of X: X ranges per block of 256 T rows,
// CTA pairs and the scratch they need.
struct KnnPlan {
    int splits, pairs, nkc, ksteps;
    int64_t units;
    size_t scratch_bytes;    // candidate buffers of the resident CTAs
    size_t lists_bytes;      // the ranges' lists (0 with one range)
};

cudaError_t knn_tc_plan(int64_t nt, int64_t n, int d, KnnPlan *p);
int64_t knn_tc_wave_rows(int d);
cudaError_t knn_tc_launch(const KnnPlan &p, const __nv_bfloat16 *T16, int64_t nt, const __nv_bfloat16 *X16, int64_t n,
                          int dp, void *scratch, void *lists, uint32_t *cand, int *err, uint64_t wait_ns,
                          cudaStream_t s);

}  // namespace roar
