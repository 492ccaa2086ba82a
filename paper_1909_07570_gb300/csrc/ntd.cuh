// nnTD of a 3-way tensor (ntd.cu): the body of ntd_fit.
#pragma once

#include "common.cuh"

namespace nnc {

// FP64 (T = double) and FP32 (T = float) paths. Arguments as ntd_fit with
// d = 3, already validated. tensor_cores (float only): FP32-accurate tensor-core passes
// where the shape allows, else SIMT.
template <typename T>
int ntd_fit3(const T* X, const int64_t* dims, const int* m, const nnc_opts* o, T* const* F, T* G,
             double* trace, double* rel_err, bool tensor_cores, cudaStream_t s);

// NNC_BF16_REFINE path; *refined_from (may be NULL) gets the index of the
// first FP32 refinement sweep (iters when there was none).
int ntd_fit3_bf16(const float* X, const int64_t* dims, const int* m, const nnc_opts* o,
                  float* const* F, float* G, double* trace, double* rel_err, int* refined_from,
                  cudaStream_t s);

// Whole fits of small tensors on one thread-block cluster (ntd_cluster.cu).
// ntd_cluster_fits: the shape is one it takes and is the faster form for.
// ntd_cluster_sweeps: `sweeps` sweeps in place on F and G in one launch; counter is
// trace_record's pair, x2 the device's ||X||^2, trace (device) may be NULL.
template <typename T>
bool ntd_cluster_fits(const int64_t* dims, const int* m);
template <typename T>
int ntd_cluster_sweeps(const T* X, const int64_t* dims, const int* m, T* const* F, T* G, double eps,
                       int sweeps, const double* x2, double* trace, int* counter, cudaStream_t s);

}  // namespace nnc
