// Coarse-probe distances on the tensor cores (see probe_tc.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace pano {

// Whether the tensor-core probe handles dimension d (bf16 16-byte chunks).
bool probe_tc_supported(int d);
// Bound on |pd - exact| / (|q| + max |c|)^2 of the tensor-core distances.
double probe_tc_gerr(int d);
// Lays out I.cent_img, the centroids' operand images, from I.cent (where
// probe_tc_supported(I.d)).
int build_cent_image(pano_index& I, cudaStream_t st);
// pd[q][c] = qn2[q] + |c|^2 - 2 q.c for q < nq, c < nlist (row-major, row
// length nlist); err gets kErrTimeout if a bounded wait gave up.
int launch_probe_tc(const float* Q, int64_t nq, const pano_index& I, const float* qn2, float* pd,
                    int* err, cudaStream_t st);
// out[i]: the nearest centroid of row i < m of X (exact distances decide, ties
// to the lower id); best: kAssignWords m words of workspace.
constexpr int kAssignWords = 12;
int launch_assign_tc(const float* X, int64_t m, const pano_index& I, unsigned long long* best,
                     int32_t* out, int* err, cudaStream_t st);

}  // namespace pano
