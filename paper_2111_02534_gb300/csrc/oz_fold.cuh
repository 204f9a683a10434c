// The symmetry-folded 1D tensor-core H-apply (oz_fold.cu), as its host code (ozaki_tc.cu) sees it.
#pragma once

#include <cuda_runtime.h>

#include "tps_internal.h"

namespace tps {
namespace ozf {

struct Operator;

// Whether both modes of a 1D operator fold into blocks short enough for base-256 digits.
bool supported(const DevOperator &op);
// Builds the folded operator (device memory, kernels on s); err is the device flag of timed-out
// waits.  Null and *e set on failure.
Operator *create(const DevOperator &op, int *err, cudaStream_t s, cudaError_t *e);
void destroy(Operator *o);
// out = (H - theta) psi; theta_dev (nullable) overrides theta per vector.
cudaError_t apply(const Operator &o, const DevOperator &op, const double *psi, double *out,
                  int nvec, const double *theta_dev, double theta, cudaStream_t s);

}  // namespace ozf
}  // namespace tps
