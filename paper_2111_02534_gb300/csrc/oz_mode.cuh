// The fused mode product of the 2D tensor-core H-apply (oz_mode.cu), as the H-apply's host
// code (ozaki_tc.cu) sees it.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace tps {
namespace ozm {

constexpr int kMaxModePoints = 64;  // longest mode the fused product takes

// K_k's digits in the layout the kernel copies to shared memory: image bytes and column count
// for a mode of n points (n <= kMaxModePoints).
size_t image_bytes(int n);
// Builds the image (device, image_bytes(n)) and the raw row exponents eK[n] of the row-major
// n x n matrix K.
void launch_build_image(const double *K, int n, uint4 *image, unsigned *eK, cudaStream_t s);

struct ModeArgs {
  const double *psi;        // [nvec][N]
  double *out;              // [nvec][N], must not overlap psi
  long long N;
  int n;                    // points of the mode
  long long sigma;          // its stride in the vector layout
  const uint4 *image;       // launch_build_image
  const unsigned *eK;
  int nvec;
  bool store;               // true: out = K psi, else out += K psi
  int *err;                 // device flag of timed-out waits
};
// One mode's product.
cudaError_t launch_mode_product(const ModeArgs &a, cudaStream_t s);
// out += (V - theta) psi; theta_dev: theta of each vector (null: theta0).
cudaError_t launch_potential_term(const double *psi, const double *V, double *out, long long N,
                                  int nvec, const double *theta_dev, double theta0,
                                  cudaStream_t s);

}  // namespace ozm
}  // namespace tps
