// The direct eigensolver of okq_eigen.cu, as the calibration calls it.
#pragma once
#include <cuda_runtime.h>

#include "okq_layout.cuh"

namespace okq {

// In the place of lambda[0], until the Jacobi solver behind has run: the matrix is left to it.  (A NaN that no result has: eigenvalues
// of the direct solver are numbers.)
constexpr unsigned EIGEN_LEFT = 0x7fe11e57u;

// eigenvalues and R = H U^T of one symmetric matrix, or lambda[0] = EIGEN_LEFT
cudaError_t launch_calib_spectrum(const float* C, const float* signs, float* R, float* lambda, int* sweeps, cudaStream_t s);

}  // namespace okq
