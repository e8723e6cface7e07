// The direct eigensolver of okq_eigen.cu, as the calibration calls it.
#pragma once
#include <cuda_runtime.h>

#include "okq_layout.cuh"

namespace okq {

constexpr size_t EIGEN_BYTES = (size_t)D * D * sizeof(double);   // workspace: 126 reflectors and the word below
constexpr size_t EIGEN_LEFT = (size_t)(D - 1) * D;               // double whose first int says that the matrix is left to the Jacobi solver

// eigenvalues and R = H U^T of one symmetric matrix, or the word at EIGEN_LEFT set
cudaError_t launch_calib_spectrum(const float* C, const float* signs, double* ws, float* R, float* lambda, int* sweeps, cudaStream_t s);

}  // namespace okq
