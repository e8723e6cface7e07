// The tensor-core form of the calibration's attention weights (okq_calib_scores.cu), as the calibration calls it.
#pragma once
#include <cuda_fp16.h>

#include "okq_common.cuh"

namespace okq {

constexpr int SCORE_TILE = 128;       // queries and keys per tile
constexpr int SCORE_MIN_STEPS = 4;    // tiles a block has at least: bounds the number of pieces of a query or key tile
// Fewest tokens of that form: three tiles.  Its scratch, two floats per query and piece of it and one per key and piece, then fits
// into what the calibration documents (2 G n + ceil(n / 64) G n floats): with at least four steps a block, a query has at most
// n_t / 4 + 2 pieces and a key G n_t / 4 + 2, n_t = ceil(n / 128).
// From there on it is the faster one, too: 257 / 384 / 511 tokens with 1 to 8 heads 18 to 20 us against 21 / 27 / 34 of the mma.sync
// kernels.
constexpr int SCORE_MIN_TOKENS = 2 * SCORE_TILE + 1;

cudaError_t launch_calib_scores(const __half* q, const __half* k, int G, int n, float scale2, int causal, int n_sm, void* ws, float* w_out,
                                long long wait_limit, int skip_step, cudaStream_t s);

}  // namespace okq
