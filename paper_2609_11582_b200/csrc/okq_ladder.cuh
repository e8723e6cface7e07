// View of an okq_ladder_cache and the value codebooks, shared by the ladder's kernels.
#pragma once
#include "okq_common.cuh"
#include "okq_device.cuh"

namespace okq {

// ascending levels / thresholds for b = 2, 3, 4 (index b - 2); the middle threshold is 0 by symmetry
#define OKQ_LADDER_LEVELS { \
    {-0x1.116a30p-3f, -0x1.47d908p-5f, 0x1.47d908p-5f, 0x1.116a30p-3f}, \
    {-0x1.858b36p-3f, -0x1.e68c10p-4f, -0x1.11b402p-4f, -0x1.62ef2ep-6f, 0x1.62ef2ep-6f, 0x1.11b402p-4f, 0x1.e68c10p-4f, \
     0x1.858b36p-3f}, \
    {-0x1.eea6ccp-3f, -0x1.76883ap-3f, -0x1.24e5cep-3f, -0x1.c6cde4p-4f, -0x1.5529e8p-4f, -0x1.db8b5ep-5f, -0x1.18fa1cp-5f, \
     -0x1.73df2ap-7f, 0x1.73df2ap-7f, 0x1.18fa1cp-5f, 0x1.db8b5ep-5f, 0x1.5529e8p-4f, 0x1.c6cde4p-4f, 0x1.24e5cep-3f, \
     0x1.76883ap-3f, 0x1.eea6ccp-3f}}
#define OKQ_LADDER_THRESHOLDS { \
    {-0x1.636072p-4f, 0.0f, 0x1.636072p-4f}, \
    {-0x1.3c689ep-3f, -0x1.7c200ap-4f, -0x1.6a6fccp-5f, 0.0f, 0x1.6a6fccp-5f, 0x1.7c200ap-4f, 0x1.3c689ep-3f}, \
    {-0x1.b29782p-3f, -0x1.4db704p-3f, -0x1.042660p-3f, -0x1.8dfbe6p-4f, -0x1.2177ccp-4f, -0x1.7a42bcp-5f, -0x1.75f1e6p-6f, 0.0f, \
     0x1.75f1e6p-6f, 0x1.7a42bcp-5f, 0x1.2177ccp-4f, 0x1.8dfbe6p-4f, 0x1.042660p-3f, 0x1.4db704p-3f, 0x1.b29782p-3f}}
static __constant__ float c_levels[3][16] = OKQ_LADDER_LEVELS;
static __constant__ float c_thresholds[3][16] = OKQ_LADDER_THRESHOLDS;
static const float h_levels[3][16] = OKQ_LADDER_LEVELS;
static const float h_thresholds[3][16] = OKQ_LADDER_THRESHOLDS;
__device__ __forceinline__ float ladder_level(int bits, int code) { return c_levels[bits - 2][code]; }

struct LadderView {
  int batch, n_kv_heads, n_q_heads, capacity, bits;
  unsigned char* k_codes;
  __half* k_norm;
  __half* k_meta;
  unsigned char* v_codes;
  __half* v_norm;
  unsigned char* modality;
  __host__ __device__ size_t unit(int b, int h) const { return (size_t)b * n_kv_heads + h; }
  __host__ __device__ int row_bytes() const { return 16 * bits; }
};

// decode attention (okq_ladder_decode.cu)
cudaError_t launch_ladder_decode(const LadderView& cv, int n_tokens, const __half* q, float sm_scale, const float* signs,
                                 const float* R, int n_R, float* out, cudaStream_t s);

// value quantiser on the tensor cores (okq_quant_tc.cu); OKQ_ERR_UNSUPPORTED for strides a tensor map cannot describe
okq_status launch_ladder_values_tc(const LadderView& lv, const __half* v, const int64_t strides[3], const unsigned char* modality,
                                   int n_tokens, const float* R, int n_R, int n_sm, cudaStream_t s, long long wait_limit = 0,
                                   int skip_tile = -1);

}  // namespace okq
