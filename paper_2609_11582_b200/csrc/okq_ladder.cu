// OmniKVQuant at 2, 3 and 4 bits per code over a canonical cache (the bit-width ladder: K2V2 / K3V3 / K4V4).
// Plain CUDA-core kernels that follow the 2-bit path's arithmetic with the number of levels changed:
//   k_ladder_keys    Eq. 2 + Eq. 4: one block per 32-token window of one (sequence, KV head)
//   k_ladder_values  Eq. 6 + Eq. 3: likewise, the rotation as one fused-multiply-add chain per coordinate
// (decode attention: okq_ladder_decode.cu)
// The value levels are the Lloyd-Max quantiser of N(0, 1/128) with 2^b levels (fixed point of: level = mean of its
// cell, threshold = mid-point of neighbouring levels), held as constants.
#include "../../include/okq_ladder.h"
#include "okq_ladder.cuh"

namespace okq {

namespace {

constexpr int GP_L = OKQ_MAX_GROUP;   // padded GQA group

// packs the 32 codes cd[0..31] (channels 32 part .. 32 part + 31 of one token) into 4 * bits bytes of its bit stream
__device__ __forceinline__ void pack_quarter(const unsigned char* cd, int bits, unsigned char* dst) {
  unsigned long long lo = 0, hi = 0;
#pragma unroll
  for (int c = 0; c < 32; c++) {
    const int pos = bits * c;
    const unsigned long long v = cd[c];
    if (pos < 64) {
      lo |= v << pos;
      if (pos + bits > 64) hi |= v >> (64 - pos);
    } else {
      hi |= v << (pos - 64);
    }
  }
  const int nb = 4 * bits;   // 8, 12 or 16 bytes
  for (int k = 0; k < nb; k++) dst[k] = (unsigned char)((k < 8 ? lo >> (8 * k) : hi >> (8 * (k - 8))) & 0xffu);
}

// code of channel c in a token's bit stream
__device__ __forceinline__ unsigned load_code(const unsigned char* row, int bits, int c) {
  const int pos = bits * c, byte = pos >> 3;
  const unsigned w = (unsigned)row[byte] | ((unsigned)row[byte + ((pos & 7) + bits > 8 ? 1 : 0)] << 8);
  return (w >> (pos & 7)) & ((1u << bits) - 1u);
}

struct QuantSmem {
  float z[W][D + 1];
  unsigned char code[W][D];
  unsigned char mod[W];
};

// grid (windows, heads, batch), 128 threads
__global__ void __launch_bounds__(128) k_ladder_keys(LadderView cv, const __half* __restrict__ k, long long sb, long long sh,
                                                     long long st, const float* __restrict__ signs) {
  __shared__ QuantSmem sm;
  const int win = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const size_t u = cv.unit(b, h);
  const float4 sg = *reinterpret_cast<const float4*>(signs + 4 * lane);
  for (int kk = 0; kk < 8; kk++) {
    const int i = warp * 8 + kk;
    const float4 x = load_row4(k + b * sb + h * sh + (long long)(win * W + i) * st, lane);
    float n = warp_norm(x);
    const __half nh = __float2half_rn(n);
    const float nf = __half2float(nh);
    const float cinv = nf != 0.0f ? __fdiv_rn(RSQRT_D, nf) : 0.0f;
    const float4 y = warp_fwht(make_float4(__fmul_rn(sg.x, x.x), __fmul_rn(sg.y, x.y), __fmul_rn(sg.z, x.z), __fmul_rn(sg.w, x.w)), lane);
    // a zero vector (norm 0) has z = +0 in every coordinate
    sm.z[i][4 * lane + 0] = nf != 0.0f ? __fmul_rn(y.x, cinv) : 0.0f; sm.z[i][4 * lane + 1] = nf != 0.0f ? __fmul_rn(y.y, cinv) : 0.0f;
    sm.z[i][4 * lane + 2] = nf != 0.0f ? __fmul_rn(y.z, cinv) : 0.0f; sm.z[i][4 * lane + 3] = nf != 0.0f ? __fmul_rn(y.w, cinv) : 0.0f;
    if (lane == 0) cv.k_norm[u * cv.capacity + (size_t)win * W + i] = nh;
  }
  __syncthreads();
  {
    const int c = tid;
    const float L = (float)((1 << cv.bits) - 1);
    float mn = sm.z[0][c], mx = mn;
    for (int i = 1; i < W; i++) { const float v = sm.z[i][c]; mn = fminf(mn, v); mx = fmaxf(mx, v); }
    const __half mh = __float2half_rn(mn);
    const float mf = __half2float(mh);
    float range = __fsub_rn(mx, mf);
    range = range < 0.0f ? 0.0f : range;
    const __half s16 = __float2half_rn(__fdiv_rn(range, L));
    const float sf = __half2float(s16);
    __half* meta = cv.k_meta + ((u * (cv.capacity / W) + win) * D + c) * 2;
    meta[0] = mh; meta[1] = s16;
    const float r = sf > 0.0f ? __fdiv_rn(1.0f, sf) : 0.0f;
    for (int i = 0; i < W; i++) {
      float q = rintf(__fmul_rn(__fsub_rn(sm.z[i][c], mf), r));
      q = q < 0.0f ? 0.0f : (q > L ? L : q);
      sm.code[i][c] = sf > 0.0f ? (unsigned char)q : (unsigned char)0;
    }
  }
  __syncthreads();
  {
    const int i = tid >> 2, part = tid & 3;
    unsigned char* row = cv.k_codes + (u * cv.capacity + (size_t)win * W + i) * cv.row_bytes();
    pack_quarter(&sm.code[i][32 * part], cv.bits, row + 4 * cv.bits * part);
  }
}

struct ValueSmem {
  __align__(16) float x[W][D + 4];   // the window's value rows (fp32), 16-byte aligned rows
  unsigned char code[W][D];
  unsigned char mod[W];
  float inv[W];
  int uniform;
};

__global__ void __launch_bounds__(128) k_ladder_values(LadderView cv, const __half* __restrict__ v, long long sb, long long sh,
                                                       long long st, const unsigned char* __restrict__ modality, int n_tokens,
                                                       const float* __restrict__ R, int n_R) {
  __shared__ ValueSmem sm;
  const int win = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const size_t u = cv.unit(b, h);
  if (tid < W) {
    unsigned m = modality[(size_t)b * n_tokens + win * W + tid];
    m = m > 2 ? 0 : m;
    sm.mod[tid] = (unsigned char)m;
    if (h == 0) cv.modality[(size_t)b * cv.capacity + win * W + tid] = (unsigned char)m;
    const unsigned m0 = __shfl_sync(0xffffffffu, m, 0);
    const int uni = __all_sync(0xffffffffu, m == m0);
    if (tid == 0) sm.uniform = uni;
  }
  for (int kk = 0; kk < 8; kk++) {
    const int i = warp * 8 + kk;
    const float4 x = load_row4(v + b * sb + h * sh + (long long)(win * W + i) * st, lane);
    const float n = warp_norm(x);
    const __half nh = __float2half_rn(n);
    const float nf = __half2float(nh);
    *reinterpret_cast<float4*>(&sm.x[i][4 * lane]) = x;
    if (lane == 0) {
      cv.v_norm[u * cv.capacity + (size_t)win * W + i] = nh;
      sm.inv[i] = nf != 0.0f ? __fdiv_rn(1.0f, nf) : 0.0f;
    }
  }
  __syncthreads();
  {
    // thread = output coordinate c: z_c = (sum_k R_m[c][k] v_k) / norm as one fused-multiply-add chain in ascending k
    const int c = tid, nth = (1 << cv.bits) - 1;
    const float* Rset = R + (size_t)(n_R == 1 ? 0 : h) * 3 * D * D;
    const float* th = c_thresholds[cv.bits - 2];
    if (sm.uniform) {   // one matrix for the window: every row element is read once for the 32 tokens
      const float4* Rrow = reinterpret_cast<const float4*>(Rset + ((size_t)sm.mod[0] * D + c) * D);
      float acc[W];
#pragma unroll
      for (int i = 0; i < W; i++) acc[i] = 0.0f;
      for (int k4 = 0; k4 < D / 4; k4++) {
        const float4 r4 = __ldg(Rrow + k4);
#pragma unroll
        for (int i = 0; i < W; i++) {
          const float4 x4 = *reinterpret_cast<const float4*>(&sm.x[i][4 * k4]);
          float a = acc[i];
          a = __fmaf_rn(r4.x, x4.x, a);
          a = __fmaf_rn(r4.y, x4.y, a);
          a = __fmaf_rn(r4.z, x4.z, a);
          a = __fmaf_rn(r4.w, x4.w, a);
          acc[i] = a;
        }
      }
#pragma unroll
      for (int i = 0; i < W; i++) {
        const float z = __fmul_rn(acc[i], sm.inv[i]);
        int code = 0;
        for (int j = 0; j < nth; j++) code += z > th[j];
        sm.code[i][c] = (unsigned char)code;
      }
    } else {
      for (int i = 0; i < W; i++) {
        const float4* Rrow = reinterpret_cast<const float4*>(Rset + ((size_t)sm.mod[i] * D + c) * D);
        float a = 0.0f;
        for (int k4 = 0; k4 < D / 4; k4++) {
          const float4 r4 = __ldg(Rrow + k4);
          const float4 x4 = *reinterpret_cast<const float4*>(&sm.x[i][4 * k4]);
          a = __fmaf_rn(r4.x, x4.x, a);
          a = __fmaf_rn(r4.y, x4.y, a);
          a = __fmaf_rn(r4.z, x4.z, a);
          a = __fmaf_rn(r4.w, x4.w, a);
        }
        const float z = __fmul_rn(a, sm.inv[i]);
        int code = 0;
        for (int j = 0; j < nth; j++) code += z > th[j];
        sm.code[i][c] = (unsigned char)code;
      }
    }
  }
  __syncthreads();
  {
    const int i = tid >> 2, part = tid & 3;
    unsigned char* row = cv.v_codes + (u * cv.capacity + (size_t)win * W + i) * cv.row_bytes();
    pack_quarter(&sm.code[i][32 * part], cv.bits, row + 4 * cv.bits * part);
  }
}

}  // namespace
}  // namespace okq

namespace okq {
namespace {

// TurboQuant codec (Preliminaries, Eq. 2-3): norm, randomised Hadamard rotation, nearest level of the fixed codebook;
// no window statistics, no modality rotation.  32 vectors per block of 128 threads.
__global__ void __launch_bounds__(128) k_turboquant_encode(const __half* __restrict__ x, long long n, int bits,
                                                           const float* __restrict__ signs, unsigned char* __restrict__ codes,
                                                           __half* __restrict__ norms) {
  __shared__ unsigned char code[W][D];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long base = (long long)blockIdx.x * W;
  const float4 sg = *reinterpret_cast<const float4*>(signs + 4 * lane);
  const float* th = c_thresholds[bits - 2];
  const int nth = (1 << bits) - 1;
  for (int kk = 0; kk < 8; kk++) {
    const int i = warp * 8 + kk;
    if (base + i >= n) break;
    const float4 v = load_row4(x + (base + i) * D, lane);
    const float nrm = warp_norm(v);
    const __half nh = __float2half_rn(nrm);
    const float nf = __half2float(nh);
    const float cinv = nf != 0.0f ? __fdiv_rn(RSQRT_D, nf) : 0.0f;
    const float4 y = warp_fwht(make_float4(__fmul_rn(sg.x, v.x), __fmul_rn(sg.y, v.y), __fmul_rn(sg.z, v.z), __fmul_rn(sg.w, v.w)), lane);
    const float z[4] = {nf != 0.0f ? __fmul_rn(y.x, cinv) : 0.0f, nf != 0.0f ? __fmul_rn(y.y, cinv) : 0.0f,
                        nf != 0.0f ? __fmul_rn(y.z, cinv) : 0.0f, nf != 0.0f ? __fmul_rn(y.w, cinv) : 0.0f};
#pragma unroll
    for (int k4 = 0; k4 < 4; k4++) {
      int cd = 0;
      for (int j = 0; j < nth; j++) cd += z[k4] > th[j];
      code[i][4 * lane + k4] = (unsigned char)cd;
    }
    if (lane == 0) norms[base + i] = nh;
  }
  __syncthreads();
  const int i = tid >> 2, part = tid & 3;
  if (base + i < n) pack_quarter(&code[i][32 * part], bits, codes + (base + i) * 16 * bits + 4 * bits * part);
}

// x_hat = |x| H^T level[code], H^T y = diag(signs) Had y / sqrt(128); one warp per vector
__global__ void __launch_bounds__(128) k_turboquant_decode(const unsigned char* __restrict__ codes, const __half* __restrict__ norms,
                                                           long long n, int bits, const float* __restrict__ signs,
                                                           float* __restrict__ x_hat) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long i = (long long)blockIdx.x * 4 + warp;
  if (i >= n) return;
  const unsigned char* row = codes + i * 16 * bits;
  const float* lv = c_levels[bits - 2];
  const float4 y = warp_fwht(make_float4(lv[load_code(row, bits, 4 * lane + 0)], lv[load_code(row, bits, 4 * lane + 1)],
                                         lv[load_code(row, bits, 4 * lane + 2)], lv[load_code(row, bits, 4 * lane + 3)]), lane);
  const float4 sg = *reinterpret_cast<const float4*>(signs + 4 * lane);
  const float f = RSQRT_D * __half2float(norms[i]);
  *reinterpret_cast<float4*>(x_hat + i * D + 4 * lane) = make_float4(sg.x * y.x * f, sg.y * y.y * f, sg.z * y.z * f, sg.w * y.w * f);
}

okq_status check_ladder(const okq_ladder_cache* c, int n_tokens) {
  if (!c) return OKQ_ERR_INVALID_ARG;
  if (c->bits < 2 || c->bits > 4) return OKQ_ERR_UNSUPPORTED;
  if (c->batch <= 0 || c->n_kv_heads <= 0 || c->n_q_heads <= 0 || c->capacity <= 0 || c->capacity % W) return OKQ_ERR_INVALID_ARG;
  if (c->n_q_heads % c->n_kv_heads || c->n_q_heads / c->n_kv_heads > GP_L) return OKQ_ERR_UNSUPPORTED;
  if (n_tokens < 0 || n_tokens % W || n_tokens > c->capacity) return OKQ_ERR_INVALID_ARG;
  if (!c->k_codes || !c->k_norm || !c->k_meta || !c->v_codes || !c->v_norm || !c->modality) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(c->k_codes) || !aligned16(c->k_norm) || !aligned16(c->k_meta) || !aligned16(c->v_codes) || !aligned16(c->v_norm))
    return OKQ_ERR_ALIGNMENT;
  return OKQ_OK;
}

LadderView ladder_view(const okq_ladder_cache* c) {
  LadderView v;
  v.batch = c->batch; v.n_kv_heads = c->n_kv_heads; v.n_q_heads = c->n_q_heads; v.capacity = c->capacity; v.bits = c->bits;
  v.k_codes = static_cast<unsigned char*>(c->k_codes); v.k_norm = static_cast<__half*>(c->k_norm);
  v.k_meta = static_cast<__half*>(c->k_meta); v.v_codes = static_cast<unsigned char*>(c->v_codes);
  v.v_norm = static_cast<__half*>(c->v_norm); v.modality = c->modality;
  return v;
}

}  // namespace
}  // namespace okq

using namespace okq;

extern "C" {

int32_t okq_ladder_codebook(int32_t bits, float* levels, float* thresholds) {
  if (bits < 2 || bits > 4 || !levels || !thresholds) return 0;
  const int n = 1 << bits;
  for (int i = 0; i < n; i++) levels[i] = h_levels[bits - 2][i];
  for (int i = 0; i < n - 1; i++) thresholds[i] = h_thresholds[bits - 2][i];
  return n;
}

okq_status okq_ladder_quantize_keys(const okq_ladder_cache* cache, const void* k_fp16, const int64_t strides[3],
                                    int32_t n_tokens, const float* signs, void* stream) {
  okq_status st = check_ladder(cache, n_tokens);
  if (st != OKQ_OK) return st;
  if (!k_fp16 || !strides || !signs) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(k_fp16) || !aligned16(signs) || strides[0] % 8 || strides[1] % 8 || strides[2] % 8) return OKQ_ERR_ALIGNMENT;
  if (n_tokens == 0) return OKQ_OK;
  const dim3 grid(n_tokens / W, cache->n_kv_heads, cache->batch);
  k_ladder_keys<<<grid, 128, 0, static_cast<cudaStream_t>(stream)>>>(ladder_view(cache), static_cast<const __half*>(k_fp16),
                                                                     strides[0], strides[1], strides[2], signs);
  return launch_status();
}

okq_status okq_ladder_quantize_values(const okq_ladder_cache* cache, const void* v_fp16, const int64_t strides[3],
                                      int32_t n_tokens, const uint8_t* modality, const float* R, int32_t n_R,
                                      void* stream) {
  okq_status st = check_ladder(cache, n_tokens);
  if (st != OKQ_OK) return st;
  if (!v_fp16 || !strides || !modality || !R || (n_R != 1 && n_R != cache->n_kv_heads)) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(v_fp16) || !aligned16(R) || strides[0] % 8 || strides[1] % 8 || strides[2] % 8) return OKQ_ERR_ALIGNMENT;
  if (n_tokens == 0) return OKQ_OK;
  const dim3 grid(n_tokens / W, cache->n_kv_heads, cache->batch);
  k_ladder_values<<<grid, 128, 0, static_cast<cudaStream_t>(stream)>>>(ladder_view(cache), static_cast<const __half*>(v_fp16),
                                                                       strides[0], strides[1], strides[2], modality, n_tokens, R, n_R);
  return launch_status();
}

okq_status okq_ladder_decode_attention(const okq_ladder_cache* cache, int32_t n_tokens, const void* q, float sm_scale,
                                       const float* signs, const float* R, int32_t n_R, float* out, void* stream) {
  okq_status st = check_ladder(cache, n_tokens);
  if (st != OKQ_OK) return st;
  if (!q || !signs || !R || !out || (n_R != 1 && n_R != cache->n_kv_heads)) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(signs) || !aligned16(R) || !aligned16(out)) return OKQ_ERR_ALIGNMENT;
  const cudaError_t e = launch_ladder_decode(ladder_view(cache), n_tokens, static_cast<const __half*>(q), sm_scale, signs, R, n_R, out,
                                             static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) { set_last_cuda_error((int)e); return OKQ_ERR_CUDA; }
  return launch_status();
}

okq_status okq_turboquant_encode(const void* x_fp16, int64_t n_vectors, int32_t bits, const float* signs, uint8_t* codes,
                                 void* norms, void* stream) {
  if (bits < 2 || bits > 4) return OKQ_ERR_UNSUPPORTED;
  if (n_vectors < 0 || !x_fp16 || !signs || !codes || !norms) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(x_fp16) || !aligned16(signs) || !aligned16(codes)) return OKQ_ERR_ALIGNMENT;
  if (n_vectors == 0) return OKQ_OK;
  if ((n_vectors + W - 1) / W > 0x7fffffffLL) return OKQ_ERR_CAPACITY;
  k_turboquant_encode<<<(unsigned)((n_vectors + W - 1) / W), 128, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const __half*>(x_fp16), n_vectors, bits, signs, codes, static_cast<__half*>(norms));
  return launch_status();
}

okq_status okq_turboquant_decode(const uint8_t* codes, const void* norms, int64_t n_vectors, int32_t bits,
                                 const float* signs, float* x_hat, void* stream) {
  if (bits < 2 || bits > 4) return OKQ_ERR_UNSUPPORTED;
  if (n_vectors < 0 || !codes || !norms || !signs || !x_hat) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(codes) || !aligned16(signs) || !aligned16(x_hat)) return OKQ_ERR_ALIGNMENT;
  if (n_vectors == 0) return OKQ_OK;
  if ((n_vectors + 3) / 4 > 0x7fffffffLL) return OKQ_ERR_CAPACITY;
  k_turboquant_decode<<<(unsigned)((n_vectors + 3) / 4), 128, 0, static_cast<cudaStream_t>(stream)>>>(
      codes, static_cast<const __half*>(norms), n_vectors, bits, signs, x_hat);
  return launch_status();
}

}  // extern "C"
