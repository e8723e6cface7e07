// OmniKVQuant at 2, 3 and 4 bits per code over a canonical cache (the bit-width ladder: K2V2 / K3V3 / K4V4).
// The 2-bit path's arithmetic with the number of levels changed:
//   k_ladder_keys    Eq. 2 + Eq. 4: one block per 32-token window of one (sequence, KV head)
//   k_ladder_values  Eq. 6 + Eq. 3: likewise, the rotation as one fused-multiply-add chain per coordinate; only for strides that
//                    a tensor map cannot describe, everything else takes the tensor-core kernel (okq_quant_tc.cu)
//   k_turboquant_encode, k_turboquant_decode   the baseline codec
// (decode attention: okq_ladder_decode.cu)
// The value levels are the Lloyd-Max quantiser of N(0, 1/128) with 2^b levels (fixed point of: level = mean of its
// cell, threshold = mid-point of neighbouring levels), held as constants.
#include "../../include/okq_ladder.h"
#include "okq_ladder.cuh"
#include "okq_rotate.cuh"

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

// Codes are integers k added to 1.5 * 2^23: the float's bits are MAGIC_BITS + k, and eight of them at 8 field positions sum to
// the packed fields plus a constant (modulo 2^32).
constexpr float MAGIC = 12582912.0f;
constexpr uint32_t MAGIC_BITS = 0x4B400000u;
template <int BITS> __host__ __device__ constexpr uint32_t magic_sum8() {
  uint32_t s = 0;
  for (int i = 0; i < 8; i++) s += MAGIC_BITS << (BITS * i);
  return s;
}
// four groups of eight codes (8 BITS bits each) -> 4 * BITS bytes of the bit stream
template <int BITS> __device__ __forceinline__ void store_groups(const uint32_t (&g8)[4], unsigned char* dst) {
  uint32_t* d = reinterpret_cast<uint32_t*>(dst);
  if constexpr (BITS == 4) *reinterpret_cast<uint4*>(d) = make_uint4(g8[0], g8[1], g8[2], g8[3]);
  else if constexpr (BITS == 2) *reinterpret_cast<uint2*>(d) = make_uint2(g8[0] | g8[1] << 16, g8[2] | g8[3] << 16);
  else {
    d[0] = g8[0] | g8[1] << 24;
    d[1] = g8[1] >> 8 | g8[2] << 16;
    d[2] = g8[2] >> 16 | g8[3] << 8;
  }
}

struct QuantSmem {
  __align__(16) float z[W * ZS];       // rotated keys
  __align__(16) float m[D], r[D];      // per channel: stored minimum, 1 / stored step (0 for a zero step)
};

// grid (windows, heads, batch), 128 threads.  Bound by issue slots, like the 2-bit key quantiser whose transform it shares;
// a thread packs the 32 codes of a quarter of one token's row in registers.
template <int BITS>
__global__ void __launch_bounds__(128) k_ladder_keys(LadderView cv, const __half* __restrict__ k, long long sb, long long sh,
                                                     long long st, const float* __restrict__ signs) {
  __shared__ QuantSmem sm;
  const int win = blockIdx.x, h = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
  const size_t u = cv.unit(b, h), tok0 = u * cv.capacity + (size_t)win * W;
  depend_wait();
  rotate_rows(k + b * sb + h * sh + (long long)win * W * st, st, W, signs, sm.z, [&](int i, __half nh) { cv.k_norm[tok0 + i] = nh; });
  __syncthreads();
  constexpr float L = (float)((1 << BITS) - 1);
  {
    const int c = tid, cp = zpos(c);
    float mn = sm.z[cp], mx = mn;
#pragma unroll 8
    for (int i = 1; i < W; i++) { const float v = sm.z[i * ZS + cp]; mn = fminf(mn, v); mx = fmaxf(mx, v); }
    const __half mh = __float2half_rn(mn);
    const float mf = __half2float(mh);
    float range = __fsub_rn(mx, mf);
    range = range < 0.0f ? 0.0f : range;
    const __half s16 = __float2half_rn(__fdiv_rn(range, L));
    const float sf = __half2float(s16);
    reinterpret_cast<__half2*>(cv.k_meta)[(u * (cv.capacity / W) + win) * D + c] = __halves2half2(mh, s16);
    sm.m[c] = mf;
    sm.r[c] = sf > 0.0f ? __fdiv_rn(1.0f, sf) : 0.0f;
  }
  __syncthreads();
  // code = clamp(rint((z - m) / s), 0, L): clamping first gives the same integer, adding MAGIC rounds to nearest even.  A zero
  // step has r = 0 and so code 0.
  const int i = tid >> 2, part = tid & 3;
  uint32_t g8[4];
#pragma unroll
  for (int q = 0; q < 4; q++) {
    uint32_t w = 0;
#pragma unroll
    for (int e = 0; e < 2; e++) {
      const int c = 32 * part + 8 * q + 4 * e;
      const float4 z = *reinterpret_cast<const float4*>(&sm.z[i * ZS + zpos(c)]);
      const float4 m = *reinterpret_cast<const float4*>(&sm.m[c]), r = *reinterpret_cast<const float4*>(&sm.r[c]);
      const float zs[4] = {z.x, z.y, z.z, z.w}, ms[4] = {m.x, m.y, m.z, m.w}, rs[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
      for (int n = 0; n < 4; n++) {
        const float x = fminf(fmaxf(__fmul_rn(__fsub_rn(zs[n], ms[n]), rs[n]), 0.0f), L);
        w += __float_as_uint(__fadd_rn(x, MAGIC)) << (BITS * (4 * e + n));
      }
    }
    g8[q] = w - magic_sum8<BITS>();
    if (BITS < 4) g8[q] &= (1u << (8 * BITS % 32)) - 1u;
  }
  store_groups<BITS>(g8, cv.k_codes + (tok0 + i) * (16 * BITS) + 4 * BITS * part);
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
// no window statistics, no modality rotation.  32 vectors per block of 128 threads, eight threads per vector in the
// transform (two in-register halves around one shared-memory exchange).  524288 vectors at 2 bits, encode and decode:
// 300 us with one warp per vector (20 shuffles per transform) and byte-wise packing, 125 us in this form.

// number of thresholds below z: compared one by one at 2 bits, at 3 and 4 bits a bit of the code at a time
// (the threshold in the middle of what is left)
template <int BITS> __device__ __forceinline__ uint32_t nearest_level(float z, const float* th) {
  if constexpr (BITS == 2) return (uint32_t)(z > th[0]) + (uint32_t)(z > th[1]) + (uint32_t)(z > th[2]);
  uint32_t code = 0;
#pragma unroll
  for (int step = 1 << (BITS - 1); step; step >>= 1)
    if (z > th[code + step - 1]) code += step;
  return code;
}

template <int BITS>
__global__ void __launch_bounds__(128) k_turboquant_encode(const __half* __restrict__ x, long long n, const float* __restrict__ signs,
                                                           unsigned char* __restrict__ codes, __half* __restrict__ norms) {
  __shared__ __align__(16) float z[W * ZS];
  __shared__ float th[16];
  const int tid = threadIdx.x;
  const long long base = (long long)blockIdx.x * W;
  const int rows = (int)(n - base < W ? n - base : W);
  depend_wait();
  if (tid < 16) th[tid] = c_thresholds[BITS - 2][tid];
  rotate_rows(x + base * D, D, rows, signs, z, [&](int i, __half nh) { if (i < rows) norms[base + i] = nh; });
  __syncthreads();
  const int i = tid >> 2, part = tid & 3;
  if (i >= rows) return;
  uint32_t g8[4];
#pragma unroll
  for (int q = 0; q < 4; q++) {
    uint32_t w = 0;
#pragma unroll
    for (int e = 0; e < 2; e++) {
      const float4 v = *reinterpret_cast<const float4*>(&z[i * ZS + zpos(32 * part + 8 * q + 4 * e)]);
      const float zs[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 4; k++) w |= nearest_level<BITS>(zs[k], th) << (BITS * (4 * e + k));
    }
    g8[q] = w;
  }
  store_groups<BITS>(g8, codes + (base + i) * (16 * BITS) + 4 * BITS * part);
}

// x_hat = |x| H^T level[code], H^T y = diag(signs) Had y / sqrt(128)
template <int BITS>
__global__ void __launch_bounds__(128) k_turboquant_decode(const unsigned char* __restrict__ codes, const __half* __restrict__ norms,
                                                           long long n, const float* __restrict__ signs, float* __restrict__ x_hat) {
  __shared__ __align__(16) float z[16 * ZS];
  __shared__ float lev[16];
  const int tid = threadIdx.x, a = tid & 7, r = tid >> 3;
  depend_wait();
  if (tid < 16) lev[tid] = c_levels[BITS - 2][tid];
  __syncthreads();
  uint64_t sg[8];   // signs of channels 16 u + 2 a, + 1
#pragma unroll
  for (int u = 0; u < 8; u++) sg[u] = *reinterpret_cast<const uint64_t*>(signs + 16 * u + 2 * a);
#pragma unroll 1
  for (int half = 0; half < 2; half++) {
    const long long i = (long long)blockIdx.x * W + 16 * half + r;
    const long long ir = i < n ? i : n - 1;
    // 16 codes: 2 BITS bytes at byte 2 BITS a of the row
    const unsigned char* src = codes + ir * (16 * BITS) + 2 * BITS * a;
    uint32_t x[2];   // eight codes each
    if constexpr (BITS == 4) { const uint2 v = *reinterpret_cast<const uint2*>(src); x[0] = v.x; x[1] = v.y; }
    else if constexpr (BITS == 2) { const uint32_t v = *reinterpret_cast<const uint32_t*>(src); x[0] = v; x[1] = v >> 16; }
    else {
      const uint16_t* s2 = reinterpret_cast<const uint16_t*>(src);
      const uint32_t v0 = s2[0], v1 = s2[1], v2 = s2[2];
      x[0] = v0 | v1 << 16;
      x[1] = v1 >> 8 | v2 << 8;
    }
    const float f = RSQRT_D * __half2float(norms[ir]);
    uint64_t P[8], Q[8];
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const uint32_t w = x[q >> 2] >> (2 * BITS * (q & 3));
      P[q] = pack2(lev[w & ((1u << BITS) - 1u)], lev[(w >> BITS) & ((1u << BITS) - 1u)]);
    }
    hadamard_eight(P, Q, z + r * ZS, a);
    __syncwarp();   // (the row is written again in the next half)
    if (i < n) {
      const uint64_t f2 = pack2(f, f);
#pragma unroll
      for (int u = 0; u < 8; u++) *reinterpret_cast<uint64_t*>(x_hat + i * D + 16 * u + 2 * a) = mul2(mul2(sg[u], Q[u]), f2);
    }
  }
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
  auto go = [&](auto kernel) {
    launch_dependent(kernel, dim3(grid), 128, 0, static_cast<cudaStream_t>(stream), 1, ladder_view(cache), static_cast<const __half*>(k_fp16), strides[0], strides[1],
                                                                strides[2], signs);
  };
  if (cache->bits == 2) go(k_ladder_keys<2>);
  else if (cache->bits == 3) go(k_ladder_keys<3>);
  else go(k_ladder_keys<4>);
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
  // the tensor-core kernel, whose codes are the exact chain's; the chain kernel stays for strides that a tensor map cannot
  // describe (zero, 2^40 bytes or more)
  st = launch_ladder_values_tc(ladder_view(cache), static_cast<const __half*>(v_fp16), strides, modality, n_tokens, R, n_R, sm_count(),
                               static_cast<cudaStream_t>(stream));
  if (st == OKQ_OK) return launch_status();
  if (st != OKQ_ERR_UNSUPPORTED) return st;
  const dim3 grid(n_tokens / W, cache->n_kv_heads, cache->batch);
  k_ladder_values<<<grid, 128, 0, static_cast<cudaStream_t>(stream)>>>(ladder_view(cache), static_cast<const __half*>(v_fp16),
                                                                       strides[0], strides[1], strides[2], modality, n_tokens, R, n_R);
  return launch_status();
}

okq_status okq_debug_ladder_timeout(const okq_ladder_cache* cache, const void* v_fp16, const int64_t strides[3], int32_t n_tokens,
                                    const uint8_t* modality, const float* R, int32_t n_R, int64_t limit_clocks, void* stream) {
  okq_status st = check_ladder(cache, n_tokens);
  if (st != OKQ_OK) return st;
  if (!v_fp16 || !strides || !modality || !R || (n_R != 1 && n_R != cache->n_kv_heads) || limit_clocks <= 0) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(v_fp16) || !aligned16(R) || strides[0] % 8 || strides[1] % 8 || strides[2] % 8) return OKQ_ERR_ALIGNMENT;
  if (n_tokens == 0) return OKQ_OK;
  st = launch_ladder_values_tc(ladder_view(cache), static_cast<const __half*>(v_fp16), strides, modality, n_tokens, R, n_R, sm_count(),
                               static_cast<cudaStream_t>(stream), (long long)limit_clocks, 0);
  return st != OKQ_OK ? st : launch_status();
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
  auto go = [&](auto kernel) {
    launch_dependent(kernel, dim3((unsigned)((n_vectors + W - 1) / W)), 128, 0, static_cast<cudaStream_t>(stream), 1, 
        static_cast<const __half*>(x_fp16), n_vectors, signs, codes, static_cast<__half*>(norms));
  };
  if (bits == 2) go(k_turboquant_encode<2>);
  else if (bits == 3) go(k_turboquant_encode<3>);
  else go(k_turboquant_encode<4>);
  return launch_status();
}

okq_status okq_turboquant_decode(const uint8_t* codes, const void* norms, int64_t n_vectors, int32_t bits,
                                 const float* signs, float* x_hat, void* stream) {
  if (bits < 2 || bits > 4) return OKQ_ERR_UNSUPPORTED;
  if (n_vectors < 0 || !codes || !norms || !signs || !x_hat) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(codes) || !aligned16(signs) || !aligned16(x_hat)) return OKQ_ERR_ALIGNMENT;
  if (n_vectors == 0) return OKQ_OK;
  if ((n_vectors + 3) / 4 > 0x7fffffffLL) return OKQ_ERR_CAPACITY;
  auto go = [&](auto kernel) {
    launch_dependent(kernel, dim3((unsigned)((n_vectors + W - 1) / W)), 128, 0, static_cast<cudaStream_t>(stream), 1, 
        codes, static_cast<const __half*>(norms), n_vectors, signs, x_hat);
  };
  if (bits == 2) go(k_turboquant_decode<2>);
  else if (bits == 3) go(k_turboquant_decode<3>);
  else go(k_turboquant_decode<4>);
  return launch_status();
}

}  // extern "C"
