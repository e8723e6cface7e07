// Norm and randomised Hadamard transform (Eq. 2) of up to 32 rows by 128 threads, shared by the key quantisers and the
// baseline codec.
#pragma once
#include "okq_device.cuh"

namespace okq {

constexpr int ZS = 144;  // row stride (floats) of the per-window staging buffers: neighbouring rows 16 banks apart

// Position of channel c inside a staged key row: the four 4-float chunks of every 16-channel block are
// rotated by (block >> 1), which makes the three access patterns of the key quantiser (16-byte stores of a
// block per thread, 8-byte accesses with stride 16 channels, 8-byte reads of the code-word order) free of
// shared-memory bank conflicts.
__device__ __forceinline__ int zpos(int c) {
  return (c & ~15) + 4 * ((((c >> 2) & 3) + ((c >> 5) & 3)) & 3) + (c & 3);
}

// two fp32 values in one 64-bit register and the packed arithmetic on them (each half rounds like the scalar op)
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// The 128-point transform is done in two in-register halves around one shared-memory transpose:
// eight threads per token first hold 16 consecutive channels each (stages h = 1, 2, 4, 8, and the
// first four levels of the norm's summation tree), then each holds the 2 x 8 channels that differ in
// the three high index bits (stages h = 16, 32, 64).  The stage order, and with it every rounding,
// is that of the plain butterfly loop.
// Rows i < n_rows of `rows` (element stride `stride`) -> z[i * ZS + zpos(c)] = (H x)_c / |x|_16 (zeros for a zero row and
// for rows beyond n_rows); store_norm(i, fp16 norm) is called once per row, by its first thread.
template <class StoreNorm>
__device__ __forceinline__ void rotate_rows(const __half* rows, long long stride, int n_rows, const float* __restrict__ signs, float* z,
                                            StoreNorm store_norm) {
  const int tid = threadIdx.x;
  const int a = tid & 7;          // which 16-channel block (first half) / which channel pair (second half)
  uint64_t sgp[8];   // the signs of the thread's 16 channels, two per register
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const float4 s4 = *reinterpret_cast<const float4*>(signs + 16 * a + 4 * q);
    sgp[2 * q] = pack2(s4.x, s4.y); sgp[2 * q + 1] = pack2(s4.z, s4.w);
  }
#pragma unroll 1
  for (int round = 0; round < 2; round++) {
    const int i = (tid >> 3) + 16 * round;   // token; its eight threads are neighbours in one warp
    float* zrow = z + i * ZS;
    float y[16];
    {
      const uint4* src = reinterpret_cast<const uint4*>(rows + (long long)i * stride + 16 * a);
      const uint4 none = make_uint4(0u, 0u, 0u, 0u);
      const uint4 r0 = i < n_rows ? src[0] : none, r1 = i < n_rows ? src[1] : none;
      const __half2* h0 = reinterpret_cast<const __half2*>(&r0);
      const __half2* h1 = reinterpret_cast<const __half2*>(&r1);
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const float2 f0 = __half22float2(h0[q]), f1 = __half22float2(h1[q]);
        y[2 * q] = f0.x; y[2 * q + 1] = f0.y; y[8 + 2 * q] = f1.x; y[8 + 2 * q + 1] = f1.y;
      }
    }
    // Two channels per instruction (add / sub / mul .f32x2: each half is the same IEEE operation as the
    // scalar one, so the results do not change): P[i] = (y[2i], y[2i+1]).
    uint64_t P[8];
#pragma unroll
    for (int q = 0; q < 8; q++) P[q] = pack2(y[2 * q], y[2 * q + 1]);
    // norm: adjacent-pair tree (4 levels here, 3 across the eight threads)
    float t[16];
#pragma unroll
    for (int q = 0; q < 8; q++) unpack2(mul2(P[q], P[q]), t[2 * q], t[2 * q + 1]);
#pragma unroll
    for (int n = 8; n >= 1; n >>= 1)
#pragma unroll
      for (int c = 0; c < n; c++) t[c] = __fadd_rn(t[2 * c], t[2 * c + 1]);
    float ssum = t[0];
    ssum = __fadd_rn(ssum, __shfl_xor_sync(0xffffffffu, ssum, 1));
    ssum = __fadd_rn(ssum, __shfl_xor_sync(0xffffffffu, ssum, 2));
    ssum = __fadd_rn(ssum, __shfl_xor_sync(0xffffffffu, ssum, 4));
    float nrm = __fsqrt_rn(ssum);
    nrm = nrm > 65504.0f ? 65504.0f : nrm;
    const __half nh = __float2half_rn(nrm);
    const float nf = __half2float(nh);
    if (a == 0) store_norm(i, nh);
    const float cinv = nf != 0.0f ? __fdiv_rn(RSQRT_D, nf) : 0.0f;
    // D x, then stages h = 1, 2, 4, 8 inside the 16-channel block: h = 1 pairs the two halves of one P[i]
    // (scalar), h = 2, 4, 8 pair P[i] with P[i + h/2]
#pragma unroll
    for (int q = 0; q < 8; q++) {
      float lo, hi;
      unpack2(mul2(sgp[q], P[q]), lo, hi);
      P[q] = pack2(__fadd_rn(lo, hi), __fsub_rn(lo, hi));
    }
#pragma unroll
    for (int hh = 1; hh < 8; hh <<= 1)
#pragma unroll
      for (int j = 0; j < 8; j++)
        if ((j & hh) == 0) {
          const uint64_t p = P[j], q2 = P[j + hh];
          P[j] = add2(p, q2);
          P[j + hh] = sub2(p, q2);
        }
#pragma unroll
    for (int q = 0; q < 4; q++)
      *reinterpret_cast<ulonglong2*>(&zrow[zpos(16 * a + 4 * q)]) = make_ulonglong2(P[2 * q], P[2 * q + 1]);
    __syncwarp();
    // second half: channels 16*u + 2*a + e, u = 0..7: stages h = 16, 32, 64 act on u; Q[u] = both e
    uint64_t Q[8];
#pragma unroll
    for (int u = 0; u < 8; u++) Q[u] = *reinterpret_cast<const uint64_t*>(&zrow[zpos(16 * u + 2 * a)]);
#pragma unroll
    for (int hh = 1; hh < 8; hh <<= 1)
#pragma unroll
      for (int j = 0; j < 8; j++)
        if ((j & hh) == 0) {
          const uint64_t p = Q[j], q2 = Q[j + hh];
          Q[j] = add2(p, q2);
          Q[j + hh] = sub2(p, q2);
        }
    __syncwarp();   // every thread of the token has read the first-half values before they are overwritten
    const uint64_t cinv2 = pack2(cinv, cinv);
#pragma unroll
    for (int u = 0; u < 8; u++)
      *reinterpret_cast<uint64_t*>(&zrow[zpos(16 * u + 2 * a)]) = nf != 0.0f ? mul2(Q[u], cinv2) : 0ull;
  }
}

// The butterflies of the second half alone are what the inverse needs too: eight threads hold 16 consecutive channels each
// (P[q] = channels 16 a + 2 q, + 1), leave with Q[u] = channels 16 u + 2 a, + 1 of the transform; zrow: 128 floats of scratch.
__device__ __forceinline__ void hadamard_eight(uint64_t (&P)[8], uint64_t (&Q)[8], float* zrow, int a) {
#pragma unroll
  for (int q = 0; q < 8; q++) {
    float lo, hi;
    unpack2(P[q], lo, hi);
    P[q] = pack2(__fadd_rn(lo, hi), __fsub_rn(lo, hi));
  }
#pragma unroll
  for (int hh = 1; hh < 8; hh <<= 1)
#pragma unroll
    for (int j = 0; j < 8; j++)
      if ((j & hh) == 0) {
        const uint64_t p = P[j], q2 = P[j + hh];
        P[j] = add2(p, q2);
        P[j + hh] = sub2(p, q2);
      }
#pragma unroll
  for (int q = 0; q < 4; q++)
    *reinterpret_cast<ulonglong2*>(&zrow[zpos(16 * a + 4 * q)]) = make_ulonglong2(P[2 * q], P[2 * q + 1]);
  __syncwarp();
#pragma unroll
  for (int u = 0; u < 8; u++) Q[u] = *reinterpret_cast<const uint64_t*>(&zrow[zpos(16 * u + 2 * a)]);
#pragma unroll
  for (int hh = 1; hh < 8; hh <<= 1)
#pragma unroll
    for (int j = 0; j < 8; j++)
      if ((j & hh) == 0) {
        const uint64_t p = Q[j], q2 = Q[j + hh];
        Q[j] = add2(p, q2);
        Q[j + hh] = sub2(p, q2);
      }
}

}  // namespace okq
