// Offline calibration of the per-modality value rotations (Eq. 5, R_m = H U_m^T).
//
//   k_calib_pass<0>, <1>          alpha = softmax(q k^T * scale) in 128 x 64 tiles on the tensor cores
//                                 (mma.sync, fp16 products, fp32 sums): first the row maximum and
//                                 normaliser, then the column sums of alpha^2; sequences of up to 256 tokens and
//                                 scales that are not positive (the others: okq_calib_scores.cu)
//   k_calib_wsum                  w_j: fixed-order sum of the per-(query tile, head) column sums
//   k_calib_wmax, k_calib_moments C_m = sum w_j v_j^T v_j, tensor cores, values staged transposed
//   k_calib_csum                  fixed-order sum of the per-chunk partial moments
//   k_calib_eigen                 cyclic Jacobi (fp64, one cluster), ordering, signs, R = H U^T, for the matrices
//                                 that the direct solver (okq_eigen.cu) leaves
#include <cooperative_groups.h>

#include "../../include/okq_calib.h"
#include "okq_calib_scores.cuh"
#include "okq_common.cuh"
#include "okq_device.cuh"
#include "okq_eigen.cuh"

namespace cg = cooperative_groups;

namespace okq {
namespace {

constexpr int TQ = 128;         // queries per block: 4 warps x 32 rows
constexpr int TK = 64;          // keys per staged tile
constexpr int TQ_WS = 64;       // query tile the documented workspace size is counted in
constexpr int KS_STRIDE = D + 8;  // halfs per staged key row: 272 bytes, conflict-free fragment reads

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}


// One pass over the key tiles of a 128-query block of one head; scores in the log2 domain, s = (q . k) * scale2.
//   PASS 0: rowstat[g * n + i] = (-2 m_i, 1 / l_i^2), m_i = max_j s_ij, l_i = sum_j 2^(s_ij - m_i)
//   PASS 1: column sums of alpha^2 = 2^(2 s - 2 m_i) / l_i^2 over the block's queries -> partial[(itile * G + g) * n + j]
// (The exponent is one fused multiply-add with a number that is exact: with m_i + log2 l_i in one number its rounding, 2^-24 of
// it, was an error of every weight of the row, 3e-6 at scores of 2^5.)
// A warp owns 32 query rows (its fragments stay in registers, so each key fragment serves two products) and keeps the
// running maximum and sum of its own columns per lane; the four lanes of a row meet once at the end.  Keys pass through
// two cp.async buffers.  What bounds it: the products' dispatch (8.6 cycles of a sub-partition each) and one exponential
// per score.  8192 tokens x 7 heads, both passes: 1.29 ms with 16 rows per warp, unbuffered tiles, scalar fragment loads and
// expf of every score with a shuffle reduction per tile, 0.57 ms in this form.
// Block order: longest first, every other wave of blocks reversed, so that an SM's blocks add up to about the same.
template <int PASS>
__global__ void __launch_bounds__(128, 3) k_calib_pass(const __half* __restrict__ q, const __half* __restrict__ k, int G, int n,
                                                      float scale2, int causal, int n_sm, float2* __restrict__ rowstat,
                                                      float* __restrict__ partial) {
  __shared__ __align__(16) __half ks[2][TK * KS_STRIDE];
  __shared__ float colsum[4][TK];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int n_it = (n + TQ - 1) / TQ, n_blk = gridDim.x;
  int id = blockIdx.x;
  {
    const int wave = id / n_sm, first = wave * n_sm, last = min(n_blk, first + n_sm) - 1;
    if (wave & 1) id = first + last - id;
  }
  const int itile = n_it - 1 - id / G, head = id % G;
  const __half* qh = q + (size_t)head * n * D;
  // the maximum below assumes a positive scale: a negative one goes into the queries' signs, zero into zero queries
  const uint32_t flip = scale2 < 0.f ? 0x80008000u : 0u;
  const bool no_q = scale2 == 0.f;
  scale2 = no_q ? 1.0f : fabsf(scale2);
  int row[2][2];   // this lane's query rows: [m-tile][upper / lower half]
  uint32_t qa[2][8][4];
#pragma unroll
  for (int mt = 0; mt < 2; mt++) {
    row[mt][0] = itile * TQ + warp * 32 + mt * 16 + g;
    row[mt][1] = row[mt][0] + 8;
#pragma unroll
    for (int s = 0; s < 8; s++)
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const int i = row[mt][e & 1], c = 16 * s + 2 * t + 8 * (e >> 1);
        qa[mt][s][e] = i < n && !no_q ? *reinterpret_cast<const uint32_t*>(qh + (size_t)i * D + c) ^ flip : 0u;
      }
  }
  float m[2][2], l[2][2];   // PASS 0: running maximum and sum; PASS 1: rowstat
#pragma unroll
  for (int mt = 0; mt < 2; mt++)
#pragma unroll
    for (int hf = 0; hf < 2; hf++) {
      const float2 st = PASS == 1 && row[mt][hf] < n ? rowstat[(size_t)head * n + row[mt][hf]] : make_float2(-INFINITY, 0.f);
      m[mt][hf] = st.x;
      l[mt][hf] = st.y;
    }
  const int n_jt = causal ? min((n + TK - 1) / TK, (itile * TQ + TQ - 1) / TK + 1) : (n + TK - 1) / TK;
  auto fetch = [&](int jt) {
    if (jt < n_jt)
#pragma unroll
      for (int u = 0; u < TK * (D / 8) / 128; u++) {
        const int idx = tid + 128 * u, r = idx >> 4, c8 = idx & 15, j = min(n - 1, jt * TK + r);   // (rows past the end: masked)
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&ks[jt & 1][r * KS_STRIDE + c8 * 8]);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(k + (size_t)j * D + c8 * 8));
      }
    asm volatile("cp.async.commit_group;\n" ::);
  };
  fetch(0);
  for (int jt = 0; jt < n_jt; jt++) {
    fetch(jt + 1);
    asm volatile("cp.async.wait_group 1;\n" ::);
    __syncthreads();
    const __half* kt = ks[jt & 1];
    // masks matter on the last tiles only (and in rows of no token: their zero queries times infinite keys are NaN)
    const bool edge = (jt + 1) * TK > n || itile * TQ + warp * 32 + 32 > n || (causal && (jt + 1) * TK - 1 > itile * TQ + warp * 32);
#pragma unroll
    for (int half = 0; half < 2; half++) {   // 32 keys at a time
      float d[2][4][4];
#pragma unroll
      for (int mt = 0; mt < 2; mt++)
#pragma unroll
        for (int nt = 0; nt < 4; nt++)
#pragma unroll
          for (int e = 0; e < 4; e++) d[mt][nt][e] = 0.f;
#pragma unroll
      for (int s2 = 0; s2 < 4; s2++)         // two k-steps per fragment load
#pragma unroll
        for (int nt = 0; nt < 4; nt++) {
          uint32_t kb[4];
          ldsm_x4(kb, kt + (half * 32 + nt * 8 + (lane & 7)) * KS_STRIDE + 32 * s2 + 8 * (lane >> 3));
#pragma unroll
          for (int mt = 0; mt < 2; mt++) {
            mma16816(d[mt][nt], qa[mt][2 * s2][0], qa[mt][2 * s2][1], qa[mt][2 * s2][2], qa[mt][2 * s2][3], kb[0], kb[1]);
            mma16816(d[mt][nt], qa[mt][2 * s2 + 1][0], qa[mt][2 * s2 + 1][1], qa[mt][2 * s2 + 1][2], qa[mt][2 * s2 + 1][3], kb[2], kb[3]);
          }
        }
      if (edge) {
#pragma unroll
        for (int mt = 0; mt < 2; mt++)
#pragma unroll
          for (int nt = 0; nt < 4; nt++)
#pragma unroll
            for (int e = 0; e < 4; e++) {
              const int j = jt * TK + half * 32 + nt * 8 + 2 * t + (e & 1), i = row[mt][e >> 1];
              if (j >= n || i >= n || (causal && j > i)) d[mt][nt][e] = -INFINITY;
            }
      }
      if (PASS == 0) {
#pragma unroll
        for (int mt = 0; mt < 2; mt++)
#pragma unroll
          for (int hf = 0; hf < 2; hf++) {
            float mx = -INFINITY;
#pragma unroll
            for (int nt = 0; nt < 4; nt++) mx = fmaxf(mx, fmaxf(d[mt][nt][2 * hf], d[mt][nt][2 * hf + 1]));
            const float mn = fmaxf(m[mt][hf], mx * scale2);
            if (mn != -INFINITY) {
              float a = l[mt][hf] * ex2(m[mt][hf] - mn);   // 0 for the first finite maximum
#pragma unroll
              for (int nt = 0; nt < 4; nt++)
                a += ex2(fmaf(d[mt][nt][2 * hf], scale2, -mn)) + ex2(fmaf(d[mt][nt][2 * hf + 1], scale2, -mn));
              l[mt][hf] = a;
              m[mt][hf] = mn;
            }
          }
      } else {
        const float two = 2.0f * scale2;
        float c[8];   // column 8 (i >> 1) + 2 t + (i & 1): sums over this lane's four rows
#pragma unroll
        for (int nt = 0; nt < 4; nt++)
#pragma unroll
          for (int e = 0; e < 2; e++)
            c[2 * nt + e] = fmaf(ex2(fmaf(d[0][nt][e], two, m[0][0])), l[0][0], ex2(fmaf(d[0][nt][2 + e], two, m[0][1])) * l[0][1]) +
                            fmaf(ex2(fmaf(d[1][nt][e], two, m[1][0])), l[1][0], ex2(fmaf(d[1][nt][2 + e], two, m[1][1])) * l[1][1]);
        // over the eight row groups, each lane ending with one column: n-tile bits 1, 0 and e by lane bits 4, 3, 2
#pragma unroll
        for (int w = 4, bit = 16; w >= 1; w >>= 1, bit >>= 1) {
          const bool up = (lane & bit) != 0;
#pragma unroll
          for (int i = 0; i < w; i++) {
            const float give = up ? c[i] : c[i + w], keep = up ? c[i + w] : c[i];
            c[i] = keep + __shfl_xor_sync(0xffffffffu, give, bit);
          }
        }
        colsum[warp][half * 32 + 8 * (g >> 1) + 2 * t + (g & 1)] = c[0];
      }
    }
    __syncthreads();   // the tile has been read (and the column sums are in place)
    if (PASS == 1) {
      if (tid < TK) {
        const int j = jt * TK + tid;
        if (j < n)
          partial[((size_t)itile * G + head) * n + j] = (colsum[0][tid] + colsum[1][tid]) + (colsum[2][tid] + colsum[3][tid]);
      }
      __syncthreads();
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::);
  if (PASS == 0) {
#pragma unroll
    for (int mt = 0; mt < 2; mt++)
#pragma unroll
      for (int hf = 0; hf < 2; hf++) {
        float mm = m[mt][hf], ll = l[mt][hf];
#pragma unroll
        for (int dl = 1; dl < 4; dl <<= 1) {
          const float mo = __shfl_xor_sync(0xffffffffu, mm, dl), lo = __shfl_xor_sync(0xffffffffu, ll, dl);
          const float mn = fmaxf(mm, mo);
          ll = (mm == -INFINITY ? 0.f : ll * ex2(mm - mn)) + (mo == -INFINITY ? 0.f : lo * ex2(mo - mn));
          mm = mn;
        }
        if (t == 0 && row[mt][hf] < n) rowstat[(size_t)head * n + row[mt][hf]] = make_float2(-2.0f * mm, 1.0f / (ll * ll));
      }
  }
}

// w_j = sum over (query tile, head) of the column sums, in a fixed order: a warp per 32 keys' slice, its lanes one key each;
// the block's warps take every eighth (tile, head) row and meet in shared memory
__global__ void __launch_bounds__(256) k_calib_wsum(const float* __restrict__ partial, int G, int n, int causal, float* __restrict__ w) {
  __shared__ float part[8][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, j = blockIdx.x * 32 + lane;
  const int rows = (n + TQ - 1) / TQ * G, r0 = causal ? (blockIdx.x * 32) / TQ * G : 0;
  float acc = 0.f;
  if (j < n)
#pragma unroll 4
    for (int r = r0 + warp; r < rows; r += 8) acc += partial[(size_t)r * n + j];
  part[warp][lane] = acc;
  __syncthreads();
  if (warp == 0 && j < n) {
    float s = 0.f;
    for (int i = 0; i < 8; i++) s += part[i][lane];
    w[j] = s;
  }
}

// ---------------------------------------------------------------- weighted moments

constexpr int MT = 32;             // tokens per staged tile (two k-steps)
constexpr int VT_STRIDE = MT + 8;  // halves per transposed row: 80 bytes
constexpr int MAX_CHUNKS = 64;     // token ranges (blocks) per modality

// exponent e with 2^e >= max_j w_j (0 when all weights are 0): the weights are used as w_j * 2^-e <= 1
__global__ void k_calib_wmax(const float* __restrict__ w, int n, int* __restrict__ e_out) {
  __shared__ float red[32];
  depend_wait();
  float mx = 0.f;
#pragma unroll 8
  for (int j = threadIdx.x; j < n; j += blockDim.x) mx = fmaxf(mx, w[j]);
  for (int d = 16; d; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < (int)(blockDim.x >> 5); i++) mx = fmaxf(mx, red[i]);
    int e = 0;
    if (mx > 0.f) { frexpf(mx, &e); }   // mx = f * 2^e, f in [0.5, 1)
    *e_out = e;
  }
}

// grid (n_chunks, 3), 256 threads: block (chunk, m) adds the tokens of modality m in its token range into
// a 128 x 128 partial moment matrix.  Warp w owns rows 16 w .. 16 w + 15 (all 128 columns).  A tile without a token of the modality
// is left out: modalities come in runs, so a tile is mostly one block's.  Staging puts a tile's 32 tokens on the lanes, whose
// transposed halves are then 64 contiguous bytes (channels on the lanes instead were sixteen stores on one bank).
// 8192 tokens, the three kernels: 55 -> 23 us.
__global__ void __launch_bounds__(256) k_calib_moments(const __half* __restrict__ v, const float* __restrict__ w,
                                                      const unsigned char* __restrict__ modality, int n, int n_chunks,
                                                      const int* __restrict__ w_exp, float* __restrict__ partial) {
  __shared__ __align__(16) __half vt[D * VT_STRIDE];    // values, transposed: [channel][token]
  __shared__ __align__(16) __half xh[D * VT_STRIDE];    // w v, high fp16 term
  __shared__ __align__(16) __half xl[D * VT_STRIDE];    // w v, low fp16 term
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int chunk = blockIdx.x, m = blockIdx.y;
  depend_wait();
  const int n_tiles = (n + MT - 1) / MT;
  const int per = (n_tiles + n_chunks - 1) / n_chunks;
  const int t_begin = chunk * per, t_end = min(n_tiles, t_begin + per);
  const float wscale = exp2f((float)-(*w_exp));
  float acc[16][4];
#pragma unroll
  for (int nt = 0; nt < 16; nt++)
#pragma unroll
    for (int e = 0; e < 4; e++) acc[nt][e] = 0.f;
  for (int tile = t_begin; tile < t_end; tile++) {
    const int j = tile * MT + lane;
    bool mine = false;
    if (j < n) {
      unsigned mm = modality[j];
      mm = mm > 2 ? 0 : mm;
      mine = (int)mm == m;
    }
    if (!__any_sync(0xffffffffu, mine)) continue;   // (the same in every warp)
    const float wj = mine ? w[j] * wscale : 0.f;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < D / 64; i++) {
      const int r = lane, c8 = warp + 8 * i;
      uint4 raw = make_uint4(0u, 0u, 0u, 0u);
      if (mine) raw = *reinterpret_cast<const uint4*>(v + (size_t)j * D + c8 * 8);
      const __half* hv = reinterpret_cast<const __half*>(&raw);
#pragma unroll
      for (int u = 0; u < 8; u++) {
        const float x = __half2float(hv[u]) * wj;
        const __half hi = __float2half_rn(x);
        vt[(c8 * 8 + u) * VT_STRIDE + r] = hv[u];
        xh[(c8 * 8 + u) * VT_STRIDE + r] = hi;
        xl[(c8 * 8 + u) * VT_STRIDE + r] = __float2half_rn(x - __half2float(hi));
      }
    }
    __syncthreads();
#pragma unroll
    for (int st = 0; st < MT / 16; st++) {
      const int row0 = (16 * warp + g) * VT_STRIDE + 16 * st + 2 * t, row1 = row0 + 8 * VT_STRIDE;
      const uint32_t h0 = *reinterpret_cast<const uint32_t*>(&xh[row0]), h1 = *reinterpret_cast<const uint32_t*>(&xh[row1]);
      const uint32_t h2 = *reinterpret_cast<const uint32_t*>(&xh[row0 + 8]), h3 = *reinterpret_cast<const uint32_t*>(&xh[row1 + 8]);
      const uint32_t l0 = *reinterpret_cast<const uint32_t*>(&xl[row0]), l1 = *reinterpret_cast<const uint32_t*>(&xl[row1]);
      const uint32_t l2 = *reinterpret_cast<const uint32_t*>(&xl[row0 + 8]), l3 = *reinterpret_cast<const uint32_t*>(&xl[row1 + 8]);
#pragma unroll
      for (int nt = 0; nt < 16; nt++) {
        const __half* br = &vt[(nt * 8 + g) * VT_STRIDE + 16 * st + 2 * t];
        const uint32_t b0 = *reinterpret_cast<const uint32_t*>(br), b1 = *reinterpret_cast<const uint32_t*>(br + 8);
        mma16816(acc[nt], h0, h1, h2, h3, b0, b1);
        mma16816(acc[nt], l0, l1, l2, l3, b0, b1);
      }
    }
  }
  float* out = partial + ((size_t)chunk * 3 + m) * D * D;
#pragma unroll
  for (int nt = 0; nt < 16; nt++) {
    const int col = nt * 8 + 2 * t, r0 = 16 * warp + g;
    *reinterpret_cast<float2*>(&out[r0 * D + col]) = make_float2(acc[nt][0], acc[nt][1]);
    *reinterpret_cast<float2*>(&out[(r0 + 8) * D + col]) = make_float2(acc[nt][2], acc[nt][3]);
  }
}

// C = 2^e * (sum of the partial matrices in chunk order), made exactly symmetric.  Block = a 32 x 32 tile on or above the diagonal of
// one matrix, and its mirror image; 1024 threads, an element of each.
__global__ void __launch_bounds__(1024) k_calib_csum(const float* __restrict__ partial, int n_chunks, const int* __restrict__ w_exp,
                                                    float* __restrict__ C) {
  __shared__ float mirror[32][33];
  depend_wait();
  const int m = blockIdx.y, r = threadIdx.x >> 5, c = threadIdx.x & 31;
  int ta = 0, tb = blockIdx.x;                 // tile (ta, tb), ta <= tb
  while (tb >= D / 32 - ta) { tb -= D / 32 - ta; ta++; }
  tb += ta;
  const float* p0 = partial + (size_t)m * D * D + (32 * ta + r) * D + 32 * tb + c;
  const float* p1 = partial + (size_t)m * D * D + (32 * tb + r) * D + 32 * ta + c;
  float s0 = 0.f, s1 = 0.f;
#pragma unroll 8
  for (int k = 0; k < n_chunks; k++) {
    s0 += p0[(size_t)k * 3 * D * D];
    s1 += p1[(size_t)k * 3 * D * D];
  }
  mirror[r][c] = s1;
  __syncthreads();
  const float val = 0.5f * (s0 + mirror[c][r]) * exp2f((float)*w_exp);
  if (ta < tb || r <= c) C[(size_t)m * D * D + (32 * ta + r) * D + 32 * tb + c] = val;
  __syncthreads();
  mirror[r][c] = val;
  __syncthreads();
  if (ta < tb || r > c) C[(size_t)m * D * D + (32 * tb + r) * D + 32 * ta + c] = mirror[c][r];
}

// ---------------------------------------------------------------- eigenbasis and rotation

constexpr int EIG_THREADS = 1024;
constexpr int MAX_SWEEPS = 30;
constexpr int NPOS = D / 2;                        // pairs per round
constexpr int NBLK = NPOS * (NPOS - 1) / 2;        // 2 x 2 blocks above the diagonal
constexpr int ROUNDS = D - 1;
constexpr int V_CTAS = 4, V_COLS = D / V_CTAS;     // blocks that carry the eigenvectors, columns of each

// Cyclic Jacobi on a symmetric 128 x 128 matrix, one cluster of 1 + V_CTAS blocks; the result is fp64-converged.
//
// The round-robin pairing is kept as a ring (Brent and Luk): after every round each index moves one place, so the pair
// k of a round is always positions (top k, bottom k) and a sweep of 127 rounds brings everybody home.  Block 0 holds the
// matrix in position order, upper half only, as 2 x 2 blocks (pair k, pair l), one plane per block element: a thread owns
// two blocks, reads them at fixed addresses, applies its rows' and its columns' rotation in registers and stores the
// results where the move takes them, at fixed addresses of a second buffer.  A pair's next off-diagonal element comes out
// of one such block, so 64 threads work out the next round's angles while everybody applies this round: one block barrier
// per round.  (With the matrix in place, rows first and columns then, it was 512 KB of shared-memory traffic per round,
// the eigenvectors' rows through L2 and three barriers: 5.2 us per round, 7.2 ms per matrix; now about 1.05 us, 1.48 ms.)
// The rotations of a sweep go to the other blocks, which apply them to V^T (row = eigenvector estimate, V_COLS columns
// each) while block 0 works on the next sweep.
// A round is bound by the chain of its angle threads (loads queued behind the other warps', about 1200 cycles in fp32, 1900
// in fp64) and by block 0's shared-memory traffic, so the first sweeps run on an fp32 copy of the
// matrix, at half the traffic: they only choose the angles.  The eigenvectors take the same rotations with fp64 cosines and
// stay orthogonal to fp64; V A V^T is then formed in fp64 from the original matrix and the fp64 sweeps finish on that.
// Angles are taken in fp32 throughout (the residual element is computed, not assumed zero, so that only costs a factor 1e-7
// per visit); cosine and sine of the fp64 rotations are orthonormal to fp64 by two Newton steps.  Stops after a sweep whose
// largest tangent was below 1e-8: what is left is quadratically smaller.
// Then: eigenvalues in descending order, every eigenvector with its largest-magnitude component positive, R = H U^T with
// H = Had_128 diag(signs) / sqrt(128), a Hadamard transform per column.
constexpr int CHUNK = 32;               // rounds whose rotations are worked out together
template <class T> struct __align__(2 * sizeof(T)) Pair2 { T x, y; };
template <class T> struct EigA {
  T buf[2][4 * NBLK];                   // off-diagonal planes [2 * row part + column part][block]
  __align__(16) Pair2<T> cs[2][NPOS];   // rotations of this round and of the next
  T dg[2][D];                           // diagonal, by position, after the rotations of the round (before its move)
  T own[NPOS];                          // the pairs' own off-diagonal elements at the start of a phase
  float tmax[2];                        // largest |tangent| of the sweep, per angle warp; 0: nothing rotated
};
struct EigV {
  double v[D][V_COLS];                  // V^T, rows by index
  union {
    double t[2][ROUNDS * NPOS];         // tangents of a sweep, written by block 0
    double other[V_CTAS - 1][D][V_COLS];   // between the phases: the other slices of V^T, then this slice's part of V A
  };
  union {
    double a[D][V_COLS];                // between the phases: this slice's columns of the matrix
    Pair2<double> cs[CHUNK][NPOS];      // rotations of the rounds being applied
  };
  double lam[D];
  double best[V_CTAS][D];               // per slice and eigenvector: the slice's component of largest magnitude
  int done[2];
  int order[D];
};
constexpr int EIG_SMEM = sizeof(EigA<double>) > sizeof(EigV) ? (int)sizeof(EigA<double>) : (int)sizeof(EigV);
constexpr int FP32_SWEEPS = 7;                     // at most; of 11 to 13 in all
static_assert(EIG_SMEM <= 227 * 1024, "shared memory of one block");

// position 2 k: top of pair k, 2 k + 1: bottom
__device__ __forceinline__ int eig_move(int pos) {
  const int k = pos >> 1;
  if ((pos & 1) == 0) return k == 0 ? 0 : (k == NPOS - 1 ? 2 * k + 1 : 2 * (k + 1));
  return k == 0 ? 2 : 2 * (k - 1) + 1;
}
// index that sits at a position in round r
__device__ __forceinline__ int eig_index(int pos, int r) {
  const int k = pos >> 1;
  if (pos == 0) return 0;
  int x = ((pos & 1) ? 2 * NPOS - 2 - k : k - 1) - r;
  return (x < 0 ? x + ROUNDS : x) + 1;
}
// blocks (k, l), k < l, numbered so that 32 warps own 63 each: warp w the rows w and 63 - w
__device__ __forceinline__ int eig_block(int k, int l) {
  return k < NPOS / 2 ? k * (NPOS - 1) + l - k - 1 : (NPOS - 1 - k) * (NPOS - 1) + k + (l - k - 1);
}
// where the element of positions (a, b) of different pairs is kept
__device__ __forceinline__ int eig_slot(int a, int b) {
  if ((a >> 1) > (b >> 1)) { const int x = a; a = b; b = x; }
  return (2 * (a & 1) + (b & 1)) * NBLK + eig_block(a >> 1, b >> 1);
}
// position of index i in round 0
__device__ __forceinline__ int eig_home(int i) { return i < NPOS ? 2 * i : 2 * (D - 1 - i) + 1; }
__device__ __forceinline__ Pair2<double> eig_cos_sin(double t) {   // c = 1 / sqrt(1 + t^2) to fp64, s = t c
  const double x = fma(t, t, 1.0), hx = 0.5 * x;
  double y = (double)rsqrtf((float)x);
  y = y * fma(-hx * y, y, 1.5);
  y = y * fma(-hx * y, y, 1.5);
  return {y, t * y};
}
__device__ __forceinline__ Pair2<float> eig_cos_sin(float t) {
  const float y = rsqrtf(fmaf(t, t, 1.0f));
  return {y, t * y};
}

// Block 0: sweeps on the matrix in sa (buf[0], own, dg[0] = diagonal by position) until the largest tangent of a sweep is at
// most `stop` or `max_sweeps` are done; an element is rotated if its magnitude exceeds `tiny` and its square `rel2` times the
// product of its diagonal elements.  Returns the number of sweeps that rotated something; *diag: the buffer of dg that holds
// the rotated diagonal of the last round.  One cluster barrier per sweep.
template <class T>
__device__ int eig_sweeps(cg::cluster_group& cluster, EigA<T>& sa, EigV& sv, T tiny, T rel2, float stop, int max_sweeps, int* diag) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // this thread's two blocks: where they are read, the rows' and columns' pairs, where their elements go.  Elements that
  // become a pair's own are worked out by its angle thread instead and dropped here (slot -1).
  int rd[2], pk[2], pl[2], wr[2][4];
#pragma unroll
  for (int u = 0; u < 2; u++) {
    const int j = lane + 32 * u;
    const bool first = j < NPOS - 1 - warp;
    pk[u] = first ? warp : NPOS - 1 - warp;
    pl[u] = first ? warp + 1 + j : NPOS - warp + (j - (NPOS - 1 - warp));
    rd[u] = warp * (NPOS - 1) + j;
    if (j >= NPOS - 1) { rd[u] = -1; pk[u] = 0; pl[u] = 1; }
#pragma unroll
    for (int e = 0; e < 4; e++) {
      const int pa = eig_move(2 * pk[u] + (e >> 1)), pb = eig_move(2 * pl[u] + (e & 1));
      wr[u][e] = (pa >> 1) == (pb >> 1) ? -1 : eig_slot(pa, pb);
    }
  }
  // Angle threads: thread dk < 64 has pair dk.  Of the round under way it knows the tangent t, the rotated pair's own
  // off-diagonal element res (moved like any other) and, through dg, the rotated diagonal.
  const int dk = tid & (NPOS - 1);
  const int d_off = eig_slot(eig_move(2 * dk), eig_move(2 * dk + 1));
  // positions that move to (top dk, bottom dk); always of two different pairs, the first one lower
  const int pa = dk == 0 ? 0 : (dk == 1 ? 1 : 2 * (dk - 1)), pb = dk == NPOS - 1 ? 2 * (NPOS - 1) : 2 * (dk + 1) + 1;
  const int src = eig_block(pa >> 1, pb >> 1);
  double* t_remote[V_CTAS];
#pragma unroll
  for (int r = 0; r < V_CTAS; r++) t_remote[r] = cluster.map_shared_rank(&sv.t[0][0], r + 1);
  T t = 0, res = 0;
  float tmax = 0.f;
  auto angle = [&](T app, T aqq, T apq, int to) {
    Pair2<T> cs = {1, 0};
    t = 0; res = apq;
    if ((apq < 0 ? -apq : apq) > tiny && apq * apq > rel2 * (app * aqq < 0 ? -(app * aqq) : app * aqq)) {
      const float tau = __fdividef((float)(aqq - app), 2.0f * (float)apq);
      float root;
      asm("sqrt.approx.ftz.f32 %0, %1;\n" : "=f"(root) : "f"(fmaf(tau, tau, 1.0f)));
      t = (T)__fdividef(copysignf(1.0f, tau), fabsf(tau) + root);
      cs = eig_cos_sin(t);
      res = cs.x * cs.x * ((1 - t * t) * apq + t * (app - aqq));
    }
    sa.cs[to][dk] = cs;
    sa.dg[to][2 * dk] = app - t * (apq + res);
    sa.dg[to][2 * dk + 1] = aqq + t * (apq + res);
  };
  __syncthreads();
  T app = 0, aqq = 0;
  if (tid < NPOS) { app = sa.dg[0][2 * dk]; aqq = sa.dg[0][2 * dk + 1]; angle(app, aqq, sa.own[dk], 0); }
  __syncthreads();
  int cur = 0, sweeps = 0, sweep = 0;
  for (;; sweep++) {
    const int tbase = (sweep & 1) * ROUNDS * NPOS;
#pragma unroll 1
    for (int round = 0; round < ROUNDS; round++) {
      const T* in = sa.buf[cur];
      T* out = sa.buf[cur ^ 1];
      const Pair2<T>* cs = sa.cs[cur];
      if (tid < NPOS) {
        out[d_off] = res;
        tmax = fmaxf(tmax, fabsf((float)t));
#pragma unroll
        for (int r = 0; r < V_CTAS; r++) t_remote[r][tbase + round * NPOS + dk] = (double)t;
        // the next round's pair: rows (c, -s) of a top, (s, c) of a bottom
        const Pair2<T> ca = cs[pa >> 1], cb = cs[pb >> 1];
        const T u0 = (pa & 1) ? ca.y : ca.x, u1 = (pa & 1) ? ca.x : -ca.y;
        const T w0 = (pb & 1) ? cb.y : cb.x, w1 = (pb & 1) ? cb.x : -cb.y;
        const T m0 = w0 * in[src] + w1 * in[NBLK + src], m1 = w0 * in[2 * NBLK + src] + w1 * in[3 * NBLK + src];
        angle(sa.dg[cur][pa], sa.dg[cur][pb], u0 * m0 + u1 * m1, cur ^ 1);
      }
#pragma unroll
      for (int u = 0; u < 2; u++)
        if (rd[u] >= 0) {
          T x[4];
#pragma unroll
          for (int e = 0; e < 4; e++) x[e] = in[e * NBLK + rd[u]];
          const Pair2<T> ck = cs[pk[u]], cl = cs[pl[u]];
          const T r00 = ck.x * x[0] - ck.y * x[2], r01 = ck.x * x[1] - ck.y * x[3];
          const T r10 = ck.y * x[0] + ck.x * x[2], r11 = ck.y * x[1] + ck.x * x[3];
          const T y[4] = {cl.x * r00 - cl.y * r01, cl.y * r00 + cl.x * r01, cl.x * r10 - cl.y * r11, cl.y * r10 + cl.x * r11};
#pragma unroll
          for (int e = 0; e < 4; e++)
            if (wr[u][e] >= 0) out[wr[u][e]] = y[e];
        }
      __syncthreads();
      cur ^= 1;
    }
    if (warp < 2) {
      for (int d = 16; d; d >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, d));
      if (lane == 0) sa.tmax[warp] = tmax;
      tmax = 0.f;
    }
    __syncthreads();
    const float mt = fmaxf(sa.tmax[0], sa.tmax[1]);
    if (mt > 0.0f) sweeps++;
    const bool done = !(mt > stop) || sweep + 1 >= max_sweeps;
    if (tid < V_CTAS) cluster.map_shared_rank(&sv.done[0], tid + 1)[sweep & 1] = done;
    cluster.sync();   // the sweep's tangents are in place; the sweep before has been applied
    if (done) break;
  }
  *diag = cur ^ 1;    // dg[cur] already has the rotations of a round that does not happen
  return sweeps;
}

// the other blocks: the sweeps of one phase applied to this slice of V^T
__device__ __forceinline__ void eig_apply(cg::cluster_group& cluster, EigV& sv) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int sweep = 0;; sweep++) {
    cluster.sync();
    const double* ts = sv.t[sweep & 1];
    for (int r0 = 0; r0 < ROUNDS; r0 += CHUNK) {
      const int nr = min(CHUNK, ROUNDS - r0);
      // each rotation once per block (every warp for itself: 900 cycles per round)
      for (int i = threadIdx.x; i < nr * NPOS; i += EIG_THREADS) (&sv.cs[0][0])[i] = eig_cos_sin(ts[r0 * NPOS + i]);
      __syncthreads();
      for (int round = r0; round < r0 + nr; round++) {
        // a warp takes two pairs, a lane one column
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const int k = warp + 32 * u;
          const Pair2<double> cs = sv.cs[round - r0][k];
          double* vp = &sv.v[eig_index(2 * k, round)][lane];
          double* vq = &sv.v[eig_index(2 * k + 1, round)][lane];
          const double a = *vp, b = *vq;
          *vp = cs.x * a - cs.y * b;
          *vq = cs.y * a + cs.x * b;
        }
        __syncthreads();
      }
    }
    if (sv.done[sweep & 1]) break;
  }
}

__global__ void __launch_bounds__(EIG_THREADS) k_calib_eigen(const float* __restrict__ C, const float* __restrict__ signs,
                                                           float* __restrict__ R, float* __restrict__ lambda,
                                                           int* __restrict__ sweeps_out) {
  extern __shared__ __align__(16) unsigned char eig_raw[];
  __shared__ double red[32];
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = blockIdx.x;
  EigV& sv = *reinterpret_cast<EigV*>(eig_raw);
  EigA<double>& sd = *reinterpret_cast<EigA<double>*>(eig_raw);
  EigA<float>& sf = *reinterpret_cast<EigA<float>*>(eig_raw);
  depend_wait();
  if (__float_as_uint(__ldcg(lambda)) != EIGEN_LEFT) return;   // the direct solver has done it
  cluster.sync();   // every block runs before its shared memory is written from outside
  // largest magnitude (the matrix is scaled by a power of two to at most 1) and trace
  double mx = 0.0, tr = 0.0;
  for (int i = tid; i < D * D; i += EIG_THREADS) mx = fmax(mx, fabs((double)C[i]));
  if (tid < D) tr = fabs((double)C[tid * D + tid]);
  for (int d = 16; d; d >>= 1) {
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, d));
    tr += __shfl_xor_sync(0xffffffffu, tr, d);
  }
  if (lane == 0) red[warp] = mx;
  __syncthreads();
  for (int i = 0; i < 32; i++) mx = fmax(mx, red[i]);
  __syncthreads();
  if (lane == 0 && warp < 4) red[warp] = tr;
  __syncthreads();
  int ex = 0;
  if (mx > 0.0) frexp(mx, &ex);   // mx < 2^ex
  const double scale = ldexp(1.0, -ex);
  auto element = [&](int i, int j) { return 0.5 * ((double)C[i * D + j] + (double)C[j * D + i]) * scale; };
  if (rank == 0) {
    for (int i = tid; i < D * D; i += EIG_THREADS) {
      const int a = i / D, b = i % D;
      if (a > b) continue;
      const float x = (float)element(eig_index(a, 0), eig_index(b, 0));
      if (a == b) sf.dg[0][a] = x;
      else if ((a >> 1) == (b >> 1)) sf.own[a >> 1] = x;
      else sf.buf[0][eig_slot(a, b)] = x;
    }
    int diag;
    // fp32: elements below the rounding noise of the largest or of their diagonal are left to the second phase
    int sweeps = eig_sweeps<float>(cluster, sf, sv, 1e-8f, 1e-13f, 1e-3f, FP32_SWEEPS, &diag);
    cluster.sync();   // V^T is complete
    cluster.sync();   // the products are ready
    for (int r = 0; r < V_CTAS; r++) cluster.sync();   // ... and added up here, slice by slice
    // the size below which an off-diagonal element is left alone
    const double tiny = fmax(((red[0] + red[1]) + (red[2] + red[3])) * scale * 1e-18, 1e-30);
    sweeps += eig_sweeps<double>(cluster, sd, sv, tiny, 1e-34, 1e-8f, MAX_SWEEPS - FP32_SWEEPS, &diag);
    if (tid == 0 && sweeps_out) *sweeps_out = sweeps;
    if (tid < D) {
      const double l = sd.dg[diag][tid] * ldexp(1.0, ex);
      const int idx = eig_index(tid, ROUNDS - 1);   // who sat there in the last round
      for (int r = 0; r < V_CTAS; r++) cluster.map_shared_rank(&sv.lam[0], r + 1)[idx] = l;
    }
    cluster.sync();   // eigenvalues are out
    cluster.sync();   // (the other blocks exchange their slices' largest components)
    return;
  }
  const int slice = rank - 1, col0 = slice * V_COLS;
  for (int i = tid; i < D * V_COLS; i += EIG_THREADS) {
    sv.v[i / V_COLS][i % V_COLS] = i / V_COLS == col0 + i % V_COLS ? 1.0 : 0.0;
  }
  __syncthreads();
  eig_apply(cluster, sv);
  cluster.sync();     // V^T is complete
  {
    // this slice's columns of V^T A: all of V^T (the other slices from their blocks) times the slice's columns of A
    for (int i = tid; i < D * V_COLS; i += EIG_THREADS) sv.a[i / V_COLS][i % V_COLS] = element(i / V_COLS, col0 + i % V_COLS);
    for (int o = 1; o < V_CTAS; o++) {
      const double* src = cluster.map_shared_rank(&sv.v[0][0], (slice + o) % V_CTAS + 1);
      for (int i = tid; i < D * V_COLS; i += EIG_THREADS) (&sv.other[o - 1][0][0])[i] = src[i];
    }
    __syncthreads();
    double z[4] = {0.0, 0.0, 0.0, 0.0};   // rows l = warp + 32 i, column lane
    for (int o = 0; o < V_CTAS; o++) {
      const double (*v)[V_COLS] = o == 0 ? sv.v : sv.other[o - 1];
      const int i0 = (slice + o) % V_CTAS * V_COLS;
      for (int i = 0; i < V_COLS; i++) {
        const double x = sv.a[i0 + i][lane];
#pragma unroll
        for (int q = 0; q < 4; q++) z[q] = fma(v[warp + 32 * q][i], x, z[q]);
      }
    }
    cluster.sync();   // every slice has been read: the space is free for the products
    double (*zs)[V_COLS] = sv.other[0];
#pragma unroll
    for (int q = 0; q < 4; q++) zs[warp + 32 * q][lane] = z[q];
    __syncthreads();
    // this slice's share of V^T A V: rows l = warp + 32 i, columns m = lane + 32 k
    double p[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int k = 0; k < 4; k++) p[i][k] = 0.0;
    for (int jj = 0; jj < V_COLS; jj++) {
      const int j = (jj + lane) & (V_COLS - 1);   // (a column of V^T per step would put all lanes on one bank pair)
      double vm[4];
#pragma unroll
      for (int k = 0; k < 4; k++) vm[k] = sv.v[lane + 32 * k][j];
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const double x = zs[warp + 32 * i][j];
#pragma unroll
        for (int k = 0; k < 4; k++) p[i][k] = fma(x, vm[k], p[i][k]);
      }
    }
    EigA<double>& dst = *cluster.map_shared_rank(&sd, 0);
    for (int r = 0; r < V_CTAS; r++) {   // added up in block 0, in slice order
      if (r == slice)
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
          for (int k = 0; k < 4; k++) {
            const int a = eig_home(warp + 32 * i), b = eig_home(lane + 32 * k);
            if (a > b) continue;
            double* at = a == b ? &dst.dg[0][a] : (a >> 1) == (b >> 1) ? &dst.own[a >> 1] : &dst.buf[0][eig_slot(a, b)];
            *at = r == 0 ? p[i][k] : *at + p[i][k];
          }
      cluster.sync();
    }
  }
  eig_apply(cluster, sv);
  cluster.sync();   // eigenvalues are here
  if (tid < D) {    // the slice's component of largest magnitude (the first of equals), to all slices
    double best = 0.0, val = 0.0;
    for (int j = 0; j < V_COLS; j++) {
      const double x = sv.v[tid][j];
      if (fabs(x) > best) { best = fabs(x); val = x; }
    }
    for (int r = 0; r < V_CTAS; r++) cluster.map_shared_rank(&sv.best[0][0], r + 1)[(rank - 1) * D + tid] = val;
    // descending order, ties by index, on the numbers' bit patterns made monotone: a permutation whatever the input (NaN too)
    auto key = [](double x) {
      const long long b = __double_as_longlong(x + 0.0);   // (-0 counts as 0)
      return b < 0 ? b ^ 0x7fffffffffffffffll : b;
    };
    const double li = sv.lam[tid];
    const long long ki = key(li);
    int pos = 0;
    for (int j = 0; j < D; j++) {
      const long long kj = key(sv.lam[j]);
      pos += (kj > ki) || (kj == ki && j < tid);
    }
    sv.order[pos] = tid;
    if (rank == 1) lambda[pos] = (float)li;
  }
  cluster.sync();
  {  // R[c][k] = sum_l H[c][l] U[k][l]: warp = column k, lane holds l = lane + 32 i
    double x[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const int l = lane + 32 * i, src = sv.order[l];
      double best = 0.0, val = 1.0;
      for (int r = 0; r < V_CTAS; r++)
        if (fabs(sv.best[r][src]) > best) { best = fabs(sv.best[r][src]); val = sv.best[r][src]; }
      x[i] = (val < 0.0 ? -1.0 : 1.0) * (double)signs[l] * sv.v[src][warp];
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const double o = __shfl_xor_sync(0xffffffffu, x[i], d);
        x[i] = (lane & d) ? o - x[i] : x[i] + o;
      }
    const double y0 = x[0] + x[1], y1 = x[0] - x[1], y2 = x[2] + x[3], y3 = x[2] - x[3];
    const double o[4] = {y0 + y2, y1 + y3, y0 - y2, y1 - y3};
#pragma unroll
    for (int i = 0; i < 4; i++) R[(size_t)(lane + 32 * i) * D + col0 + warp] = (float)(o[i] * 0.08838834764831845);   // 1 / sqrt(128)
  }
}

size_t attn_bytes(int group, int n) {
  const size_t n_it = (size_t)(n + TQ_WS - 1) / TQ_WS;
  return ((size_t)group * n * 2 + n_it * group * n) * sizeof(float);
}
constexpr size_t EIGEN_BYTES = (size_t)D * D * sizeof(double);   // what the rotation documents; it touches none of it
size_t moments_bytes() { return (size_t)MAX_CHUNKS * 3 * D * D * sizeof(float) + 16; }

}  // namespace
}  // namespace okq

using namespace okq;

extern "C" {

size_t okq_calib_workspace_bytes(int32_t group, int32_t n) {
  if (group <= 0 || n <= 0) return 0;
  size_t b = attn_bytes(group, n);
  if (moments_bytes() > b) b = moments_bytes();
  if (EIGEN_BYTES > b) b = EIGEN_BYTES;
  return (b + 255) & ~(size_t)255;
}

static okq_status attention_weights(const void* q_fp16, const void* k_fp16, int32_t group, int32_t n, float sm_scale, int32_t causal,
                                    void* workspace, size_t workspace_bytes, float* w_out, long long wait_limit, int skip_step, void* stream) {
  if (!q_fp16 || !k_fp16 || !w_out || !workspace || group <= 0 || n <= 0) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(q_fp16) || !aligned16(k_fp16) || !aligned16(workspace) || !aligned16(w_out)) return OKQ_ERR_ALIGNMENT;
  if (workspace_bytes < attn_bytes(group, n)) return OKQ_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int n_sm = sm_count();
  const __half* q = static_cast<const __half*>(q_fp16);
  const __half* k = static_cast<const __half*>(k_fp16);
  const float scale2 = sm_scale * 1.4426950408889634f;
  if (n >= SCORE_MIN_TOKENS && scale2 > 0.f) {   // (a zero or negative scale: the kernels that take any)
    const cudaError_t e = launch_calib_scores(q, k, group, n, scale2, causal, n_sm, workspace, w_out, wait_limit, skip_step, s);
    if (e != cudaSuccess) { set_last_cuda_error((int)e); return OKQ_ERR_CUDA; }
    return OKQ_OK;
  }
  float2* rowstat = static_cast<float2*>(workspace);
  float* partial = reinterpret_cast<float*>(rowstat + (size_t)group * n);
  const int grid = (n + TQ - 1) / TQ * group;
  k_calib_pass<0><<<grid, 128, 0, s>>>(q, k, group, n, scale2, causal, n_sm, rowstat, partial);
  k_calib_pass<1><<<grid, 128, 0, s>>>(q, k, group, n, scale2, causal, n_sm, rowstat, partial);
  k_calib_wsum<<<(n + 31) / 32, 256, 0, s>>>(partial, group, n, causal, w_out);
  return launch_status();
}

okq_status okq_calib_attention_weights(const void* q_fp16, const void* k_fp16, int32_t group, int32_t n,
                                       float sm_scale, int32_t causal, void* workspace, size_t workspace_bytes,
                                       float* w_out, void* stream) {
  return attention_weights(q_fp16, k_fp16, group, n, sm_scale, causal, workspace, workspace_bytes, w_out, 0, -1, stream);
}

okq_status okq_debug_calib_timeout(const void* q_fp16, const void* k_fp16, int32_t group, int32_t n, void* workspace,
                                   size_t workspace_bytes, float* w_out, int64_t limit_clocks, void* stream) {
  return attention_weights(q_fp16, k_fp16, group, n, 0.08838834764831845f, 1, workspace, workspace_bytes, w_out, limit_clocks, 0, stream);
}

okq_status okq_calib_moments(const void* v_fp16, const float* w, const uint8_t* modality, int32_t n,
                             void* workspace, size_t workspace_bytes, float* C_out, void* stream) {
  if (!v_fp16 || !w || !modality || !C_out || !workspace || n <= 0) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(v_fp16) || !aligned16(workspace) || !aligned16(C_out)) return OKQ_ERR_ALIGNMENT;
  if (workspace_bytes < moments_bytes()) return OKQ_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  float* partial = static_cast<float*>(workspace);
  int* w_exp = reinterpret_cast<int*>(partial + (size_t)MAX_CHUNKS * 3 * D * D);
  const int n_tiles = (n + MT - 1) / MT;
  const int n_chunks = n_tiles < MAX_CHUNKS ? n_tiles : MAX_CHUNKS;
  cudaError_t e = launch_dependent(k_calib_wmax, dim3(1), 1024, 0, s, 1, w, n, w_exp);
  if (e == cudaSuccess)
    e = launch_dependent(k_calib_moments, dim3(n_chunks, 3), 256, 0, s, 1, static_cast<const __half*>(v_fp16), w, modality, n, n_chunks, w_exp, partial);
  constexpr int TILES = D / 32 * (D / 32 + 1) / 2;
  if (e == cudaSuccess) e = launch_dependent(k_calib_csum, dim3(TILES, 3), 1024, 0, s, 1, partial, n_chunks, w_exp, C_out);
  if (e != cudaSuccess) { set_last_cuda_error((int)e); return OKQ_ERR_CUDA; }
  return launch_status();
}

okq_status okq_calib_rotation(const float* C, const float* signs, void* workspace, size_t workspace_bytes,
                              float* R_out, float* lambda_out, int32_t* sweeps_out, void* stream) {
  if (!C || !signs || !workspace || !R_out || !lambda_out) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(C) || !aligned16(workspace) || !aligned16(R_out)) return OKQ_ERR_ALIGNMENT;
  if (workspace_bytes < EIGEN_BYTES) return OKQ_ERR_WORKSPACE;
  static thread_local unsigned long long attr_mask = 0;
  int attr_dev = 0;
  if (attr_needed(attr_mask, attr_dev)) {
    cudaError_t e = cudaFuncSetAttribute(k_calib_eigen, cudaFuncAttributeMaxDynamicSharedMemorySize, EIG_SMEM);
    if (e != cudaSuccess) { set_last_cuda_error((int)e); return OKQ_ERR_CUDA; }
    attr_done(attr_mask, attr_dev);
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = launch_calib_spectrum(C, signs, R_out, lambda_out, sweeps_out, st);
  if (e == cudaSuccess)
    e = launch_dependent(k_calib_eigen, dim3(1 + V_CTAS), EIG_THREADS, EIG_SMEM, st, 1 + V_CTAS, C, signs, R_out, lambda_out, sweeps_out);
  if (e != cudaSuccess) { set_last_cuda_error((int)e); return OKQ_ERR_CUDA; }
  return launch_status();
}

okq_status okq_debug_calib_direct(const float* C, const float* signs, float* R_out, float* lambda_out, int32_t* sweeps_out, void* stream) {
  if (!C || !signs || !R_out || !lambda_out) return OKQ_ERR_INVALID_ARG;
  if (!aligned16(C) || !aligned16(R_out)) return OKQ_ERR_ALIGNMENT;
  const cudaError_t e = launch_calib_spectrum(C, signs, R_out, lambda_out, sweeps_out, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) { set_last_cuda_error((int)e); return OKQ_ERR_CUDA; }
  return launch_status();
}

}  // extern "C"
