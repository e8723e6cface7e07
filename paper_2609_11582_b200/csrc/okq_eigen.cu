// Direct eigensolver of the calibration: one symmetric 128 x 128 matrix by one cluster of eight blocks, all in fp64.
//
//   1. Householder reduction to a tridiagonal matrix (block 0, the matrix in registers); the reflectors go to R's place
//   2. eigenvalues by 33-section on Sturm counts, two eigenvalues per warp, 16 per block
//   3. eigenvectors of the tridiagonal matrix from its two factorisations, twisted where the residual is least
//   4. the reflectors applied to them, half a warp per two vectors
//   5. Newton-Schulz steps V <- V (3 I - V^T V) / 2 on the fp64 tensor cores: vectors of close eigenvalues, orthogonal only to
//      (rounding / gap) after step 3, become orthogonal to fp64
//   6. descending order, signs, R = H U^T
//
// Every vector's residual is known from step 3, and orthonormal vectors with small residuals are a complete eigenbasis: if a
// residual is not at rounding level, or V^T V is too far from the identity for step 5 (equal eigenvalues of one tridiagonal
// block; exhausted reductions - zero, diagonal, low-rank matrices - fall apart into blocks and are no such case), the call is
// left to the Jacobi solver, which needs no gaps: it runs behind this kernel and returns at once when there is nothing to do.
//
// Its errors are roundings of the largest eigenvalue, the Jacobi solver's those of the channels involved: a matrix whose channels
// differ in scale has small eigenvalues that only the latter keeps.  Scales from 1 to 1e-6 over the channels: the smallest to
// 3e-6 here, to fp32 there.  So matrices with diagonal elements below 2^-20 of the largest (and channels that are zero, whose
// eigenvalues stay exactly 0) go there at once; at that ratio the error, 1e-16 times 2^20, is still hidden behind fp32's 6e-8.
//
// What the blocks exchange - the reflectors, then the vectors - passes through R's own 64 KB and shared memory: the workspace stays
// untouched, so that calls which overlap may share it.
//
// Why: cyclic Jacobi is 11 to 13 sweeps of 127 dependent rounds of about a microsecond, whatever the number of SMs; the
// reduction is 126 dependent steps of 0.9 us, and everything behind it is parallel over the vectors.  One matrix 1503 -> 201 us
// (cycles: reduction 214 000, eigenvalues 82 000, tridiagonal vectors 20 000, reflectors 40 000, Newton-Schulz 19 000, the rest 12 000);
// a matrix that is left to the Jacobi solver after the reduction pays both (two eigenvalues, 64 times each: 2.60 -> 2.75 ms).
#include <cooperative_groups.h>
#include <type_traits>

#include "okq_common.cuh"
#include "okq_eigen.cuh"

namespace cg = cooperative_groups;

namespace okq {
namespace {

constexpr int CTAS = 8, THREADS = 256, WARPS = THREADS / 32;
constexpr int VEC = D / CTAS;               // eigenvectors of a block
constexpr int PITCH = D + 4;                // doubles per row: the fragment reads of a half-warp fall on all 32 banks
static_assert(VEC == 2 * WARPS, "two eigenvalues per warp");

constexpr double EPS = 0x1p-53;
constexpr double RESIDUAL_TOL = 512.0;      // in EPS times the matrix's size
constexpr float GRADED = 0x1p-20f;          // ratio of diagonal elements below which a matrix is left to the Jacobi solver
constexpr int MAX_STEPS = 8;                // Newton-Schulz steps: 0.5 -> 0.19 -> 0.03 -> 5e-4 -> 2e-7 -> 3e-14, and one to spare

struct Smem {
  union {
    __align__(16) double refl[D][D];        // reflectors (copies)
    double all[D][PITCH];                   // all eigenvectors (rows), gathered from the blocks
  };
  __align__(16) double own[VEC][PITCH];     // this block's eigenvectors
  union {
    struct {                                // reduction (block 0)
      __align__(16) double x[D], y[D], a1[D];   // tail of the column, matrix times it, next column
      __align__(16) double v[D], w[D];      // reflector, update vector
      __align__(16) double part[WARPS];
      double alpha, gamma, tau;
    } red;
    double2 seq[VEC][2][D];                 // consecutive terms of the two Sturm sequences of a vector
    struct {
      double cross[D / 4][6];               // products of the reflectors of a group of four
    } wy;
    struct {
      __align__(16) double g[VEC][PITCH];   // rows of V^T V
    } ns;
  };
  double2 de[D];                            // (d_i, e_{i-1}^2) of the tridiagonal matrix
  double d[D], e[D], tau[D];
  double lam[D];                            // all eigenvalues (by position)
  double err[CTAS];                         // squared distance of V^T V from the identity, per block; NaN if a residual is too large
  double redw[WARPS];
  int order[D];
  int expo;
};
static_assert(sizeof(Smem) <= 227 * 1024, "shared memory of one block");

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int s = 16; s; s >>= 1) x += __shfl_xor_sync(0xffffffffu, x, s);
  return x;
}

// fp64 tensor-core product, 8 x 8 x 4: a = A[lane / 4][lane % 4], b = B[lane % 4][lane / 4], c = C[lane / 4][2 (lane % 4) + {0, 1}]
__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
  asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}

__device__ __forceinline__ void copy_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem));
}

// both numbers times the power of two that brings the larger near one (sequences that grow or shrink; nothing if both are tiny)
__device__ __forceinline__ void rescale(double& p, double& q) {
  const int e = max(__double2hiint(p) & 0x7ff00000, __double2hiint(q) & 0x7ff00000);
  const double f = e == 0 || e >= 0x7fe00000 ? 1.0 : __hiloint2double(0x7fe00000 - e, 0);
  p *= f;
  q *= f;
}

// 1 / sqrt(x) and 1 / x for normal x: the hardware's approximation (20 bits) and two Newton steps
__device__ __forceinline__ double fast_rsqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;\n" : "=d"(y) : "d"(x));
  const double h = 0.5 * x;
  y = y * fma(-h * y, y, 1.5);
  return y * fma(-h * y, y, 1.5);
}
__device__ __forceinline__ double fast_rcp(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;\n" : "=d"(y) : "d"(x));
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}

// Step 1.  Half-warp h holds the rows 8 h .. 8 h + 7, its lane u the columns 32 j + 2 u + {0, 1}, j = 0..3.  Step k: with the tail
// x of column k below its first element alpha, the reflector is v = x + gamma e_{k+1}, gamma = alpha + sign(alpha) |column|,
// tau = 2 / v^T v, and the rest of the matrix becomes A - v w^T - w v^T, w = tau A v - (tau^2 / 2)(v^T A v) v.  A v comes from
// y = A x and the next column, so the product can start before the norm is known; warp 0, whose rows are done first, works out
// the scalars meanwhile.  The update of a step is made together with the product of the next one, whose column is worked out
// ahead of it, an element per thread: two block barriers per step.
// What bounds it: the chain of a step (product 200 cycles, sums over 16 lanes 46 per level, barriers 40), and shared memory, which
// delivers 128 bytes a cycle however many lanes read the same number: a tile of 8 x 8 elements per thread uses each number it
// loads eight times.  Steps of product, w and update behind three barriers took 2500 cycles (3100 with one row per thread).
// Reflector k has components k + 1 .. 127: two of them share a row of 128 numbers of `rows`, and all fit into 64.  Row r: reflector r
// from the left, 126 - r reversed.
__device__ void reduce_to_tridiagonal(Smem& sm, const float* __restrict__ C, double* __restrict__ rows) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, u = lane & 15, r0 = 8 * (tid >> 4);
  auto& rd = sm.red;
  double a[8][8];
  float mx = 0.f;
#pragma unroll
  for (int i = 0; i < 8; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int r = r0 + i, c = 32 * j + 2 * u;
      const float2 x = *reinterpret_cast<const float2*>(C + r * D + c);
      const float t0 = C[c * D + r], t1 = C[(c + 1) * D + r];
      mx = fmaxf(mx, fmaxf(fabsf(x.x), fabsf(x.y)));
      a[i][2 * j] = 0.5 * ((double)x.x + (double)t0);
      a[i][2 * j + 1] = 0.5 * ((double)x.y + (double)t1);
    }
  for (int s = 16; s; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
  if (lane == 0) sm.redw[warp] = mx;
  __syncthreads();
  for (int i = 0; i < WARPS; i++) mx = fmaxf(mx, (float)sm.redw[i]);
  int ex = 0;
  if (mx > 0.f) frexp((double)mx, &ex);     // mx < 2^ex: the matrix is used with magnitudes of at most 1
  if (tid == 0) sm.expo = ex;
  const double scale = ldexp(1.0, -ex);
#pragma unroll
  for (int i = 0; i < 8; i++)
#pragma unroll
    for (int j = 0; j < 8; j++) a[i][j] *= scale;
  // row 0 of the matrix = its column 0: the tail, the element before it
  if (r0 == 0) {
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int c = 32 * j + 2 * u;
      *reinterpret_cast<double2*>(&rd.x[c]) = make_double2(c > 1 ? a[0][2 * j] : 0.0, c > 0 ? a[0][2 * j + 1] : 0.0);
    }
    if (u == 0) { sm.d[0] = a[0][0]; rd.alpha = a[0][1]; }
  }
  if (tid < D) { rd.v[tid] = 0.0; rd.w[tid] = 0.0; }
  __syncthreads();
  double* to = rows + tid;
  int step = D;
#pragma unroll 1
  for (int k = 0; k < D - 2; k++) {
    if (warp == 0) {
      const double2 x0 = *reinterpret_cast<const double2*>(&rd.x[2 * lane]), x1 = *reinterpret_cast<const double2*>(&rd.x[64 + 2 * lane]);
      const double s2 = warp_sum((x0.x * x0.x + x0.y * x0.y) + (x1.x * x1.x + x1.y * x1.y));
      const double al = rd.alpha;
      double beta = al, gamma = 0.0, tau = 0.0;   // nothing to reflect
      if (s2 > 1e-280) {
        const double n2 = fma(al, al, s2), nrm = n2 * fast_rsqrt(n2);
        beta = al > 0.0 ? -nrm : nrm;
        gamma = al - beta;
        tau = 2.0 * fast_rcp(fma(gamma, gamma, s2));
      }
      if (lane == 0) { rd.gamma = gamma; rd.tau = tau; sm.e[k] = beta; sm.tau[k] = tau; }
    }
    if (16 * warp + 15 > k) {   // (of a warp's rows some may be finished: x is zero there, and their results are not used)
      double v[8], w[8], s[8];
#pragma unroll
      for (int i = 0; i < 8; i += 2) {
        const double2 f = *reinterpret_cast<const double2*>(&rd.v[r0 + i]), g = *reinterpret_cast<const double2*>(&rd.w[r0 + i]);
        v[i] = -f.x; v[i + 1] = -f.y;
        w[i] = -g.x; w[i + 1] = -g.y;
        s[i] = s[i + 1] = 0.0;
      }
#pragma unroll
      for (int j = 0; j < 4; j++)
        if (32 * j + 31 > k) {
          const int c = 32 * j + 2 * u;
          const double2 cv = *reinterpret_cast<const double2*>(&rd.v[c]), cw = *reinterpret_cast<const double2*>(&rd.w[c]);
          const double2 x = *reinterpret_cast<const double2*>(&rd.x[c]);
#pragma unroll
          for (int i = 0; i < 8; i++) {
            a[i][2 * j] = fma(v[i], cw.x, fma(w[i], cv.x, a[i][2 * j]));
            a[i][2 * j + 1] = fma(v[i], cw.y, fma(w[i], cv.y, a[i][2 * j + 1]));
            s[i] = fma(a[i][2 * j + 1], x.y, fma(a[i][2 * j], x.x, s[i]));
          }
        }
      double p = 0.0, p1 = 0.0;
#pragma unroll
      for (int i = 0; i < 8; i += 2) {
        const double2 xr = *reinterpret_cast<const double2*>(&rd.x[r0 + i]);
        p = fma(xr.x, s[i], p);
        p1 = fma(xr.y, s[i + 1], p1);
      }
      p += p1;
      // the rows' sums over the half-warp: three exchanges leave each lane one row, one more finishes it
      auto exchange = [&](auto n) {
        constexpr int N = decltype(n)::value;
        const bool up = (lane & (2 * N)) != 0;
#pragma unroll
        for (int i = 0; i < N; i++) {
          const double give = up ? s[i] : s[i + N], keep = up ? s[i + N] : s[i];
          s[i] = keep + __shfl_xor_sync(0xffffffffu, give, 2 * N);
        }
        p += __shfl_xor_sync(0xffffffffu, p, 2 * N);
      };
      exchange(std::integral_constant<int, 4>());
      exchange(std::integral_constant<int, 2>());
      exchange(std::integral_constant<int, 1>());
      const double y = s[0] + __shfl_xor_sync(0xffffffffu, s[0], 1);
      p += __shfl_xor_sync(0xffffffffu, p, 1);
      p += __shfl_xor_sync(0xffffffffu, p, 16);
      const int r = r0 + (u >> 1);
      if ((lane & 1) == 0) rd.y[r] = y;
      if (lane == 0) rd.part[warp] = p;
#pragma unroll
      for (int i = 0; i < 8; i++)
        if (r0 + i == k + 1) {   // column k + 1
#pragma unroll
          for (int j = 0; j < 4; j++) *reinterpret_cast<double2*>(&rd.a1[32 * j + 2 * u]) = make_double2(a[i][2 * j], a[i][2 * j + 1]);
        }
    } else if (lane == 0) {
      rd.part[warp] = 0.0;
    }
    __syncthreads();
    if (tid < D) {
      const double gamma = rd.gamma, tau = rd.tau;
      double q[4];
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const double2 f = *reinterpret_cast<const double2*>(&rd.part[2 * i]);
        q[i] = f.x + f.y;
      }
      const double xy = (q[0] + q[1]) + (q[2] + q[3]), a11 = rd.a1[k + 1], y1 = rd.y[k + 1], a1 = rd.a1[tid];
      const double vav = fma(gamma, fma(gamma, a11, 2.0 * y1), xy);
      const double half = 0.5 * tau * tau * vav;
      const double v = tid == k + 1 ? gamma : rd.x[tid];
      const double w = tid > k ? fma(tau, fma(gamma, a1, rd.y[tid]), -half * v) : 0.0;
      const double w1 = fma(tau, fma(gamma, a11, y1), -half * gamma);
      const double next = fma(-gamma, w, fma(-w1, v, a1));   // column k + 1 after the update
      rd.v[tid] = v;
      rd.w[tid] = w;
      rd.x[tid] = tid > k + 2 ? next : 0.0;
      if (tid == k + 2) rd.alpha = next;
      if (tid == k + 1) sm.d[k + 1] = next;
      if (tid > k) *to = v;
      to += step;
      if (k == D / 2 - 1) { to = rows + (D / 2 - 2) * D + D - 1 - tid; step = -D; }
    }
    __syncthreads();
  }
  // what is left: the last diagonal element and the one beside it
  if (tid == THREADS - 1) sm.d[D - 1] = fma(-2.0 * rd.v[D - 1], rd.w[D - 1], a[7][7]);
  if (tid == 0) { sm.e[D - 2] = rd.alpha; sm.e[D - 1] = 0.0; sm.tau[D - 2] = 0.0; sm.tau[D - 1] = 0.0; }
  if (tid == 0) rows[0] = 0.0;   // the last one, which reflects nothing
}

// Eigenvalues below x[n] of the rows lo .. hi of the tridiagonal matrix: sign changes of the sequence of leading minors,
// p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2}, brought back near one every eight terms.  (As accurate as the sequence of
// quotients, whose division would be a chain of about 100 cycles per row.)  Two points of different eigenvalues share the
// loads: shared memory's 128 bytes a cycle bounded it with one point per lane.
template <int N>
__device__ __forceinline__ void sturm_count(const double2* de, int lo, int hi, const double (&x)[N], int (&cnt)[N]) {
  double p[N], q[N];
  int i = lo;
#pragma unroll
  for (int n = 0; n < N; n++) { p[n] = 1.0; q[n] = 0.0; cnt[n] = 0; }
  auto term = [&](const double2 c) {
#pragma unroll
    for (int n = 0; n < N; n++) {
      const double t = fma(c.x - x[n], p[n], -c.y * q[n]);
      cnt[n] += (unsigned)(__double2hiint(t) ^ __double2hiint(p[n])) >> 31;
      q[n] = p[n];
      p[n] = t;
    }
  };
  for (; i + 8 <= hi + 1; i += 8) {
    double2 c[8];
#pragma unroll
    for (int j = 0; j < 8; j++) c[j] = de[i + j];
#pragma unroll
    for (int j = 0; j < 8; j++) term(c[j]);
#pragma unroll
    for (int n = 0; n < N; n++) rescale(p[n], q[n]);
  }
  for (; i <= hi; i++) term(de[i]);
}

__global__ void __launch_bounds__(THREADS, 1) k_calib_spectrum(const float* __restrict__ C, const float* __restrict__ signs, float* __restrict__ R,
                                                              float* __restrict__ lambda, int* __restrict__ sweeps_out) {
  extern __shared__ __align__(16) unsigned char raw[];
  Smem& sm = *reinterpret_cast<Smem*>(raw);
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = blockIdx.x;
  double* const rows = reinterpret_cast<double*>(R);   // exchanged between the blocks until R is written
  depend_wait();
  {
    float least = INFINITY, most = 0.f;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const float x = fabsf(C[(lane + 32 * q) * (D + 1)]);
      least = fminf(least, x);
      most = fmaxf(most, x);
    }
#pragma unroll
    for (int s = 16; s; s >>= 1) {
      least = fminf(least, __shfl_xor_sync(0xffffffffu, least, s));
      most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, s));
    }
    if (least < GRADED * most) {   // (the same in every warp of every block)
      if (rank == 0 && tid == 0) lambda[0] = __uint_as_float(EIGEN_LEFT);
      return;
    }
  }
  if (rank == 0) {
    reduce_to_tridiagonal(sm, C, rows);
    __threadfence();
  }
  cluster.sync();   // the tridiagonal matrix and the reflectors are there
  if (rank != 0) {
    Smem* s0 = cluster.map_shared_rank(&sm, 0);
    if (tid < D) { sm.d[tid] = s0->d[tid]; sm.e[tid] = s0->e[tid]; sm.tau[tid] = s0->tau[tid]; }
    if (tid == 0) sm.expo = s0->expo;
  }
  auto pairs = [&](auto f) {   // of the reflectors' 64 rows, the same ones of a thread each time
    for (int i = tid; i < D / 2 * D / 2; i += THREADS) f(i / (D / 2), 2 * (i % (D / 2)));
  };
  pairs([&](int r, int c) {
    copy_async16(&sm.refl[r][c], rows + r * D + c);
    *reinterpret_cast<double2*>(&sm.refl[D / 2 + r][c]) = make_double2(0.0, 0.0);
  });
  asm volatile("cp.async.commit_group;\n" ::);
  __syncthreads();

  // ---- sizes, blocks: an off-diagonal element at rounding level of the matrix is none
  double tn = 0.0, gl = 1e300, gu = -1e300;
  unsigned long long cut_lo, cut_hi;   // bit i: the matrix falls apart between i and i + 1
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const int i = lane + 32 * q;
    const double d = sm.d[i], rad = (i > 0 ? fabs(sm.e[i - 1]) : 0.0) + fabs(sm.e[i]);
    tn = fmax(tn, fabs(d) + rad);
    gl = fmin(gl, d - rad);
    gu = fmax(gu, d + rad);
  }
#pragma unroll
  for (int s = 16; s; s >>= 1) {
    tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, s));
    gl = fmin(gl, __shfl_xor_sync(0xffffffffu, gl, s));
    gu = fmax(gu, __shfl_xor_sync(0xffffffffu, gu, s));
  }
  {
    unsigned m[4];
#pragma unroll
    for (int q = 0; q < 4; q++) m[q] = __ballot_sync(0xffffffffu, fabs(sm.e[lane + 32 * q]) <= EPS * tn);
    cut_lo = m[0] | (unsigned long long)m[1] << 32;
    cut_hi = m[2] | (unsigned long long)m[3] << 32;   // (the last bit is always set)
  }
  // eigenvalues go by position: the one of position p is number p - lo of the block p is in; a warp has two
  auto block_of = [&](int p, int& lo, int& hi) {
    const unsigned long long above_lo = p < 64 ? cut_lo >> p << p : 0ull, above_hi = p < 64 ? cut_hi : cut_hi >> (p - 64) << (p - 64);
    hi = above_lo ? __ffsll((long long)above_lo) - 1 : (above_hi ? 63 + __ffsll((long long)above_hi) : D - 1);
    const unsigned long long below_lo = p >= 64 ? cut_lo : cut_lo & ((1ull << p) - 1), below_hi = p > 64 ? cut_hi & ((1ull << (p - 64)) - 1) : 0ull;
    lo = below_hi ? 128 - __clzll((long long)below_hi) : (below_lo ? 64 - __clzll((long long)below_lo) : 0);
  };
  if (tid < D) sm.de[tid] = make_double2(sm.d[tid], tid > 0 ? sm.e[tid - 1] * sm.e[tid - 1] : 0.0);
  __syncthreads();

  // ---- eigenvalues: 32 inner points of the interval per round, a factor 33; eleven rounds reach rounding level
  const int j0 = rank * VEC + 2 * warp;
  int lo[2], hi[2];
  double lam[2];
  {
    double a[2], b[2];
#pragma unroll
    for (int n = 0; n < 2; n++) {
      block_of(j0 + n, lo[n], hi[n]);
      a[n] = gl - 4 * EPS * tn;
      b[n] = gu + 4 * EPS * tn;
    }
#pragma unroll 1
    for (int it = 0; it < 12; it++) {
      double h[2], x[2];
      int cnt[2];
#pragma unroll
      for (int n = 0; n < 2; n++) {
        h[n] = (b[n] - a[n]) * (1.0 / 33.0);
        x[n] = fma(h[n], (double)(lane + 1), a[n]);
      }
      if (!(fmax(b[0] - a[0], b[1] - a[1]) > EPS * tn)) break;
      if (lo[0] == lo[1]) {
        sturm_count<2>(sm.de, lo[0], hi[0], x, cnt);
      } else {
#pragma unroll
        for (int n = 0; n < 2; n++) {
          const double x1[1] = {x[n]};
          int c1[1];
          sturm_count<1>(sm.de, lo[n], hi[n], x1, c1);
          cnt[n] = c1[0];
        }
      }
#pragma unroll
      for (int n = 0; n < 2; n++) {
        const unsigned above = __ballot_sync(0xffffffffu, cnt[n] > j0 + n - lo[n]);
        const int first = above ? __ffs(above) - 1 : 32;
        const double a0 = a[n];
        if (first > 0) a[n] = fma(h[n], (double)first, a0);
        if (first < 32) b[n] = fma(h[n], (double)(first + 1), a0);
      }
    }
#pragma unroll
    for (int n = 0; n < 2; n++) lam[n] = hi[n] > lo[n] ? 0.5 * (a[n] + b[n]) : sm.d[j0 + n];
  }
  // ---- eigenvectors: the sequences of leading minors (lanes 0, 2 for the warp's two) and of trailing ones (lanes 1, 3) are the
  // pivots of the two factorisations as quotients of neighbours
  {
    const int back = lane & 1, n = (lane >> 1) & 1, l = n ? lo[1] : lo[0], h = n ? hi[1] : hi[0], m = h - l + 1;
    const int step = back ? -1 : 1, i0 = back ? h : l;
    const double x = n ? lam[1] : lam[0];
    double2* seq = sm.seq[2 * warp + n][back];
    double p = 1.0, q = 0.0;
    // the element before row i on the way: e_{i-1}^2 going forward, e_i^2 = de[i + 1].y going back (none at the first row)
    for (int s = 0; s < max(hi[0] - lo[0], hi[1] - lo[1]) + 1; s += 8) {
      double dd[8], ee[8];
#pragma unroll
      for (int v = 0; v < 8; v++) {
        const int i = min(max(i0 + step * (s + v), l), h);
        dd[v] = sm.de[i].x - x;
        ee[v] = sm.de[min(i + back, D - 1)].y;
      }
      if (s == 0) ee[0] = 0.0;
#pragma unroll
      for (int v = 0; v < 8; v++) {
        double t = fma(dd[v], p, -ee[v] * q);
        if (t == 0.0) t = 1e-60 * p;
        if (lane < 4 && s + v < m) seq[i0 + step * (s + v)] = make_double2(t, p);
        q = p;
        p = t;
      }
      rescale(p, q);
    }
  }
  __syncwarp();
  bool resid_ok = true;
  int at2[2];
  double best2[2];
#pragma unroll
  for (int n = 0; n < 2; n++) {
    // the residual of the vector that is 1 at i: the sum of the two pivots there less the diagonal element
    const double2 (*seq)[D] = sm.seq[2 * warp + n];
    double best = INFINITY;
    int at = lo[n];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int i = lane + 32 * q;
      if (i >= lo[n] && i <= hi[n]) {
        const double2 f = seq[0][i], g = seq[1][i];
        const double gam = f.x / f.y + (g.x / g.y - (sm.d[i] - lam[n]));
        if (fabs(gam) < fabs(best)) { best = gam; at = i; }
      }
    }
#pragma unroll
    for (int s = 16; s; s >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, s);
      const int oa = __shfl_xor_sync(0xffffffffu, at, s);
      if (fabs(ob) < fabs(best) || (fabs(ob) == fabs(best) && oa < at)) { best = ob; at = oa; }
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {   // quotient of each component and its neighbour on the side of `at`
      const int i = lane + 32 * q;
      double f = 0.0;
      if (i >= lo[n] && i < at) f = -sm.e[i] * seq[0][i].y / seq[0][i].x;
      else if (i > at && i <= hi[n]) f = -sm.e[i - 1] * seq[1][i].y / seq[1][i].x;
      else if (i == at) f = 1.0;
      sm.own[2 * warp + n][i] = f;
    }
    at2[n] = at;
    best2[n] = best;
  }
  __syncwarp();
  if (lane < 4) {
    const int n = lane >> 1, at = n ? at2[1] : at2[0], step = (lane & 1) ? 1 : -1;
    const int len = (lane & 1) ? (n ? hi[1] : hi[0]) - at : at - (n ? lo[1] : lo[0]);
    double* z = sm.own[2 * warp + n];
    double c = 1.0;
    for (int s = 0; s < len; s += 8) {
      double f[8];
#pragma unroll
      for (int v = 0; v < 8; v++) f[v] = s + v < len ? z[at + step * (s + v + 1)] : 0.0;
#pragma unroll
      for (int v = 0; v < 8; v++)
        if (s + v < len) { c *= f[v]; z[at + step * (s + v + 1)] = c; }
    }
  }
  __syncwarp();
#pragma unroll
  for (int n = 0; n < 2; n++) {
    double* z = sm.own[2 * warp + n];
    double zz[4], s2 = 0.0;
#pragma unroll
    for (int q = 0; q < 4; q++) { zz[q] = z[lane + 32 * q]; s2 = fma(zz[q], zz[q], s2); }
    const double inv = 1.0 / sqrt(warp_sum(s2));
#pragma unroll
    for (int q = 0; q < 4; q++) z[lane + 32 * q] = zz[q] * inv;
    if (hi[n] > lo[n]) {
      lam[n] = fma(best2[n] * inv, inv, lam[n]);
      resid_ok = resid_ok && fabs(best2[n]) * inv <= RESIDUAL_TOL * EPS * tn;   // (false for NaN)
    }
    resid_ok = resid_ok && isfinite(lam[n]);
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  pairs([&](int r, int c) {   // the reversed ones go to rows of their own
    if (c > r) return;
    const double2 x = *reinterpret_cast<const double2*>(&sm.refl[r][c]);
    *reinterpret_cast<double2*>(&sm.refl[r][c]) = make_double2(0.0, c == r ? x.y : 0.0);
    if (r < D / 2 - 1) *reinterpret_cast<double2*>(&sm.refl[126 - r][126 - c]) = make_double2(c == r ? 0.0 : x.y, x.x);
  });
  const int bad = __syncthreads_or(!resid_ok);   // (the vectors and the reflectors are in place)

  // ---- V = H_0 H_1 ... H_125 Z: reflectors in groups of four, last ones first, their products with the vector taken together
  for (int i = warp; i < (D / 4) * 6; i += WARPS) {
    const int grp = i / 6, pr = i % 6, x = pr < 3 ? 0 : (pr < 5 ? 1 : 2), y = pr < 3 ? pr + 1 : (pr < 5 ? pr - 1 : 3);
    const double* vx = sm.refl[4 * grp + 3 - x];
    const double* vy = sm.refl[4 * grp + 3 - y];
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < 4; q++) s = fma(vx[lane + 32 * q], vy[lane + 32 * q], s);
    s = warp_sum(s);
    if (lane == 0) sm.wy.cross[grp][pr] = s;   // (0,1) (0,2) (0,3) (1,2) (1,3) (2,3), counted from the group's last
  }
  __syncthreads();
  if (warp < VEC / 4) {   // half a warp takes two vectors: each number of a reflector is loaded once for both, and kept
    const int u = lane & 15, vec = 4 * warp + 2 * (lane >> 4);
    double zr[2][8];
#pragma unroll
    for (int n = 0; n < 2; n++)
#pragma unroll
      for (int m = 0; m < 4; m++) {
        const double2 t = *reinterpret_cast<const double2*>(&sm.own[vec + n][32 * m + 2 * u]);
        zr[n][2 * m] = t.x; zr[n][2 * m + 1] = t.y;
      }
#pragma unroll 1
    for (int grp = D / 4 - 1; grp >= 0; grp--) {
      double dot[2][4];
      double2 v[4][4];
#pragma unroll
      for (int x = 0; x < 4; x++)
#pragma unroll
        for (int m = 0; m < 4; m++) v[x][m] = *reinterpret_cast<const double2*>(&sm.refl[4 * grp + 3 - x][32 * m + 2 * u]);
#pragma unroll
      for (int x = 0; x < 4; x++)
#pragma unroll
        for (int n = 0; n < 2; n++) {
          double s0 = v[x][0].x * zr[n][0], s1 = v[x][0].y * zr[n][1];
#pragma unroll
          for (int m = 1; m < 4; m++) {
            s0 = fma(v[x][m].x, zr[n][2 * m], s0);
            s1 = fma(v[x][m].y, zr[n][2 * m + 1], s1);
          }
          dot[n][x] = s0 + s1;
        }
#pragma unroll
      for (int s = 1; s < 16; s <<= 1)
#pragma unroll
        for (int x = 0; x < 4; x++)
#pragma unroll
          for (int n = 0; n < 2; n++) dot[n][x] += __shfl_xor_sync(0xffffffffu, dot[n][x], s);
      const double* x6 = sm.wy.cross[grp];
      const double* tau = &sm.tau[4 * grp];
#pragma unroll
      for (int n = 0; n < 2; n++) {
        double c[4];
        c[0] = tau[3] * dot[n][0];
        c[1] = tau[2] * fma(-x6[0], c[0], dot[n][1]);
        c[2] = tau[1] * fma(-x6[3], c[1], fma(-x6[1], c[0], dot[n][2]));
        c[3] = tau[0] * fma(-x6[5], c[2], fma(-x6[4], c[1], fma(-x6[2], c[0], dot[n][3])));
#pragma unroll
        for (int x = 0; x < 4; x++)
#pragma unroll
          for (int m = 0; m < 4; m++) {
            zr[n][2 * m] = fma(-c[x], v[x][m].x, zr[n][2 * m]);
            zr[n][2 * m + 1] = fma(-c[x], v[x][m].y, zr[n][2 * m + 1]);
          }
      }
    }
#pragma unroll
    for (int n = 0; n < 2; n++)
#pragma unroll
      for (int m = 0; m < 4; m++)
        *reinterpret_cast<double2*>(&sm.own[vec + n][32 * m + 2 * u]) = make_double2(zr[n][2 * m], zr[n][2 * m + 1]);
  }
  if (lane < CTAS) {
    double* l = cluster.map_shared_rank(&sm.lam[0], lane);
    l[j0] = lam[0];
    l[j0 + 1] = lam[1];
  }

  // ---- Newton-Schulz: this block's rows of V^T V, then of V
  int steps = 0;
  bool good = false;
#pragma unroll 1
  for (; steps < MAX_STEPS;) {
    // half of the columns through R, whose reflectors every block has copied, half straight into the other blocks' shared memory
    cluster.sync();   // (nobody reads the reflectors, or the vectors of the step before, any more)
    for (int i = tid; i < VEC * D / 4; i += THREADS) {
      const int row = i / (D / 4), c = 2 * (i % (D / 4));
      const double2 x = *reinterpret_cast<const double2*>(&sm.own[row][D / 2 + c]);
#pragma unroll
      for (int r = 0; r < CTAS; r++) *reinterpret_cast<double2*>(cluster.map_shared_rank(&sm.all[rank * VEC + row][D / 2 + c], r)) = x;
      __stcg(reinterpret_cast<double2*>(rows + (rank * VEC + row) * (D / 2) + c), *reinterpret_cast<const double2*>(&sm.own[row][c]));
    }
    __threadfence();
    cluster.sync();   // every block's vectors are there
    for (int i = tid; i < D * D / 4; i += THREADS) {
      const int row = i / (D / 4), c = 2 * (i % (D / 4));
      copy_async16(&sm.all[row][c], rows + row * (D / 2) + c);
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    const int g = lane >> 2, t = lane & 3, r0 = 8 * (warp & 1), c0 = 8 * (warp >> 1);
    double dist = 0.0;
    {
      double acc[4][2] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
#pragma unroll 8
      for (int s = 0; s < D; s += 4) {
        const double x = sm.own[r0 + g][s + t];
#pragma unroll
        for (int h = 0; h < 4; h++) dmma(acc[h], x, sm.all[32 * h + c0 + g][s + t]);
      }
#pragma unroll
      for (int h = 0; h < 4; h++)
#pragma unroll
        for (int e = 0; e < 2; e++) {
          const int col = 32 * h + c0 + 2 * t + e;
          sm.ns.g[r0 + g][col] = acc[h][e];
          const double o = acc[h][e] - (col == rank * VEC + r0 + g ? 1.0 : 0.0);
          dist = fma(o, o, dist);
        }
    }
    dist = warp_sum(dist);
    if (lane == 0) sm.redw[warp] = dist;
    __syncthreads();
    if (tid < CTAS) {
      double s = bad ? NAN : 0.0;
      for (int i = 0; i < WARPS; i++) s += sm.redw[i];
      cluster.map_shared_rank(&sm.err[0], tid)[rank] = s;
    }
    cluster.sync();   // every block has read everyone's vectors; the distances are there
    double err = 0.0;
    for (int i = 0; i < CTAS; i++) err += sm.err[i];
    if (!(err < 0.25)) break;
    steps++;
    {
      double acc[4][2] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
#pragma unroll 8
      for (int s = 0; s < D; s += 4) {
        const double x = sm.ns.g[r0 + g][s + t];
#pragma unroll
        for (int h = 0; h < 4; h++) dmma(acc[h], x, sm.all[s + t][32 * h + c0 + g]);
      }
#pragma unroll
      for (int h = 0; h < 4; h++)
#pragma unroll
        for (int e = 0; e < 2; e++) {
          double* o = &sm.own[r0 + g][32 * h + c0 + 2 * t + e];
          *o = fma(-0.5, acc[h][e], 1.5 * *o);
        }
    }
    __syncthreads();
    if (err < 1e-16) { good = true; break; }   // the step just made leaves 3/4 of that, the squared distance
  }
  if (rank == 0 && tid == 0) {
    if (!good) lambda[0] = __uint_as_float(EIGEN_LEFT);
    else if (sweeps_out) *sweeps_out = steps;
  }
  if (!good) return;   // (the same for every block, none of which reads another's memory any more)

  // ---- every vector's component of largest magnitude positive (the first of equals); descending order, ties by position
#pragma unroll
  for (int n = 0; n < 2; n++) {
    double* z = sm.own[2 * warp + n];
    double best = 0.0, val = 1.0;
    int at = D;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const double x = z[lane + 32 * q];
      if (fabs(x) > best) { best = fabs(x); val = x; at = lane + 32 * q; }
    }
#pragma unroll
    for (int s = 16; s; s >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, s), ov = __shfl_xor_sync(0xffffffffu, val, s);
      const int oa = __shfl_xor_sync(0xffffffffu, at, s);
      if (ob > best || (ob == best && oa < at)) { best = ob; val = ov; at = oa; }
    }
    if (val < 0.0)
#pragma unroll
      for (int q = 0; q < 4; q++) z[lane + 32 * q] = -z[lane + 32 * q];
  }
  {
    const int i = tid >> 1, q = tid & 1;
    const double l = sm.lam[i];
    int pos = 0;
#pragma unroll 8
    for (int o = q; o < D; o += 2) pos += sm.lam[o] > l || (sm.lam[o] == l && o < i);
    pos += __shfl_xor_sync(0xffffffffu, pos, 1);
    if (q == 0) {
      sm.order[pos] = i;
      if (rank == 0) lambda[pos] = (float)ldexp(l, sm.expo);
    }
  }
  cluster.sync();   // signs are in place everywhere
  {  // R[c][k] = sum_l H[c][l] U[k][l]: two columns k per warp, lane holds l = lane + 32 i; a Hadamard transform per column
    double x[2][4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const int l = lane + 32 * i, src = sm.order[l];
      const double sg = (double)signs[l];
      const double2 v = *reinterpret_cast<const double2*>(cluster.map_shared_rank(&sm.own[0][0], src / VEC) + (src % VEC) * PITCH + j0);
      x[0][i] = sg * v.x;
      x[1][i] = sg * v.y;
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
#pragma unroll
      for (int n = 0; n < 2; n++)
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const double o = __shfl_xor_sync(0xffffffffu, x[n][i], d);
          x[n][i] = (lane & d) ? o - x[n][i] : x[n][i] + o;
        }
#pragma unroll
    for (int n = 0; n < 2; n++) {
      const double y0 = x[n][0] + x[n][1], y1 = x[n][0] - x[n][1], y2 = x[n][2] + x[n][3], y3 = x[n][2] - x[n][3];
      x[n][0] = y0 + y2; x[n][1] = y1 + y3; x[n][2] = y0 - y2; x[n][3] = y1 - y3;
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
      *reinterpret_cast<float2*>(R + (size_t)(lane + 32 * i) * D + j0) =
          make_float2((float)(x[0][i] * 0.08838834764831845), (float)(x[1][i] * 0.08838834764831845));   // 1 / sqrt(128)
  }
  cluster.sync();   // nobody's vectors are read any more
}

}  // namespace

cudaError_t launch_calib_spectrum(const float* C, const float* signs, float* R, float* lambda, int* sweeps, cudaStream_t s) {
  static thread_local unsigned long long attr_mask = 0;
  int dev = 0;
  if (attr_needed(attr_mask, dev)) {
    const cudaError_t e = cudaFuncSetAttribute(k_calib_spectrum, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
    if (e != cudaSuccess) return e;
    attr_done(attr_mask, dev);
  }
  return launch_dependent(k_calib_spectrum, dim3(CTAS), THREADS, sizeof(Smem), s, CTAS, C, signs, R, lambda, sweeps);
}

}  // namespace okq
