// Direct eigensolver of the calibration: one symmetric 128 x 128 matrix by one cluster of eight blocks, all in fp64.
//
//   1. Householder reduction to a tridiagonal matrix (block 0, the matrix in registers); the reflectors go to the workspace
//   2. eigenvalues by 33-section on Sturm counts, a warp per eigenvalue, 16 eigenvalues per block
//   3. eigenvectors of the tridiagonal matrix from its two factorisations, twisted where the residual is least
//   4. the reflectors applied to them, a quarter of a warp per vector
//   5. Newton-Schulz steps V <- V (3 I - V^T V) / 2 on the fp64 tensor cores: vectors of close eigenvalues, orthogonal only to
//      (rounding / gap) after step 3, become orthogonal to fp64
//   6. descending order, signs, R = H U^T
//
// Every vector's residual is known from step 3, and orthonormal vectors with small residuals are a complete eigenbasis: if a
// residual is not at rounding level, or V^T V is too far from the identity for step 5 (equal eigenvalues of one tridiagonal
// block; exhausted reductions - zero, diagonal, low-rank matrices - fall apart into blocks and are no such case), the call is
// left to the Jacobi solver, which needs no gaps: it runs behind this kernel and returns at once when there is nothing to do.
//
// Why: cyclic Jacobi is 11 to 13 sweeps of 127 dependent rounds of about a microsecond, whatever the number of SMs; the
// reduction is 126 dependent steps of half a microsecond, once, and everything behind it is parallel over the vectors.
#include <cooperative_groups.h>

#include "okq_common.cuh"
#include "okq_eigen.cuh"

namespace cg = cooperative_groups;

namespace okq {
namespace {

constexpr int CTAS = 8, THREADS = 512, WARPS = THREADS / 32;
constexpr int VEC = D / CTAS;               // eigenvectors of a block
constexpr int PITCH = D + 4;                // doubles per row: the fragment reads of a half-warp fall on all 32 banks
static_assert(VEC == WARPS, "a warp per eigenvalue");

constexpr double EPS = 0x1p-53;
constexpr double RESIDUAL_TOL = 512.0;      // in EPS times the matrix's size
constexpr int MAX_STEPS = 8;                // Newton-Schulz steps: 0.5 -> 0.19 -> 0.03 -> 5e-4 -> 2e-7 -> 3e-14, and one to spare

struct Smem {
  union {
    double refl[D][D];                      // reflectors (copies)
    double all[D][PITCH];                   // all eigenvectors (rows), gathered from the blocks
  };
  __align__(16) double own[VEC][PITCH];     // this block's eigenvectors
  union {
    struct {                                // reduction (block 0)
      __align__(16) double x[D], y[D], a1[D];   // tail of the column, matrix times it, next column
      __align__(16) double2 vw[D];          // reflector, update vector
      double part[WARPS];
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

// Step 1.  Thread (row r = tid / 4, u = tid % 4) holds the columns 8 j + 2 u + {0, 1} of its row.  Step k: with the tail x of
// column k below its first element alpha, the reflector is v = x + gamma e_{k+1}, gamma = alpha + sign(alpha) |column|,
// tau = 2 / v^T v, and the rest of the matrix becomes A - v w^T - w v^T, w = tau A v - (tau^2 / 2)(v^T A v) v.  A v comes from
// y = A x and the next column, so the product can start before the norm is known; warp 0, whose rows are done first, works out
// the scalars meanwhile.  Three block barriers per step; bound by their chain (product, two sums over lanes, w, update).
__device__ void reduce_to_tridiagonal(Smem& sm, const float* __restrict__ C, double (*__restrict__ refl)[D]) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, r = tid >> 2, u = tid & 3;
  auto& rd = sm.red;
  double a[32];
  float mx = 0.f;
#pragma unroll
  for (int j = 0; j < 16; j++) {
    const float2 c = *reinterpret_cast<const float2*>(C + r * D + 8 * j + 2 * u);
    const float t0 = C[(8 * j + 2 * u) * D + r], t1 = C[(8 * j + 2 * u + 1) * D + r];
    mx = fmaxf(mx, fmaxf(fabsf(c.x), fabsf(c.y)));
    a[2 * j] = 0.5 * ((double)c.x + (double)t0);
    a[2 * j + 1] = 0.5 * ((double)c.y + (double)t1);
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
  for (int i = 0; i < 32; i++) a[i] *= scale;

  // row k of the matrix = its column k: the tail beyond column k + 1, the element there
  auto publish = [&](int k) {
    if (r != k) return;
#pragma unroll
    for (int j = 0; j < 16; j++) {
      const int c = 8 * j + 2 * u;
      *reinterpret_cast<double2*>(&rd.x[c]) = make_double2(c > k + 1 ? a[2 * j] : 0.0, c + 1 > k + 1 ? a[2 * j + 1] : 0.0);
      if (c == k + 1) rd.alpha = a[2 * j];
      if (c + 1 == k + 1) rd.alpha = a[2 * j + 1];
      if (c == k) sm.d[k] = a[2 * j];
      if (c + 1 == k) sm.d[k] = a[2 * j + 1];
    }
  };
  publish(0);
  __syncthreads();
#pragma unroll 1
  for (int k = 0; k < D - 2; k++) {
    if (warp == 0) {
      const double2 x0 = *reinterpret_cast<const double2*>(&rd.x[4 * lane]), x1 = *reinterpret_cast<const double2*>(&rd.x[4 * lane + 2]);
      const double s2 = warp_sum((x0.x * x0.x + x0.y * x0.y) + (x1.x * x1.x + x1.y * x1.y));
      const double al = rd.alpha;
      double beta = al, gamma = 0.0, tau = 0.0;   // nothing to reflect
      if (s2 > 1e-280) {
        const double nrm = sqrt(fma(al, al, s2));
        beta = al > 0.0 ? -nrm : nrm;
        gamma = al - beta;
        tau = 2.0 / fma(gamma, gamma, s2);
      }
      if (lane == 0) { rd.gamma = gamma; rd.tau = tau; sm.e[k] = beta; sm.tau[k] = tau; }
    }
    // (whole warps: rows up to 8 (k / 8) + 7 may include finished ones, whose results are zeroed)
    double y = 0.0;
    if (8 * warp + 7 > k) {
      double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int j = 0; j < 16; j++)
        if (8 * j + 7 > k) {
          const double2 x = *reinterpret_cast<const double2*>(&rd.x[8 * j + 2 * u]);
          s[2 * (j & 1)] = fma(a[2 * j], x.x, s[2 * (j & 1)]);
          s[2 * (j & 1) + 1] = fma(a[2 * j + 1], x.y, s[2 * (j & 1) + 1]);
        }
      y = (s[0] + s[1]) + (s[2] + s[3]);
      y += __shfl_xor_sync(0xffffffffu, y, 1);
      y += __shfl_xor_sync(0xffffffffu, y, 2);
      if (r <= k) y = 0.0;
      if (u == 0) rd.y[r] = y;
      double p = rd.x[r] * y;
      p += __shfl_xor_sync(0xffffffffu, p, 4);
      p += __shfl_xor_sync(0xffffffffu, p, 8);
      p += __shfl_xor_sync(0xffffffffu, p, 16);
      if (lane == 0) rd.part[warp] = p;
      if (r == k + 1) {
#pragma unroll
        for (int j = 0; j < 16; j++) *reinterpret_cast<double2*>(&rd.a1[8 * j + 2 * u]) = make_double2(a[2 * j], a[2 * j + 1]);
      }
    } else {
      if (u == 0) rd.y[r] = 0.0;
      if (lane == 0) rd.part[warp] = 0.0;
    }
    __syncthreads();
    if (tid < D) {
      const double gamma = rd.gamma, tau = rd.tau;
      double xy = 0.0;
      {
        double q[4];
#pragma unroll
        for (int i = 0; i < 4; i++) q[i] = (rd.part[4 * i] + rd.part[4 * i + 1]) + (rd.part[4 * i + 2] + rd.part[4 * i + 3]);
        xy = (q[0] + q[1]) + (q[2] + q[3]);
      }
      const double vav = fma(gamma, fma(gamma, rd.a1[k + 1], 2.0 * rd.y[k + 1]), xy);
      const double half = 0.5 * tau * tau * vav;
      const double v = tid == k + 1 ? gamma : rd.x[tid];
      const double w = tid > k ? fma(tau, fma(gamma, rd.a1[tid], rd.y[tid]), -half * v) : 0.0;
      rd.vw[tid] = make_double2(v, w);
      refl[k][tid] = v;
    }
    __syncthreads();
    if (8 * warp + 7 > k) {
      const double2 m = rd.vw[r];
#pragma unroll
      for (int j = 0; j < 16; j++)
        if (8 * j + 7 > k) {
#pragma unroll
          for (int i = 0; i < 2; i++) {
            const double2 c = rd.vw[8 * j + 2 * u + i];
            a[2 * j + i] = fma(-m.x, c.y, fma(-m.y, c.x, a[2 * j + i]));
          }
        }
      publish(k + 1);
    }
    __syncthreads();
  }
  // what is left: the last two diagonal elements and the one between them
  if (r == D - 1 && u == 3) sm.d[D - 1] = a[31];
  if (tid == 0) { sm.e[D - 2] = rd.alpha; sm.e[D - 1] = 0.0; sm.tau[D - 2] = 0.0; sm.tau[D - 1] = 0.0; }
  if (tid < D) { refl[D - 2][tid] = 0.0; }
}

// Eigenvalues below x of the rows lo .. hi of the tridiagonal matrix: sign changes of the sequence of leading minors,
// p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2}, brought back near one every eight terms.  (As accurate as the sequence of
// quotients, whose division would be a chain of about 100 cycles per row.)
__device__ __forceinline__ int sturm_count(const double2* de, int lo, int hi, double x) {
  double p = 1.0, q = 0.0;
  int n = 0, i = lo;
  auto term = [&](const double2 c) {
    const double t = fma(c.x - x, p, -c.y * q);
    n += (unsigned)(__double2hiint(t) ^ __double2hiint(p)) >> 31;
    q = p;
    p = t;
  };
  for (; i + 8 <= hi + 1; i += 8) {
    double2 c[8];
#pragma unroll
    for (int j = 0; j < 8; j++) c[j] = de[i + j];
#pragma unroll
    for (int j = 0; j < 8; j++) term(c[j]);
    rescale(p, q);
  }
  for (; i <= hi; i++) term(de[i]);
  return n;
}

__global__ void __launch_bounds__(THREADS, 1) k_calib_spectrum(const float* __restrict__ C, const float* __restrict__ signs, double* __restrict__ ws,
                                                              float* __restrict__ R, float* __restrict__ lambda, int* __restrict__ sweeps_out) {
  extern __shared__ __align__(16) unsigned char raw[];
  Smem& sm = *reinterpret_cast<Smem*>(raw);
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = blockIdx.x;
  double (*refl)[D] = reinterpret_cast<double (*)[D]>(ws);
  depend_wait();
  if (rank == 0) {
    reduce_to_tridiagonal(sm, C, refl);
    __threadfence();
  }
  cluster.sync();   // the tridiagonal matrix and the reflectors are there
  if (rank != 0) {
    Smem* s0 = cluster.map_shared_rank(&sm, 0);
    if (tid < D) { sm.d[tid] = s0->d[tid]; sm.e[tid] = s0->e[tid]; sm.tau[tid] = s0->tau[tid]; }
    if (tid == 0) sm.expo = s0->expo;
  }
  for (int i = tid; i < (D - 1) * D / 2; i += THREADS) copy_async16(&sm.refl[0][2 * i], &refl[0][2 * i]);
  asm volatile("cp.async.commit_group;\n" ::);
  if (tid < D) sm.refl[D - 1][tid] = 0.0;
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
  const int j = rank * VEC + warp;     // this warp's eigenvalue: by position, that is number j - lo of the block that position is in
  int lo, hi;
  {
    const unsigned long long above_lo = j < 64 ? cut_lo >> j << j : 0ull, above_hi = j < 64 ? cut_hi : cut_hi >> (j - 64) << (j - 64);
    hi = above_lo ? __ffsll((long long)above_lo) - 1 : (above_hi ? 63 + __ffsll((long long)above_hi) : D - 1);
    const unsigned long long below_lo = j >= 64 ? cut_lo : cut_lo & ((1ull << j) - 1), below_hi = j > 64 ? cut_hi & ((1ull << (j - 64)) - 1) : 0ull;
    lo = below_hi ? 128 - __clzll((long long)below_hi) : (below_lo ? 64 - __clzll((long long)below_lo) : 0);
  }
  if (tid < D) sm.de[tid] = make_double2(sm.d[tid], tid > 0 ? sm.e[tid - 1] * sm.e[tid - 1] : 0.0);
  __syncthreads();

  // ---- eigenvalue: 32 inner points of the interval per round, a factor 33; eleven rounds reach rounding level
  double lam = sm.d[j];
  double resid = 0.0;
  double* z = sm.own[warp];
  if (hi > lo) {
    double a = gl - 4 * EPS * tn, b = gu + 4 * EPS * tn;
#pragma unroll 1
    for (int it = 0; it < 12 && b - a > EPS * tn; it++) {
      const double h = (b - a) * (1.0 / 33.0);
      const int n = sturm_count(sm.de, lo, hi, fma(h, (double)(lane + 1), a));
      const unsigned above = __ballot_sync(0xffffffffu, n > j - lo);
      const int first = above ? __ffs(above) - 1 : 32;
      const double a0 = a;
      if (first > 0) a = fma(h, (double)first, a0);
      if (first < 32) b = fma(h, (double)(first + 1), a0);
    }
    lam = 0.5 * (a + b);
    // ---- eigenvector: the sequences of leading minors (even lanes) and of trailing ones (odd lanes) are the pivots of the two
    // factorisations as quotients of neighbours
    double2 (*seq)[D] = sm.seq[warp];
    {
      const int back = lane & 1;
      double p = 1.0, q = 0.0;
      int i = back ? hi : lo;
      for (int s = 0; s <= hi - lo; s++) {
        const double ee = back ? (i + 1 < D ? sm.de[i + 1].y : 0.0) : sm.de[i].y;
        double t = fma(sm.de[i].x - lam, p, s == 0 ? 0.0 : -ee * q);
        if (t == 0.0) t = 1e-60 * p;
        if (lane < 2) seq[back][i] = make_double2(t, p);
        q = p;
        p = t;
        if ((s & 7) == 7) rescale(p, q);
        i += back ? -1 : 1;
      }
    }
    __syncwarp();
    // the residual of the vector that is 1 at i: the sum of the two pivots there less the diagonal element
    double best = INFINITY;
    int at = lo;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int i = lane + 32 * q;
      if (i >= lo && i <= hi) {
        const double2 f = seq[0][i], g = seq[1][i];
        const double gam = f.x / f.y + (g.x / g.y - (sm.d[i] - lam));
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
      if (i >= lo && i < at) f = -sm.e[i] * seq[0][i].y / seq[0][i].x;
      else if (i > at && i <= hi) f = -sm.e[i - 1] * seq[1][i].y / seq[1][i].x;
      else if (i == at) f = 1.0;
      z[i] = f;
    }
    __syncwarp();
    if (lane < 2) {
      const int step = lane ? 1 : -1, n = lane ? hi - at : at - lo;
      double c = 1.0;
      for (int s = 0; s < n; s += 8) {
        double f[8];
#pragma unroll
        for (int v = 0; v < 8; v++) f[v] = s + v < n ? z[at + step * (s + v + 1)] : 0.0;
#pragma unroll
        for (int v = 0; v < 8; v++)
          if (s + v < n) { c *= f[v]; z[at + step * (s + v + 1)] = c; }
      }
    }
    __syncwarp();
    double zz[4], s2 = 0.0;
#pragma unroll
    for (int q = 0; q < 4; q++) { zz[q] = z[lane + 32 * q]; s2 = fma(zz[q], zz[q], s2); }
    s2 = warp_sum(s2);
    const double inv = 1.0 / sqrt(s2);
#pragma unroll
    for (int q = 0; q < 4; q++) z[lane + 32 * q] = zz[q] * inv;
    resid = fabs(best) * inv;
    lam = fma(best * inv, inv, lam);
  } else {
#pragma unroll
    for (int q = 0; q < 4; q++) z[lane + 32 * q] = lane + 32 * q == j ? 1.0 : 0.0;
  }
  const bool resid_ok = resid <= RESIDUAL_TOL * EPS * tn && isfinite(lam);   // (false for NaN)
  asm volatile("cp.async.wait_group 0;\n" ::);
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
  if (warp < VEC / 4) {
    const int u = lane & 7, vec = 4 * warp + (lane >> 3);
    double zr[16];
#pragma unroll
    for (int m = 0; m < 8; m++) {
      const double2 t = *reinterpret_cast<const double2*>(&sm.own[vec][16 * m + 2 * u]);
      zr[2 * m] = t.x; zr[2 * m + 1] = t.y;
    }
#pragma unroll 1
    for (int grp = D / 4 - 1; grp >= 0; grp--) {
      double dot[4], c[4];
#pragma unroll
      for (int x = 0; x < 4; x++) {
        const double* v = sm.refl[4 * grp + 3 - x];
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int m = 0; m < 8; m++) {
          const double2 t = *reinterpret_cast<const double2*>(&v[16 * m + 2 * u]);
          s0 = fma(t.x, zr[2 * m], s0);
          s1 = fma(t.y, zr[2 * m + 1], s1);
        }
        dot[x] = s0 + s1;
      }
#pragma unroll
      for (int s = 1; s < 8; s <<= 1)
#pragma unroll
        for (int x = 0; x < 4; x++) dot[x] += __shfl_xor_sync(0xffffffffu, dot[x], s);
      const double* x6 = sm.wy.cross[grp];
      const double* tau = &sm.tau[4 * grp];
      c[0] = tau[3] * dot[0];
      c[1] = tau[2] * fma(-x6[0], c[0], dot[1]);
      c[2] = tau[1] * fma(-x6[3], c[1], fma(-x6[1], c[0], dot[2]));
      c[3] = tau[0] * fma(-x6[5], c[2], fma(-x6[4], c[1], fma(-x6[2], c[0], dot[3])));
#pragma unroll
      for (int x = 0; x < 4; x++) {
        const double* v = sm.refl[4 * grp + 3 - x];
#pragma unroll
        for (int m = 0; m < 8; m++) {
          const double2 t = *reinterpret_cast<const double2*>(&v[16 * m + 2 * u]);
          zr[2 * m] = fma(-c[x], t.x, zr[2 * m]);
          zr[2 * m + 1] = fma(-c[x], t.y, zr[2 * m + 1]);
        }
      }
    }
#pragma unroll
    for (int m = 0; m < 8; m++) *reinterpret_cast<double2*>(&sm.own[vec][16 * m + 2 * u]) = make_double2(zr[2 * m], zr[2 * m + 1]);
  }
  if (lane < CTAS) cluster.map_shared_rank(&sm.lam[0], lane)[j] = lam;

  // ---- Newton-Schulz: this block's rows of V^T V, then of V
  int steps = 0;
  bool good = false;
#pragma unroll 1
  for (; steps < MAX_STEPS;) {
    cluster.sync();   // every block's vectors are ready
    for (int i = tid; i < D * D / 2; i += THREADS) {
      const int row = i / (D / 2), c = 2 * (i % (D / 2));
      const double* src = cluster.map_shared_rank(&sm.own[0][0], row / VEC);
      *reinterpret_cast<double2*>(&sm.all[row][c]) = *reinterpret_cast<const double2*>(src + (row % VEC) * PITCH + c);
    }
    __syncthreads();
    const int g = lane >> 2, t = lane & 3, r0 = 8 * (warp & 1);
    double dist = 0.0;
    {
      double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
      const int c0 = 8 * (warp >> 1);
#pragma unroll 8
      for (int s = 0; s < D; s += 4) {
        const double x = sm.own[r0 + g][s + t];
        dmma(acc[0], x, sm.all[c0 + g][s + t]);
        dmma(acc[1], x, sm.all[64 + c0 + g][s + t]);
      }
#pragma unroll
      for (int h = 0; h < 2; h++)
#pragma unroll
        for (int e = 0; e < 2; e++) {
          const int col = 64 * h + c0 + 2 * t + e;
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
      double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
      const int c0 = 8 * (warp >> 1);
#pragma unroll 8
      for (int s = 0; s < D; s += 4) {
        const double x = sm.ns.g[r0 + g][s + t];
        dmma(acc[0], x, sm.all[s + t][c0 + g]);
        dmma(acc[1], x, sm.all[s + t][64 + c0 + g]);
      }
#pragma unroll
      for (int h = 0; h < 2; h++)
#pragma unroll
        for (int e = 0; e < 2; e++) {
          double* o = &sm.own[r0 + g][64 * h + c0 + 2 * t + e];
          *o = fma(-0.5, acc[h][e], 1.5 * *o);
        }
    }
    __syncthreads();
    if (err < 1e-16) { good = true; break; }   // the step just made leaves 3/4 of that, the squared distance
  }
  if (rank == 0 && tid == 0) {
    reinterpret_cast<int*>(refl[D - 1])[0] = good ? 0 : 1;   // (0: nothing left for the Jacobi solver)
    if (good && sweeps_out) *sweeps_out = steps;
  }
  if (!good) return;   // (the same for every block, none of which reads another's memory any more)

  // ---- every vector's component of largest magnitude positive (the first of equals); descending order, ties by position
  {
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
  if (tid < D) {
    const double l = sm.lam[tid];
    int pos = 0;
#pragma unroll 8
    for (int i = 0; i < D; i++) pos += sm.lam[i] > l || (sm.lam[i] == l && i < tid);
    sm.order[pos] = tid;
    if (rank == 0) lambda[pos] = (float)ldexp(l, sm.expo);
  }
  cluster.sync();   // signs are in place everywhere
  {  // R[c][k] = sum_l H[c][l] U[k][l]: warp = column k, lane holds l = lane + 32 i; a Hadamard transform per column
    double x[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const int l = lane + 32 * i, src = sm.order[l];
      x[i] = (double)signs[l] * cluster.map_shared_rank(&sm.own[0][0], src / VEC)[(src % VEC) * PITCH + j];
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
    for (int i = 0; i < 4; i++) R[(size_t)(lane + 32 * i) * D + j] = (float)(o[i] * 0.08838834764831845);   // 1 / sqrt(128)
  }
  cluster.sync();   // nobody's vectors are read any more
}

}  // namespace

cudaError_t launch_calib_spectrum(const float* C, const float* signs, double* ws, float* R, float* lambda, int* sweeps, cudaStream_t s) {
  static thread_local unsigned long long attr_mask = 0;
  int dev = 0;
  if (attr_needed(attr_mask, dev)) {
    const cudaError_t e = cudaFuncSetAttribute(k_calib_spectrum, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
    if (e != cudaSuccess) return e;
    attr_done(attr_mask, dev);
  }
  return launch_dependent(k_calib_spectrum, dim3(CTAS), THREADS, sizeof(Smem), s, CTAS, C, signs, ws, R, lambda, sweeps);
}

}  // namespace okq
