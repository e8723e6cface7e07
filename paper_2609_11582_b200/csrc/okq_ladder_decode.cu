// Decode attention over the canonical cache of the bit-width ladder (2, 3 and 4 bits per code).
//
// A thread-block cluster owns one (sequence, KV head); its warps take contiguous ranges of 32-token windows and do
// everything of a window by themselves:
//   * scores S^T[head][token] = W[head][channel] C[channel][token] on mma.sync: a code masked out of its word becomes an fp16
//     number with one addition, the weights q'_c s_gc are split into fp16 high and low parts in the 16 rows of the m16 tile, so a
//     product has 2^-22 of the weight; the channels of a k-step are those whose codes lie together in a lane's bytes of the
//     token's bit stream (3-bit codes are first spread to nibbles, seven operations for eight codes);
//   * online softmax in fp32, the reference maximum moving only when it is exceeded by 2^RESCALE;
//   * value sums in fp32 multiply-adds: half a warp per token parity, eight channels and all heads per lane, levels from a
//     16-entry table in shared memory.  (Tensor cores would need the numerators and the levels in two fp16 parts each: as
//     many dispatch cycles, and the table look-ups twice.)
// A lane's registers hold the sums of one modality; they are added to the warp's sums in shared memory at a change.
// At the end a block merges its warps, the cluster its blocks through distributed shared memory, and each block applies
// R_m^T for its share of the output columns.
// What bounds it: issue slots, about 900 multiply-adds, 128 look-ups and 40 products per window of seven heads.
// 64 sequences x 4 heads x 8192 tokens at 4 bits: 2382 us with one block per (sequence, head), block-wide steps per window
// and shuffle-reduced scores, 251 us in this form (243 us with the codes as subnormals).
// Error against 64 bits, 32 to 16384 tokens: 0.3 to 0.9e-6 (the fp32 kernel it replaced: 0.4 to 1.9e-6).
#include <cooperative_groups.h>
#include "../../include/okq_ladder.h"
#include "okq_decode_frag.cuh"
#include "okq_ladder.cuh"

namespace cg = cooperative_groups;

namespace okq {

namespace {

constexpr int NW = 8;                     // warps per block
constexpr int NT_L = NW * 32;
constexpr int NS = 3;                     // staged windows per warp
constexpr float RESCALE = 8.0f;
constexpr int P_PITCH = 12;               // floats per token of the numerators: eight rows of a column over all banks

template <int BITS> struct SlotL {
  static constexpr int CODE = W * 16 * BITS;             // bytes of a window's code rows
  static constexpr int META = 0, KC = 512, VC = KC + CODE, KN = VC + CODE, VN = KN + 64, BYTES = VN + 64;
};
template <int BITS> struct WarpL {
  __align__(16) unsigned char slot[NS][SlotL<BITS>::BYTES];
  __align__(16) float p[W][P_PITCH];      // numerators times value norms, [token][head]
  __align__(16) float sum[3][GP][D];      // rotated-basis sums per modality
};
template <int BITS> struct BlockL {
  WarpL<BITS> w[NW];
  __align__(16) float q[GP][D];           // rotated queries, scaled by 2^kh
  float fsc[GP], lev[16];
  float m[NW][GP], l[NW][GP];             // per warp: reference maximum, sum of exp2(score - maximum)
  int held[NW];                           // modalities a warp holds sums of
  float M[GP], L[GP];                     // the block's
  float fac[16][GP];                      // factors of the parts being merged
};

__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src));
}

// eight 3-bit codes in the low 24 bits -> eight nibbles (bit 3 of a nibble is not defined)
__device__ __forceinline__ uint32_t spread3(uint32_t x) {
  x = (x & 0x00000fffu) | ((x << 4) & ~0x00000fffu);
  x = (x & 0x003f003fu) | ((x << 2) & ~0x003f003fu);
  return (x & 0x07070707u) | ((x << 1) & ~0x07070707u);
}

// The two masked fields of x as fp16 numbers.  Masked fields alone are subnormals, which the tensor cores multiply exactly but
// align like numbers of the smallest normal exponent: with up to ten leading zeros that leaves as many digits fewer to the
// sums (scores 7e-6 off at 2 bits, results ten times further off than fp32 arithmetic).  1024 + code is exact, and so is the
// difference.
__device__ __forceinline__ uint32_t code_pair(uint32_t x, uint32_t mask) {
  return h2u(__hsub2(u2h((x & mask) | 0x64006400u), u2h(0x64006400u)));
}

// pair p of a lane's 32 channels 32 t + ..: the two codes of one mask (low and high half of a register), their distance,
// and the power of two by which the masked field exceeds the code
template <int BITS> struct Pairs {
  static constexpr int WORDS = BITS == 2 ? 2 : 4;        // words of codes per lane and token (3 bits: as nibbles)
  static constexpr int PER = 16 / WORDS;                 // pairs per word
  static constexpr int DIST = BITS == 2 ? 8 : 4;
  static constexpr int FIELD = BITS == 2 ? 2 : 4;
  static constexpr int IN_BYTE = 8 / FIELD;              // fields of the low byte
  __host__ __device__ static constexpr int channel(int p) { return (p / PER) * (32 / WORDS) + p % PER; }
  __host__ __device__ static constexpr int shift(int p) { return FIELD * ((p % PER) % IN_BYTE); }
  static constexpr uint32_t ONES = (BITS == 2 ? 0x3u : BITS == 3 ? 0x7u : 0xfu) * 0x00010001u;
};

// NH: heads whose value sums are formed, the group rounded up to 2, 5, 7 or 8 (the scores' m16 tile holds eight either way)
template <int BITS, int NH>
__global__ void __launch_bounds__(NT_L, 1) k_ladder_decode(LadderView cv, int n_tokens, const __half* __restrict__ q,
                                                          float sm_scale, const float* __restrict__ signs,
                                                          const float* __restrict__ R, int n_R, float* __restrict__ out) {
  using SL = SlotL<BITS>;
  using PR = Pairs<BITS>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BlockL<BITS>& sm = *reinterpret_cast<BlockL<BITS>*>(smem_raw);
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int unit = blockIdx.x / cs, h = unit % cv.n_kv_heads, b = unit / cv.n_kv_heads;
  const int G = cv.n_q_heads / cv.n_kv_heads;
  const int n_win = n_tokens / W;
  const size_t u = cv.unit(b, h);
  WarpL<BITS>& ws = sm.w[warp];
  depend_wait();

  // ---- this warp's windows, the first ones on their way
  const int cnt = (n_win + cs * NW - 1) / (cs * NW);
  const int w0 = min(n_win, (rank * NW + warp) * cnt), w1 = min(n_win, w0 + cnt);
  const uint32_t slots = (uint32_t)__cvta_generic_to_shared(&ws.slot[0][0]);
  auto issue = [&](int win) {
    if (win < w1) {
      const uint32_t dst = slots + (uint32_t)((win - w0) % NS) * SL::BYTES;
      const size_t tok0 = u * cv.capacity + (size_t)win * W;
      const unsigned char* kc = cv.k_codes + tok0 * (16 * BITS);
      const unsigned char* vc = cv.v_codes + tok0 * (16 * BITS);
#pragma unroll
      for (int i = 0; i < BITS; i++) {
        cp16(dst + SL::KC + 16 * (lane + 32 * i), kc + 16 * (lane + 32 * i));
        cp16(dst + SL::VC + 16 * (lane + 32 * i), vc + 16 * (lane + 32 * i));
      }
      // (m, s): chunk c = 8 t + i (channels 32 t + 4 i ..) goes to place 4 i + t: four lanes t read 64 contiguous bytes
      cp16(dst + SL::META + 16 * (4 * (lane & 7) + (lane >> 3)),
           reinterpret_cast<const unsigned char*>(cv.k_meta) + (u * (cv.capacity / W) + win) * (D * 4) + 16 * lane);
      if (lane < 4) cp16(dst + SL::KN + 16 * lane, cv.k_norm + tok0 + 8 * lane);
      else if (lane < 8) cp16(dst + SL::VN + 16 * (lane - 4), cv.v_norm + tok0 + 8 * (lane - 4));
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };
#pragma unroll
  for (int i = 0; i < NS - 1; i++) issue(w0 + i);
  const unsigned char* mod_row = cv.modality + (size_t)b * cv.capacity;
  int mod_next = w0 < w1 ? mod_row[w0 * W + lane] : 0;

  // ---- rotated queries: warp j = head j
  if (tid < 16) sm.lev[tid] = ladder_level(BITS, tid);
  {
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (warp < G) {
      x = load_row4(q + ((size_t)b * cv.n_q_heads + (size_t)h * G + warp) * D, lane);
      const float4 sg = *reinterpret_cast<const float4*>(signs + 4 * lane);
      x = warp_fwht(make_float4(sg.x * x.x, sg.y * x.y, sg.z * x.z, sg.w * x.w), lane);
      x.x *= RSQRT_D; x.y *= RSQRT_D; x.z *= RSQRT_D; x.w *= RSQRT_D;
    }
    float mx = fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w)));
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
    int ex = 0;
    if (mx > 0.f) frexpf(mx, &ex);          // mx < 2^ex
    const int kh = 13 - ex;                 // |q'| * 2^kh < 2^13; times the largest step (2 sqrt(128) / 3) still an fp16 number
    const float up = exp2f((float)kh);
    *reinterpret_cast<float4*>(&sm.q[warp][4 * lane]) = make_float4(x.x * up, x.y * up, x.z * up, x.w * up);
    if (lane == 0) sm.fsc[warp] = exp2f((float)-kh) * sm_scale * 1.4426950408889634f;
  }
  __syncthreads();
  uint32_t qh[16], ql[16];
#pragma unroll
  for (int p = 0; p < 16; p++) {
    const int c = 32 * t + PR::channel(p);
    const float f = 1.0f / (float)(1 << PR::shift(p));
    const float x0 = sm.q[g][c] * f, x1 = sm.q[g][c + PR::DIST] * f;
    const __half2 hi = __floats2half2_rn(x0, x1);
    const float2 hf = __half22float2(hi);
    qh[p] = h2u(hi);
    ql[p] = h2u(__floats2half2_rn(x0 - hf.x, x1 - hf.y));
  }
  const float fsc = sm.fsc[g];

  const int hw = lane >> 4, l16 = lane & 15;   // value sums: token parity, channels 8 l16 .. 8 l16 + 7
  float acc[NH][8];
#pragma unroll
  for (int j = 0; j < NH; j++)
#pragma unroll
    for (int c = 0; c < 8; c++) acc[j][c] = 0.f;
  float run_m = -INFINITY, run_l = 0.f;
  int cur_mod = -1, held = 0;

  auto deposit = [&]() {
    // the half-warps hold the sums of even and odd tokens: lanes of the first half take heads 0..3, of the second 4..7
    float* row = &ws.sum[cur_mod][0][8 * l16];
#pragma unroll
    for (int j = 0; j < 4; j++) {
      float v[8];
#pragma unroll
      for (int c = 0; c < 8; c++) {
        const float lo = j < NH ? acc[j < NH ? j : 0][c] : 0.f, hi = j + 4 < NH ? acc[j + 4 < NH ? j + 4 : 0][c] : 0.f;
        const float give = hw ? lo : hi, keep = hw ? hi : lo;
        v[c] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
      }
      float4* dst = reinterpret_cast<float4*>(row + (4 * hw + j) * D);
      float4 a = make_float4(v[0], v[1], v[2], v[3]), e = make_float4(v[4], v[5], v[6], v[7]);
      if ((held >> cur_mod) & 1) {
        const float4 x = dst[0], y = dst[1];
        a.x += x.x; a.y += x.y; a.z += x.z; a.w += x.w;
        e.x += y.x; e.y += y.y; e.z += y.z; e.w += y.w;
      }
      dst[0] = a;
      dst[1] = e;
    }
    held |= 1 << cur_mod;
#pragma unroll
    for (int j = 0; j < NH; j++)
#pragma unroll
      for (int c = 0; c < 8; c++) acc[j][c] = 0.f;
  };

  for (int win = w0; win < w1; win++) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(NS - 2));
    __syncwarp();   // the window has landed for every lane; everyone is done with the slot that is filled next
    issue(win + NS - 1);
    const unsigned char* st = &ws.slot[(win - w0) % NS][0];
    const int mymod = min(mod_next, 2);
    if (win + 1 < w1) mod_next = mod_row[(size_t)(win + 1) * W + lane];

    // ---- scores: head g, tokens 8 nu + 2 t + e
    float sc[4][2];
    {
      uint32_t kw[4][PR::WORDS];
#pragma unroll
      for (int nu = 0; nu < 4; nu++) {
        const unsigned char* row = st + SL::KC + (8 * nu + g) * (16 * BITS) + 4 * BITS * t;
        if constexpr (BITS == 4) {
          const uint4 x = *reinterpret_cast<const uint4*>(row);
          kw[nu][0] = x.x; kw[nu][1] = x.y; kw[nu][2] = x.z; kw[nu][3] = x.w;
        } else if constexpr (BITS == 2) {
          const uint2 x = *reinterpret_cast<const uint2*>(row);
          kw[nu][0] = x.x; kw[nu][1] = x.y;
        } else {
          const uint32_t* r = reinterpret_cast<const uint32_t*>(row);
          const uint32_t a = r[0], c = r[1], e = r[2];
          kw[nu][0] = spread3(a);
          kw[nu][1] = spread3(__funnelshift_r(a, c, 24));
          kw[nu][2] = spread3(__funnelshift_r(c, e, 16));
          kw[nu][3] = spread3(e >> 8);
        }
      }
      float d[4][4], dbA[4], dbB[4];
#pragma unroll
      for (int w = 0; w < PR::WORDS; w++) {
        // (m, s) of the word's channels: chunk i = channels 4 i .. 4 i + 3 of the lane's 32
        constexpr int CH = 8 / PR::WORDS;
        uint32_t ms[CH][4];
#pragma unroll
        for (int i = 0; i < CH; i++) {
          const uint4 x = *reinterpret_cast<const uint4*>(st + SL::META + 16 * (4 * (w * CH + i) + t));
          ms[i][0] = x.x; ms[i][1] = x.y; ms[i][2] = x.z; ms[i][3] = x.w;
        }
#pragma unroll
        for (int jk = 0; jk < PR::PER / 2; jk++) {   // k-step: pairs 2 jk, 2 jk + 1 of the word
          uint32_t a[4], mb[2];
#pragma unroll
          for (int e = 0; e < 2; e++) {
            const int j = 2 * jk + e, p = w * PR::PER + j;
            const uint32_t x = ms[j / 4][j % 4], y = ms[j / 4 + CH / 2][j % 4];
            uint32_t s2, m2;
            asm("prmt.b32 %0, %1, %2, 0x7632;\n" : "=r"(s2) : "r"(x), "r"(y));
            asm("prmt.b32 %0, %1, %2, 0x5410;\n" : "=r"(m2) : "r"(x), "r"(y));
            if (PR::shift(p)) m2 = h2u(__hmul2(u2h(m2), __float2half2_rn((float)(1 << PR::shift(p)))));   // exact: |m| <= 1
            mb[e] = m2;
            split_product(u2h(qh[p]), u2h(ql[p]), u2h(s2), a[2 * e], a[2 * e + 1]);
          }
          const int p0 = w * PR::PER + 2 * jk;
          const bool first = p0 < 2;
          float (&db)[4] = (jk & 1) ? dbB : dbA;
          if (p0 < 4) mma16816_first(db, qh[p0], ql[p0], qh[p0 + 1], ql[p0 + 1], mb[0], mb[1]);
          else mma16816(db, qh[p0], ql[p0], qh[p0 + 1], ql[p0 + 1], mb[0], mb[1]);
#pragma unroll
          for (int nu = 0; nu < 4; nu++) {
            const uint32_t x0 = (2 * jk) / PR::IN_BYTE ? kw[nu][w] >> 8 : kw[nu][w];
            const uint32_t b0 = code_pair(x0, PR::ONES << PR::shift(p0)), b1 = code_pair(x0, PR::ONES << PR::shift(p0 + 1));
            if (first) mma16816_first(d[nu], a[0], a[1], a[2], a[3], b0, b1);
            else mma16816(d[nu], a[0], a[1], a[2], a[3], b0, b1);
          }
        }
      }
      const float bias = (dbA[0] + dbB[0]) + (dbA[2] + dbB[2]);
#pragma unroll
      for (int nu = 0; nu < 4; nu++) {
        const float2 kn = __half22float2(*reinterpret_cast<const __half2*>(st + SL::KN + 2 * (8 * nu + 2 * t)));
        sc[nu][0] = ((d[nu][0] + d[nu][2]) + bias) * (kn.x * fsc);
        sc[nu][1] = ((d[nu][1] + d[nu][3]) + bias) * (kn.y * fsc);
      }
    }
    // ---- online softmax (log2 domain)
    float mx = -INFINITY;
#pragma unroll
    for (int nu = 0; nu < 4; nu++) mx = fmaxf(mx, fmaxf(sc[nu][0], sc[nu][1]));
    if (__any_sync(0xffffffffu, !(mx <= run_m + RESCALE))) {
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float m_new = fmaxf(mx, run_m);
      const float alpha = exp2f(run_m - m_new);   // 0 on the first window
      run_m = m_new;
      run_l *= alpha;
      float al[GP];
#pragma unroll
      for (int j = 0; j < GP; j++) al[j] = __shfl_sync(0xffffffffu, alpha, 4 * j);
#pragma unroll
      for (int j = 0; j < NH; j++)
#pragma unroll
        for (int c = 0; c < 8; c++) acc[j][c] *= al[j];
      for (int m = 0; m < 3; m++)
        if ((held >> m) & 1)
#pragma unroll
          for (int j = 0; j < GP; j++)
            for (int c = lane; c < D; c += 32) ws.sum[m][j][c] *= al[j];
      __syncwarp();
    }
#pragma unroll
    for (int nu = 0; nu < 4; nu++) {
      const float2 vn = __half22float2(*reinterpret_cast<const __half2*>(st + SL::VN + 2 * (8 * nu + 2 * t)));
      const float p0 = ex2(sc[nu][0] - run_m), p1 = ex2(sc[nu][1] - run_m);
      run_l += p0 + p1;
      ws.p[8 * nu + 2 * t][g] = p0 * vn.x;
      ws.p[8 * nu + 2 * t + 1][g] = p1 * vn.y;
    }
    __syncwarp();
    // ---- value sums of the tokens of modality cur_mod among `sel`
    auto token = [&](int i, bool masked, unsigned sel) {   // tokens 2 i + hw
      const int tok = 2 * i + hw;
      const unsigned char* row = st + SL::VC + tok * (16 * BITS);
      uint32_t x;   // eight codes, one nibble each (2 bits: packed)
      if constexpr (BITS == 4) x = reinterpret_cast<const uint32_t*>(row)[l16];
      else if constexpr (BITS == 2) x = reinterpret_cast<const uint16_t*>(row)[l16];
      else {
        const uint32_t* r = reinterpret_cast<const uint32_t*>(row) + ((3 * l16) >> 2);
        x = __funnelshift_r(r[0], r[1], 8 * ((3 * l16) & 3));   // (the second word may lie behind the row: not used then)
      }
      const float4 pa = *reinterpret_cast<const float4*>(&ws.p[tok][0]);
      float4 pb = make_float4(0.f, 0.f, 0.f, 0.f);
      if (NH > 4) pb = *reinterpret_cast<const float4*>(&ws.p[tok][4]);
      float pv[GP] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
      if (masked && !((sel >> tok) & 1u)) {
#pragma unroll
        for (int j = 0; j < NH; j++) pv[j] = 0.f;
      }
      const char* lev = reinterpret_cast<const char*>(sm.lev);
#pragma unroll
      for (int c = 0; c < 8; c++) {
        const int sh = BITS * c - 2;
        const uint32_t off = (sh < 0 ? x << 2 : x >> sh) & (((1u << BITS) - 1u) << 2);
        const float lv = *reinterpret_cast<const float*>(lev + off);
#pragma unroll
        for (int j = 0; j < NH; j++) acc[j][c] = fmaf(pv[j], lv, acc[j][c]);
      }
    };
    const unsigned mine = __ballot_sync(0xffffffffu, mymod == cur_mod);
    if (mine == 0xffffffffu) {
#pragma unroll 4
      for (int i = 0; i < W / 2; i++) token(i, false, 0u);
    } else {
      unsigned present = (__any_sync(0xffffffffu, mymod == 0) ? 1u : 0u) | (__any_sync(0xffffffffu, mymod == 1) ? 2u : 0u) |
                         (__any_sync(0xffffffffu, mymod == 2) ? 4u : 0u);
      while (present) {   // the modality the registers hold first
        const int m = cur_mod >= 0 && ((present >> cur_mod) & 1u) ? cur_mod : __ffs(present) - 1;
        present &= ~(1u << m);
        if (m != cur_mod) {
          if (cur_mod >= 0) deposit();
          cur_mod = m;
        }
        const unsigned sel = __ballot_sync(0xffffffffu, mymod == m);
        const int i0 = (__ffs(sel) - 1) >> 1, i1 = (31 - __clz(sel)) >> 1;
#pragma unroll 1
        for (int i = i0; i <= i1; i++)
          if ((sel >> (2 * i)) & 3u) token(i, true, sel);
      }
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::);
  if (cur_mod >= 0) deposit();
  run_l += __shfl_xor_sync(0xffffffffu, run_l, 1);
  run_l += __shfl_xor_sync(0xffffffffu, run_l, 2);
  if (t == 0) { sm.m[warp][g] = run_m; sm.l[warp][g] = run_l; }
  if (lane == 0) sm.held[warp] = held;
  __syncthreads();

  // ---- the block's sums: maximum and factors per head, then 3 x 8 x 128 sums over the warps
  if (tid < GP) {
    float M = -INFINITY, L = 0.f;
    for (int w = 0; w < NW; w++) M = fmaxf(M, sm.m[w][tid]);
    for (int w = 0; w < NW; w++) {
      const float f = sm.m[w][tid] == -INFINITY ? 0.f : exp2f(sm.m[w][tid] - M);
      sm.fac[w][tid] = f;
      L += sm.l[w][tid] * f;
    }
    sm.M[tid] = M;
    sm.L[tid] = L;
  }
  __syncthreads();
  float4 merged[3];
#pragma unroll
  for (int i = 0; i < 3; i++) {
    const int idx = 4 * (tid + NT_L * i), m = idx / (GP * D), j = (idx / D) % GP;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int w = 0; w < NW; w++)
      if ((sm.held[w] >> m) & 1) {
        const float4 x = *reinterpret_cast<const float4*>(&sm.w[w].sum[0][0][0] + idx);
        const float f = sm.fac[w][j];
        a.x = fmaf(x.x, f, a.x); a.y = fmaf(x.y, f, a.y); a.z = fmaf(x.z, f, a.z); a.w = fmaf(x.w, f, a.w);
      }
    merged[i] = a;
  }
  __syncthreads();
  float* tot = &sm.w[0].sum[0][0][0];   // [modality][head][channel]: in the first warp's place
#pragma unroll
  for (int i = 0; i < 3; i++) *reinterpret_cast<float4*>(tot + 4 * (tid + NT_L * i)) = merged[i];
  if (cs > 1) {   // ---- the cluster's: every block reads all of them
    cluster.sync();
    if (tid < GP) {
      float M = -INFINITY, L = 0.f;
      for (int r = 0; r < cs; r++) M = fmaxf(M, cluster.map_shared_rank(&sm.M[0], r)[tid]);
      for (int r = 0; r < cs; r++) {
        const float mr = cluster.map_shared_rank(&sm.M[0], r)[tid];
        const float f = mr == -INFINITY ? 0.f : exp2f(mr - M);
        sm.fac[r][tid] = f;
        L += cluster.map_shared_rank(&sm.L[0], r)[tid] * f;
      }
      sm.fsc[tid] = L;   // (L itself is still being read by the other blocks)
    }
    __syncthreads();
    float* all = &sm.w[1].sum[0][0][0];
#pragma unroll
    for (int i = 0; i < 3; i++) {
      const int idx = 4 * (tid + NT_L * i), j = (idx / D) % GP;
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int r = 0; r < cs; r++) {
        const float4 x = *reinterpret_cast<const float4*>(cluster.map_shared_rank(tot, r) + idx);
        const float f = sm.fac[r][j];
        a.x = fmaf(x.x, f, a.x); a.y = fmaf(x.y, f, a.y); a.z = fmaf(x.z, f, a.z); a.w = fmaf(x.w, f, a.w);
      }
      *reinterpret_cast<float4*>(all + idx) = a;
    }
    tot = all;
    cluster.sync();   // everyone has read everyone's sums
  } else {
    if (tid < GP) sm.fsc[tid] = sm.L[tid];
    __syncthreads();
  }
  // ---- out[j][c] = sum_r R[r][c] tot[r][j] / L for this block's columns: thread = (column, slice of the 384 rows), all heads
  {
    const int C = D / cs, c = tid % C, slices = NT_L / C, ks = tid / C, rows = 3 * D / slices;   // C = 128 .. 16: 2 .. 16 slices
    const float* Rc = R + (size_t)(n_R == 1 ? 0 : h) * 3 * D * D + rank * C + c;
    float o[GP];
#pragma unroll
    for (int j = 0; j < GP; j++) o[j] = 0.f;
#pragma unroll 8
    for (int r = ks * rows; r < (ks + 1) * rows; r++) {
      const float x = __ldg(Rc + (size_t)r * D);
      const float* v = tot + (r / D) * GP * D + (r % D);
#pragma unroll
      for (int j = 0; j < GP; j++) o[j] = fmaf(x, v[j * D], o[j]);
    }
    float* part = &sm.w[2].sum[0][0][0];   // [slice][head][column]
#pragma unroll
    for (int j = 0; j < GP; j++) part[(ks * GP + j) * C + c] = o[j];
    __syncthreads();
    for (int i = tid; i < G * C; i += NT_L) {
      const int j = i / C, cc = i % C;
      float s = 0.f;
      for (int k = 0; k < slices; k++) s += part[(k * GP + j) * C + cc];
      const float L = sm.fsc[j];
      out[((size_t)b * cv.n_q_heads + (size_t)h * G + j) * D + rank * C + cc] = L > 0.f ? s / L : 0.f;
    }
  }
}

template <int BITS, int NH>
cudaError_t launch_heads(const LadderView& cv, int cs, int n_tokens, const __half* q, float sm_scale, const float* signs, const float* R,
                   int n_R, float* out, cudaStream_t s) {
  static_assert(sizeof(BlockL<BITS>) <= 227 * 1024, "shared memory of one block");
  static thread_local unsigned long long attr_mask = 0;
  int dev = 0;
  if (attr_needed(attr_mask, dev)) {
    const cudaError_t e = cudaFuncSetAttribute(k_ladder_decode<BITS, NH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BlockL<BITS>));
    if (e != cudaSuccess) return e;
    attr_done(attr_mask, dev);
  }
  return launch_dependent(k_ladder_decode<BITS, NH>, dim3((unsigned)(cv.batch * cv.n_kv_heads * cs)), NT_L, sizeof(BlockL<BITS>), s, cs, cv,
                          n_tokens, q, sm_scale, signs, R, n_R, out);
}

template <int BITS, class... A>
cudaError_t launch(const LadderView& cv, A... args) {
  const int G = cv.n_q_heads / cv.n_kv_heads;
  return G <= 2 ? launch_heads<BITS, 2>(cv, args...) : G <= 5 ? launch_heads<BITS, 5>(cv, args...)
       : G <= 7 ? launch_heads<BITS, 7>(cv, args...) : launch_heads<BITS, 8>(cv, args...);
}

}  // namespace

// Blocks per (sequence, head): the split with the shortest makespan, waves x (windows of a warp + fixed part), with the
// fixed part (queries, merge, R_m^T) worth about eight windows; clusters of four reach 8/9 of the SMs, of eight 4/5.
cudaError_t launch_ladder_decode(const LadderView& cv, int n_tokens, const __half* q, float sm_scale, const float* signs,
                                 const float* R, int n_R, float* out, cudaStream_t s) {
  const long long units = (long long)cv.batch * cv.n_kv_heads, n_win = n_tokens / W, sms = sm_count();
  int best = 1;
  long long best_cost = 0;
  for (int cs = 1; cs <= 8; cs *= 2) {
    const long long slots = cs <= 2 ? sms / cs * cs : cs == 4 ? sms * 8 / 9 : sms * 4 / 5;
    const long long waves = (units * cs + slots - 1) / slots;
    const long long cost = waves * ((n_win + cs * NW - 1) / (cs * NW) + 8);
    if (cs == 1 || cost < best_cost) { best = cs; best_cost = cost; }
  }
  return cv.bits == 2 ? launch<2>(cv, best, n_tokens, q, sm_scale, signs, R, n_R, out, s)
       : cv.bits == 3 ? launch<3>(cv, best, n_tokens, q, sm_scale, signs, R, n_R, out, s)
                      : launch<4>(cv, best, n_tokens, q, sm_scale, signs, R, n_R, out, s);
}

}  // namespace okq
