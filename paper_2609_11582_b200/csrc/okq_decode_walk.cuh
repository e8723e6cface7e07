// One warp's pass over packed windows, shared by the split-K kernel (okq_decode_mma.cu) and the one-launch kernel for few
// (sequence, head) units (okq_decode_small.cu): scores, online softmax and value sums of a contiguous range of windows.
#pragma once
#include "okq_common.cuh"
#include "okq_device.cuh"
#include "okq_decode_shared.cuh"
#include "okq_decode_frag.cuh"

namespace okq {

namespace {

constexpr int NWARP = DECODE_WARPS;
constexpr int NTHREADS = NWARP * 32;
constexpr int PREFETCH = 3;                     // windows copied ahead of the one whose values are summed
constexpr int NSLOT = PREFETCH + 1;             // record ring per warp
constexpr int BATCH = 8;                        // windows whose bias sums come out of one set of products
constexpr int M_PITCH = 256 + 16;               // bytes between the m planes of a batch: eight rows over all banks
// Numerators are p * vnorm in fp16, p = 2^(score - reference).  The reference is chosen by the numerators themselves and not by
// the scores: when it moves, the largest numerator of the window gets a p that is a power of two (so it is exact) and lies in
// [2^TOP_LOG2, 2^(TOP_LOG2 + 1)); it moves again when one exceeds NUM_MAX.  That leaves 25 binary digits below the largest one
// whatever the values' scale is, and whatever mass a token with a small value takes.  Error against 64 bits, 16384 tokens, first
// token 20 bits above the others with a zero value, values of norm 0.004: 2.4e-2 with the reference at the largest score and 2^-4
// there, 1.4e-4 now; generator's inputs, 8192 tokens, MXFP4: 1.6e-4 and 0.6e-4.  A limit 16 to 32 times the top instead of 8 to
// 16 measured 0.5 % less time and 1.3 times the error.  step7b 508 -> 517 us.
constexpr int TOP_LOG2 = 11;
constexpr float NUM_MAX = 32768.0f;
// p itself only enters the fp32 weight sum: a token with next to no value may have a large one, up to 2^P_LOG2_MAX when the
// reference moves; a window whose sum exceeds SUM_MAX moves it.  (Where no token of a window has a value, that is where the
// reference goes: the next value brings it to where it belongs.)
constexpr float P_LOG2_MAX = 60.0f, SUM_MAX = 0x1p80f;
constexpr float REBASE_LOG2 = 30.0f;            // range of a piece's numbers above its own reference
constexpr int FLUSH = 32;                       // windows a warp accumulates in registers at most
constexpr int SWITCH_AFTER = 3;                 // pure windows of another modality in a row before the registers change over

// a staged window: the record from its s plane on (fp16 metadata) or its body alone (MXFP4)
template <int FMT> struct Slot {
  static constexpr int BODY = FMT == FMT_FP16 ? RECORD_BYTES - OFF_KS - BODY_BYTES : 0;
  static constexpr int BYTES = BODY + BODY_BYTES;
};
constexpr int MX_BLOCK_META = 2 * MX_META_BYTES;   // the two windows of a block: 272 bytes, 16-byte aligned

template <int FMT> struct WarpSmem {
  __align__(16) unsigned char slot[NSLOT][Slot<FMT>::BYTES];
  __align__(16) float bias[BATCH][GP];         // bias sums of a batch of windows
  __align__(16) unsigned char mod[2][BATCH * W];   // modality bytes of two batches: in use, on its way
  float rebase[32];                            // per lane, rarely used: reference of the piece
  // m planes of a batch of windows: as copied (fp16 metadata) or as decoded (MXFP4)
  __align__(16) unsigned char m[BATCH * M_PITCH];
  __align__(16) unsigned char s[FMT == FMT_FP16 ? 16 : BATCH * 256];                      // MXFP4: decoded s planes of the batch
  __align__(16) unsigned char mx[FMT == FMT_FP16 ? 16 : (BATCH / 2) * MX_BLOCK_META];     // MXFP4: stored metadata of the batch
};

struct Segment {
  const unsigned char* rec0;   // first record of the (layer, sequence, head)
  const unsigned char* mod0;   // modality row of the sequence
  int w0, n_my;                // this warp's windows of that (layer, sequence, head): first window, count
  WarpPiece* piece;            // where the warp leaves what it accumulated
};

// ---- level operand of the value product: fp16 numbers with a common low byte, so that a level is one byte to look up.
// The magnitudes 1542 / 1024 and 4 * 1286 / 1024 have the codebook's ratio b / a to 1.6e-5; LEVEL_UNIT (the least-squares
// scale, levels weighted with their probabilities) leaves 0.5e-5 on a and 1.1e-5 on b, below a tenth of the numerators' rounding.
constexpr uint32_t LEVEL_HI = 0x453EBEC5u;      // high bytes of -b, -a, a, b (code 0 in the low byte)
constexpr uint32_t LEVEL_LO = 0x06060606u;
constexpr double LV_A = 1542.0 / 1024.0, LV_B = 4.0 * 1286.0 / 1024.0, PR_A = 0.6738, PR_B = 0.3262;
constexpr float LEVEL_UNIT = (float)((PR_A * CB_INNER * LV_A + PR_B * CB_OUTER * LV_B) / (PR_A * LV_A * LV_A + PR_B * LV_B * LV_B));

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;\n" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}

__device__ __forceinline__ F2 half2_to_f2(uint32_t h) {
  const float2 f = __half22float2(u2h(h));
  return f2(f.x, f.y);
}

__device__ __forceinline__ void red_add(float4* p, float4 v) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// Scores of one packed window against the group's queries, by one warp, from a staged image of the window's key
// part ((m, s) planes, key norms, key codes at their record offsets): the split-K kernel's score step.
// sc[nu][e] = log2-domain score of head g = lane >> 2 against token 8 nu + 2 (lane & 3) + e.
__device__ __forceinline__ void window_scores_mma(const unsigned char* st, const uint2 (&qreg)[16], float fsc, int lane,
                                                  float (&sc)[4][2]) {
  const int t = lane & 3;
  const uint4* mp = reinterpret_cast<const uint4*>(st + OFF_KM + 64 * t);
  const uint4* sp = reinterpret_cast<const uint4*>(st + OFF_KS + 64 * t);
  float dbA[4] = {0.f, 0.f, 0.f, 0.f}, dbB[4] = {0.f, 0.f, 0.f, 0.f};
  float d[4][4];
#pragma unroll
  for (int nu = 0; nu < 4; nu++)
#pragma unroll
    for (int i = 0; i < 4; i++) d[nu][i] = 0.f;
  const uint4 kc0 = *reinterpret_cast<const uint4*>(st + OFF_KCODE + 16 * kpiece_slot(lane));
  const uint4 kc1 = *reinterpret_cast<const uint4*>(st + OFF_KCODE + 16 * kpiece_slot(32 + lane));
  const uint32_t kw[4][2] = {{kc0.x, kc0.y}, {kc0.z, kc0.w}, {kc1.x, kc1.y}, {kc1.z, kc1.w}};
#pragma unroll
  for (int kq = 0; kq < 4; kq++) {
    const uint4 m4 = mp[kq], s4 = sp[kq];
#pragma unroll
    for (int half = 0; half < 2; half++) {
      const int kappa = 2 * kq + half;
      const uint2 q0 = qreg[2 * kappa], q1 = qreg[2 * kappa + 1];
      uint32_t a0, a1, a2, a3;
      if (half) mma16816(dbB, q0.x, q0.y, q1.x, q1.y, m4.z, m4.w);
      else mma16816(dbA, q0.x, q0.y, q1.x, q1.y, m4.x, m4.y);
      split_product(u2h(q0.x), u2h(q0.y), u2h(half ? s4.z : s4.x), a0, a1);
      split_product(u2h(q1.x), u2h(q1.y), u2h(half ? s4.w : s4.y), a2, a3);
      const int ww = kappa >> 2, sh = (kappa >> 1) & 1;
      const uint32_t mk0 = half ? 0x00300030u : 0x00030003u;
      const uint32_t mk1 = half ? 0x00c000c0u : 0x000c000cu;
#pragma unroll
      for (int nu = 0; nu < 4; nu++) {
        uint32_t src = sh ? (kw[nu][ww] >> 8) : kw[nu][ww];
        mma16816(d[nu], a0, a1, a2, a3, src & mk0, src & mk1);
      }
    }
  }
  const uint4 kn4 = *reinterpret_cast<const uint4*>(st + OFF_KNORM + 16 * t);
  const uint32_t knu[4] = {kn4.x, kn4.y, kn4.z, kn4.w};
  const float bias0 = ((dbA[0] + dbB[0]) + (dbA[2] + dbB[2])) * 0x1p-24f;   // the code sums carry 2^-24, the bias does not
#pragma unroll
  for (int nu = 0; nu < 4; nu++) {
    const float2 kn = __half22float2(u2h(knu[nu]));
    sc[nu][0] = ((d[nu][0] + d[nu][2]) + bias0) * (kn.x * fsc);
    sc[nu][1] = ((d[nu][1] + d[nu][3]) + bias0) * (kn.y * fsc);
  }
}

// what a warp ends a range with, besides the piece's sums: lane (g, t) of head g
struct WalkEnd {
  float m, l;      // reference of everything in the piece (log2 domain), sum of exp2(score - reference)
  unsigned held;   // modalities the piece holds something of (bit per modality)
};

// ---------------------------------------------------------------- one warp's windows of one (sequence, head)
// queries(qh, fsc) fills the lane's 16 high query fragments and the head's scale, once the first copies are on their way;
// the low fragments stay in shared memory, qlo[kq][lane] = fragments 4 kq .. 4 kq + 3.
template <int FMT, class Queries>
__device__ __forceinline__ WalkEnd walk_segment(WarpSmem<FMT>& ws, const uint4 (*qlo)[32], const Segment& sg, int lane,
                                                Queries queries) {
  using SL = Slot<FMT>;
  const int g = lane >> 2, t = lane & 3;
  // windows counted from `base`: with MXFP4 metadata a batch starts on an even window, because two windows' metadata
  // share one aligned block
  const int base = FMT == FMT_MXFP4 ? sg.w0 & ~1 : sg.w0;
  const int k_first = sg.w0 - base, k_end = k_first + sg.n_my;
  unsigned char* const slots = &ws.slot[0][0];

  // a window's record is SL::BYTES / 16 chunks: lane l copies chunks l, l + 32, ...
  constexpr int FULL = SL::BYTES / 512, REST = SL::BYTES / 16 - 32 * FULL;
  const unsigned char* src = sg.rec0 + (FMT == FMT_FP16 ? (size_t)sg.w0 * RECORD_BYTES + OFF_KS : mx_body_off(sg.w0)) + 16 * lane;
  int i_slot = 0, odd = k_first;   // offset of the slot of the next window to be copied; MXFP4: second window of its block
  auto issue = [&](int k) {
    if (k < k_end) {
      unsigned char* dst = slots + i_slot + 16 * lane;
#pragma unroll
      for (int i = 0; i < FULL; i++) cp_async16(dst + 512 * i, src + 512 * i);
      if (lane < REST) cp_async16(dst + 512 * FULL, src + 512 * FULL);
      src += FMT == FMT_FP16 ? RECORD_BYTES : (odd ? MX_PAIR_BYTES - BODY_BYTES : BODY_BYTES);
      if (FMT == FMT_MXFP4) odd ^= 1;
      i_slot = i_slot == (NSLOT - 1) * SL::BYTES ? 0 : i_slot + SL::BYTES;
    }
  };
  auto issue_batch = [&](int k0) {   // metadata and modality bytes of the batch that starts at window k0
    if (k0 >= k_end) return;
    const unsigned char* rec = sg.rec0;
    if (FMT == FMT_FP16) {           // the m planes: half a warp per window
      const unsigned char* p = rec + (size_t)(base + k0 + (lane >> 4)) * RECORD_BYTES + OFF_KM + 16 * (lane & 15);
#pragma unroll
      for (int i = 0; i < BATCH / 2; i++)
        if (k0 + 2 * i + (lane >> 4) < k_end)
          cp_async16(&ws.m[(2 * i + (lane >> 4)) * M_PITCH + 16 * (lane & 15)], p + (size_t)i * 2 * RECORD_BYTES);
    } else {                         // the blocks' metadata, 17 chunks each
      constexpr int CH = MX_BLOCK_META / 16;
      for (int c = lane; c < (BATCH / 2) * CH; c += 32) {
        const int blk = c / CH;
        if (k0 + 2 * blk < k_end)
          cp_async16(&ws.mx[16 * c], rec + (size_t)(((base + k0) >> 1) + blk) * MX_PAIR_BYTES + 16 * (c - blk * CH));
      }
    }
    if (lane < 2 * BATCH && k0 + (lane >> 1) < k_end)   // half a lane pair per window
      cp_async16(&ws.mod[(k0 / BATCH) & 1][16 * lane], sg.mod0 + (size_t)(base + k0) * W + 16 * lane);
  };
  __syncwarp();   // everyone is done with the previous segment's slots
  issue_batch(0);
#pragma unroll
  for (int i = 0; i < PREFETCH - 1; i++) { issue(k_first + i); cp_async_commit(); }

  uint32_t qh[16];
  float fsc;
  queries(qh, fsc);
  const F2 fsc2 = f2(fsc, fsc);

  float acc[8][4];
#pragma unroll
  for (int mu = 0; mu < 8; mu++)
#pragma unroll
    for (int i = 0; i < 4; i++) acc[mu][i] = 0.f;
  F2 run_l = f2(0.f, 0.f);
  F2 noff = f2(INFINITY, INFINITY);           // minus the reference: the first window exceeds every limit
  auto run_m = [&]() { return -un2(noff).x; };
  int cur_mod = -1, since = 0, streak = 0;
  unsigned held = 0;                          // modalities the piece already holds something of

  auto piece_row = [&](int m) { return &sg.piece->frag[m][0][lane]; };
  // adds four-register rows to the piece (the first ones of a modality are stored), brought to its reference
  auto put = [&](int m, const float (*o)[4], int mu0, int n) {
    const float f = ex2(run_m() - ws.rebase[lane]);
    const float f_lo = __shfl_sync(0xffffffffu, f, 8 * t), f_hi = __shfl_sync(0xffffffffu, f, 8 * t + 4);
    float4* dst = piece_row(m) + 32 * mu0;
#pragma unroll
    for (int i = 0; i < n; i++) {
      const float4 v = make_float4(o[i][0] * f_lo, o[i][1] * f_hi, o[i][2] * f_lo, o[i][3] * f_hi);
      if ((held >> m) & 1u) red_add(dst + 32 * i, v);
      else __stcg(dst + 32 * i, v);
    }
  };
  // The tensor cores' fp32 accumulation does not round to nearest, so a long chain of products into one register drifts
  // one-sidedly; short chains added up with rounded additions do not.
  auto deposit = [&]() {
    put(cur_mod, acc, 0, 8);
    held |= 1u << cur_mod;
#pragma unroll
    for (int mu = 0; mu < 8; mu++)
#pragma unroll
      for (int i = 0; i < 4; i++) acc[mu][i] = 0.f;
    since = 0;
  };

  // window k has landed and may be read by every lane: the next copies, and the bias sums if a batch starts with it
  auto arrive = [&](int k) {
    cp_async_wait<PREFETCH - 2>();   // this lane's copies of window k (and of its batch) have landed,
    __syncwarp();                    // everyone's have, and everyone is done with window k - 2
    issue(k + PREFETCH - 1);
    if ((k & (BATCH - 3)) == 0 && (k & 2)) issue_batch((k & ~(BATCH - 1)) + BATCH);   // this batch's planes were read two windows ago
    cp_async_commit();
    if ((k & (BATCH - 1)) == 0 || k == k_first) {
      if (FMT == FMT_MXFP4) {
        for (int i = 0; i < BATCH; i++) {
          uint2 m4, s4;
          mx_decode_lane(&ws.mx[i * MX_META_BYTES], lane, m4, s4);
          *reinterpret_cast<uint2*>(&ws.m[i * M_PITCH + 8 * lane]) = m4;
          *reinterpret_cast<uint2*>(&ws.s[i * 256 + 8 * lane]) = s4;
        }
        __syncwarp();
      }
      const uint4* mp = reinterpret_cast<const uint4*>(&ws.m[g * M_PITCH + 64 * t]);
      float dbA[4], dbB[4];
#pragma unroll
      for (int kq = 0; kq < 4; kq++) {
        const uint4 m4 = mp[kq], ql = qlo[kq][lane];
        if (kq == 0) {
          mma16816_first(dbA, qh[0], ql.x, qh[1], ql.y, m4.x, m4.y);
          mma16816_first(dbB, qh[2], ql.z, qh[3], ql.w, m4.z, m4.w);
        } else {
          mma16816(dbA, qh[4 * kq], ql.x, qh[4 * kq + 1], ql.y, m4.x, m4.y);
          mma16816(dbB, qh[4 * kq + 2], ql.z, qh[4 * kq + 3], ql.w, m4.z, m4.w);
        }
      }
      // the code sums carry 2^-24 (subnormal code operands), the bias does not
      ws.bias[2 * t][g] = ((dbA[0] + dbB[0]) + (dbA[2] + dbB[2])) * 0x1p-24f;
      ws.bias[2 * t + 1][g] = ((dbA[1] + dbB[1]) + (dbA[3] + dbB[3])) * 0x1p-24f;
      __syncwarp();
    }
  };

  // ---- score products of one window, k-step (16 channels) kappa: d[nu] = head g (hi, lo rows), tokens 8 nu + 2 t + e
  uint32_t kw[4][2];
  uint4 s4, ql4;
  float d[4][4];
  auto score_load = [&](const unsigned char* st) {
    const uint4 kc0 = *reinterpret_cast<const uint4*>(st + SL::BODY + B_KCODE + 16 * kpiece_slot(lane));
    const uint4 kc1 = *reinterpret_cast<const uint4*>(st + SL::BODY + B_KCODE + 16 * kpiece_slot(32 + lane));
    kw[0][0] = kc0.x; kw[0][1] = kc0.y; kw[1][0] = kc0.z; kw[1][1] = kc0.w;
    kw[2][0] = kc1.x; kw[2][1] = kc1.y; kw[3][0] = kc1.z; kw[3][1] = kc1.w;
  };
  auto score_step = [&](const unsigned char* sp, int kappa, auto mid) {
    const int half = kappa & 1;
    if (!half) { s4 = reinterpret_cast<const uint4*>(sp)[kappa >> 1]; ql4 = qlo[kappa >> 1][lane]; }
    uint32_t a0, a1, a2, a3;
    split_product(u2h(qh[2 * kappa]), u2h(half ? ql4.z : ql4.x), u2h(half ? s4.z : s4.x), a0, a1);
    split_product(u2h(qh[2 * kappa + 1]), u2h(half ? ql4.w : ql4.y), u2h(half ? s4.w : s4.y), a2, a3);
    const int ww = kappa >> 2, sh = (kappa >> 1) & 1;
    const uint32_t mk0 = half ? 0x00300030u : 0x00030003u;
    const uint32_t mk1 = half ? 0x00c000c0u : 0x000c000cu;
#pragma unroll
    for (int nu = 0; nu < 4; nu++) {
      const uint32_t src = sh ? (kw[nu][ww] >> 8) : kw[nu][ww];
      if (kappa == 0) mma16816_first(d[nu], a0, a1, a2, a3, src & mk0, src & mk1);
      else mma16816(d[nu], a0, a1, a2, a3, src & mk0, src & mk1);
      if (nu & 1) mid(nu >> 1);
    }
  };
  // ---- value products: the 16 x 32 code block of word w as level operands, fields (0, 2) for jp = 0, (1, 3) for jp = 1,
  // token parity e = 0, 1
  auto levels = [&](uint32_t w, int jp, uint32_t (&a)[4]) {
    const uint32_t sel = (jp ? w >> 2 : w) & 0x33333333u;
    const uint32_t x0 = prmt(LEVEL_HI, LEVEL_HI, sel), x1 = prmt(LEVEL_HI, LEVEL_HI, sel >> 16);
    a[0] = prmt(x0, LEVEL_LO, 0x1404u); a[1] = prmt(x0, LEVEL_LO, 0x3424u);
    a[2] = prmt(x1, LEVEL_LO, 0x1404u); a[3] = prmt(x1, LEVEL_LO, 0x3424u);
  };

  // ---- online softmax (log2 domain): scores of the window staged at `st` from its products, then its numerators in fp16
  // (operand pairs of tokens nu and nu + 2, parity e, for the value product) and the sum of their p; true if this lane's
  // exceed what the reference allows
  auto scores = [&](const unsigned char* st, float bias, F2 (&sc)[4]) {
    const uint4 kn4 = *reinterpret_cast<const uint4*>(st + SL::BODY + B_KNORM + 16 * t);
    const uint32_t knu[4] = {kn4.x, kn4.y, kn4.z, kn4.w};
    const F2 bb = f2(bias, bias);
#pragma unroll
    for (int nu = 0; nu < 4; nu++)
      sc[nu] = mul2(add2(add2(f2(d[nu][0], d[nu][1]), f2(d[nu][2], d[nu][3])), bb), half2_to_f2(knu[nu]));
  };
  auto numerators = [&](const unsigned char* st, const F2 (&sc)[4], uint32_t (&pb)[2][2], F2& ps) {
    const uint4 vn4 = *reinterpret_cast<const uint4*>(st + SL::BODY + B_VNORM + 16 * t);
    const uint32_t vnu[4] = {vn4.x, vn4.y, vn4.z, vn4.w};
    float2 pn[4];
    float mx = 0.f;
#pragma unroll
    for (int nu = 0; nu < 4; nu++) {
      const float2 x = un2(fma2(sc[nu], fsc2, noff));
      const F2 p = f2(ex2(x.x), ex2(x.y));
      ps = nu == 0 ? p : add2(ps, p);
      pn[nu] = un2(mul2(p, half2_to_f2(vnu[nu])));
      mx = fmaxf(mx, fmaxf(pn[nu].x, pn[nu].y));
    }
#pragma unroll
    for (int jp = 0; jp < 2; jp++) {
      pb[jp][0] = pack_sat(pn[jp].x, pn[jp + 2].x);
      pb[jp][1] = pack_sat(pn[jp].y, pn[jp + 2].y);
    }
    const float2 s2 = un2(ps);
    return mx > NUM_MAX || s2.x > SUM_MAX || s2.y > SUM_MAX;
  };
  // The reference moves for every head, to where the window's largest numerator has its place.  That one is found by
  // score + log2(vnorm), the logarithm taken as the straight line between powers of two: biased exponent and mantissa, read as
  // one number (a zero norm counts as 2^-127).
  auto move = [&](const unsigned char* st, const F2 (&sc)[4], bool first) {
    const uint4 vn4 = *reinterpret_cast<const uint4*>(st + SL::BODY + B_VNORM + 16 * t);
    const uint32_t vnu[4] = {vn4.x, vn4.y, vn4.z, vn4.w};
    float top = -INFINITY, top_u = 0.f, hi = -INFINITY;
    uint32_t top_v = 0;
#pragma unroll
    for (int nu = 0; nu < 4; nu++) {
      const float2 s = un2(mul2(sc[nu], fsc2)), v = un2(half2_to_f2(vnu[nu]));
#pragma unroll
      for (int e = 0; e < 2; e++) {
        const float u = e ? s.y : s.x;
        const uint32_t vb = __float_as_uint(e ? v.y : v.x);
        const float lg = fmaf(__uint_as_float(0x4B000000u | (vb >> 9)), 0x1p-14f, u - 639.0f);   // 2^23 + 2^14 (exponent + mantissa)
        hi = fmaxf(hi, u);
        if (lg > top) { top = lg; top_u = u; top_v = vb; }
      }
    }
    float ref = top_u + (float)((int)(top_v >> 23) - 127 - TOP_LOG2);
#pragma unroll
    for (int dl = 1; dl < 4; dl <<= 1) {   // over the head's four lanes, of equals the higher reference
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, dl));
      const float ot = __shfl_xor_sync(0xffffffffu, top, dl), oref = __shfl_xor_sync(0xffffffffu, ref, dl);
      if (ot > top || (ot == top && oref > ref)) { top = ot; ref = oref; }
    }
    const float m_new = fmaxf(fmaxf(ref, hi - P_LOG2_MAX), run_m());
    if (first) ws.rebase[lane] = m_new;
    const float alpha = ex2(run_m() - m_new);     // 0 on the first window
    noff = f2(-m_new, -m_new);
    run_l = mul2(run_l, f2(alpha, alpha));
    const float a_lo = __shfl_sync(0xffffffffu, alpha, 8 * t), a_hi = __shfl_sync(0xffffffffu, alpha, 8 * t + 4);
#pragma unroll
    for (int mu = 0; mu < 8; mu++) { acc[mu][0] *= a_lo; acc[mu][1] *= a_hi; acc[mu][2] *= a_lo; acc[mu][3] *= a_hi; }
    const float piece_m = ws.rebase[lane];
    if (__any_sync(0xffffffffu, m_new - piece_m > REBASE_LOG2)) {   // the piece follows before its numbers could overflow
      const float f = ex2(piece_m - m_new);
      const float f_lo = __shfl_sync(0xffffffffu, f, 8 * t), f_hi = __shfl_sync(0xffffffffu, f, 8 * t + 4);
      ws.rebase[lane] = m_new;
#pragma unroll 1
      for (int m = 0; m < 3; m++)
        if ((held >> m) & 1u)
#pragma unroll 1
          for (int mu = 0; mu < 8; mu++) {
            float4* p = piece_row(m) + 32 * mu;
            const float4 v = __ldcg(p);
            __stcg(p, make_float4(v.x * f_lo, v.y * f_hi, v.z * f_lo, v.w * f_hi));
          }
    }
  };

  const unsigned char* st = slots;                     // slot of window k
  const unsigned char* stn = slots;                    // slot of window k + 1
  auto s_plane = [&](int k) {
    return FMT == FMT_FP16 ? stn + 64 * t : (const unsigned char*)&ws.s[(k & (BATCH - 1)) * 256 + 64 * t];
  };
  arrive(k_first);
  float bias = ws.bias[k_first][g];
  score_load(stn);
#pragma unroll
  for (int kappa = 0; kappa < 8; kappa++) score_step(s_plane(k_first), kappa, [](int) {});

  for (int k = k_first; k < k_end; k++) {
    st = stn;
    // (the numerators' check is part of the test for the common case below)
    uint32_t pb[2][2];
    F2 ps;
    const float bias_k = bias;
    bool over;
    {
      F2 sc[4];
      scores(st, bias_k, sc);
      over = numerators(st, sc, pb, ps);
    }
    const int mymod = ws.mod[(k / BATCH) & 1][(k & (BATCH - 1)) * W + lane];
    const uint4 vc0 = *reinterpret_cast<const uint4*>(st + SL::BODY + B_VCODE + 16 * vpiece_slot(lane));
    const uint4 vc1 = *reinterpret_cast<const uint4*>(st + SL::BODY + B_VCODE + 16 * vpiece_slot(32 + lane));
    const uint32_t vw[8] = {vc0.x, vc0.y, vc0.z, vc0.w, vc1.x, vc1.y, vc1.z, vc1.w};

    // ---- window k + 1 (behind the last window: products of a stale slot, never used)
    stn = st == slots + (NSLOT - 1) * SL::BYTES ? slots : st + SL::BYTES;
    arrive(k + 1);
    bias = ws.bias[(k + 1) & (BATCH - 1)][g];
    score_load(stn);
    const unsigned char* sp = s_plane(k + 1);

    unsigned mine = __ballot_sync(0xffffffffu, mymod == cur_mod && !over);
    if (mine != 0xffffffffu) {
      if (__any_sync(0xffffffffu, over)) {   // the reference moves and the numerators are taken again
        F2 sc[4];
        scores(st, bias_k, sc);
        move(st, sc, k == k_first);
        numerators(st, sc, pb, ps);
        mine = __ballot_sync(0xffffffffu, mymod == cur_mod);
      }
    }
    run_l = add2(run_l, ps);
    if (mine != 0xffffffffu) {
      const int first = __shfl_sync(0xffffffffu, mymod, 0);
      const bool pure = __all_sync(0xffffffffu, mymod == first);
      streak = pure ? streak + 1 : 0;
      if (cur_mod < 0 || (pure && streak >= SWITCH_AFTER)) {   // the registers change over to another modality
        if (cur_mod >= 0 && since > 0) deposit();
        cur_mod = first;
        mine = __ballot_sync(0xffffffffu, mymod == cur_mod);
      }
    }
    if (mine == 0xffffffffu) {
      // the common case, every token of the modality the registers hold: the value products of window k and the score
      // products of window k + 1 in one stretch, each filling the other's waits
      streak = 0;
#pragma unroll
      for (int kappa = 0; kappa < 8; kappa++)
        score_step(sp, kappa, [&](int jp) {
          uint32_t a[4];
          levels(vw[kappa], jp, a);
          mma16816(acc[kappa], a[0], a[1], a[2], a[3], pb[jp][0], pb[jp][1]);
        });
      if (++since >= FLUSH) deposit();
    } else {
      // visitors: tokens of another modality, their products go straight to the piece
      uint32_t pm[2][2];
#pragma unroll
      for (int jp = 0; jp < 2; jp++)
#pragma unroll
        for (int e = 0; e < 2; e++) pm[jp][e] = pb[jp][e] & (((mine >> (8 * jp + 2 * t + e)) & 0x00010001u) * 0xffffu);
#pragma unroll 1
      for (int m = 0; m < 3; m++) {
        const unsigned sel = __ballot_sync(0xffffffffu, mymod == m);
        if (m == cur_mod || sel == 0) continue;
        uint32_t pv[2][2];
#pragma unroll
        for (int jp = 0; jp < 2; jp++)
#pragma unroll
          for (int e = 0; e < 2; e++) pv[jp][e] = pb[jp][e] & (((sel >> (8 * jp + 2 * t + e)) & 0x00010001u) * 0xffffu);
#pragma unroll
        for (int mq = 0; mq < 8; mq += 4) {
          float o[4][4];
#pragma unroll
          for (int jp = 0; jp < 2; jp++)
#pragma unroll
            for (int i = 0; i < 4; i++) {
              uint32_t a[4];
              levels(vw[mq + i], jp, a);
              mma16816(acc[mq + i], a[0], a[1], a[2], a[3], pm[jp][0], pm[jp][1]);
              if (jp == 0) mma16816_first(o[i], a[0], a[1], a[2], a[3], pv[jp][0], pv[jp][1]);
              else mma16816(o[i], a[0], a[1], a[2], a[3], pv[jp][0], pv[jp][1]);
            }
          put(m, o, mq, 4);
        }
        held |= 1u << m;
        pm[0][0] = pm[0][1] = pm[1][0] = pm[1][1] = 0;   // a second visitor: the registers have had their share
      }
      if (mine != 0) since++;
#pragma unroll
      for (int kappa = 0; kappa < 8; kappa++) score_step(sp, kappa, [](int) {});
      if (since >= FLUSH) deposit();
    }
  }
  cp_async_wait<0>();
  if (since > 0) deposit();
  const float2 l2 = un2(run_l);
  const float piece_m = ws.rebase[lane];
  float l = (l2.x + l2.y) * ex2(run_m() - piece_m);
  l += __shfl_xor_sync(0xffffffffu, l, 1);
  l += __shfl_xor_sync(0xffffffffu, l, 2);
  return WalkEnd{piece_m, l, held};
}

}  // namespace

}  // namespace okq
