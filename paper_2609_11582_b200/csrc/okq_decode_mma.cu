// Fused decode attention, tensor-core version (the production path of okq_decode_attention).
//
// The GQA group's scores and value sums are dense contractions over the cached tokens
//     S^T[head][token]   = W[head][channel] * C_k[channel][token]        (per 32-token window)
//     O^T[channel][head] = C_v[channel][token] * P[token][head]
// and run on mma.sync.m16n8k16 with the 2-bit codes unpacked in registers:
//   * a key-code field masked out of its 32-bit word *is* an fp16 subnormal (code * 4^j * 2^-24,
//     j the field's position), so unpacking is one AND per two codes; the factor 4^j is folded
//     into the query weights;
//   * W = q'_c * s_gc is split into an fp16 high and low part, which fill the 16 rows of the
//     m16 tile (8 heads x {hi, lo}), so the split costs no extra tensor work;
//   * the bias sum_c q'_c m_gc of eight consecutive windows comes out of one set of eight products,
//     the windows' m planes being the eight columns of the B operand (one window at a time the same
//     products would have eight equal columns);
//   * value codes become fp16 codebook levels by byte permutes: four codes are four nibbles of a
//     selector, one look-up gives the high bytes of their levels, and two permutes put the common low
//     byte under them.  One product per 16 x 16 codes then replaces two bit-plane products.
// A warp does all of a window by itself: scores, online softmax (FlashAttention order), value sums.
// The score tile's accumulator layout is the value product's operand layout, so the numerators
// never leave their lane.  Records arrive through a cp.async ring, PREFETCH windows ahead (bulk copies were measured too:
// each costs the warp about 15 instructions to hand over, against 5 copies of 512 bytes with immediate offsets).
// A warp's registers hold the value sums of one modality in its rotated basis; tokens of another
// modality inside its range are "visitors", whose products are added straight to the warp's piece
// in global memory (vector reductions), as are the registers every FLUSH windows.
// What bounds it: dispatch slots.  Per window a warp issues about 650 instructions (53 of them products); LOP3, PRMT,
// IMAD and HFMA2 take two dispatch cycles of an SM sub-partition each, a product 8.6 by itself and about 10 with the
// masks that feed it, so more warps do not help: 12 per CTA with 168 registers each is where the accumulators, both
// operand sets and the next window's scores fit without spills.  step7b (28 layers x 8 x 16384 tokens, 1.233 GB of
// records), whole call: 570 us with a score and a value warp per window pair and two bit-plane products per 16 x 16
// codes, 517 us in this form.  Two windows per turn (8 warps, 233 registers) measured 541 us, an unrolled pair of turns
// 594 us (the loop outgrows the instruction cache).
// The grid is persistent: CTA i owns an equal slice of the flattened (layer, sequence, head,
// window) axis, each of its warps an equal part of that slice, which the warp walks without any
// block-wide step; at the end the block merges its warps' pieces into one partial per
// (sequence, head) it touched.  The combine kernel merges the partials, adds the raw fp16 tail
// tokens, applies R_m^T once per head and normalises.
#include "okq_decode_walk.cuh"

namespace okq {

namespace {

template <int FMT> struct MmaSmem {
  WarpSmem<FMT> w[NWARP];
  __align__(16) uint4 qlo[NWARP][4][32];   // low parts of a warp's query fragments
  int prefix[MAX_ENTRIES + 1];
};

constexpr int MB_SEG = 32;                      // (sequence, head) units merged per batch at the end of the launch
struct MergeSmem {
  int pa[MB_SEG], pb[MB_SEG];                   // first and last warp that worked on the unit (pb < pa: none)
  float meta[MB_SEG + NWARP][2 * GP];           // per piece: wm[GP], wl[GP]; index = unit + warp - pa[0]
  int mask[MB_SEG + NWARP];                     // per piece: modalities it holds
  float fac[MB_SEG + NWARP][GP];                // per piece and head: exp2(wm - merged maximum)
};

}  // namespace

// grid = n_cta (persistent), NTHREADS threads
//
// CTA i owns the windows [i * per, (i + 1) * per) of the flattened (layer, sequence, head, window) axis and
// cuts them into NWARP contiguous ranges.  A warp walks its range on its own, with no block-wide step in
// between: where the range crosses into another (sequence, head) it leaves what it accumulated in a piece and
// starts afresh.  At the end of the launch the block merges, per (sequence, head) it touched, the pieces of
// the warps that worked on it into one PartialF.
template <int FMT>
__global__ void __launch_bounds__(NTHREADS, 1) k_decode_mma(DecodeParams P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MmaSmem<FMT>& sm = *reinterpret_cast<MmaSmem<FMT>*>(smem_raw);
  const CacheView& cv = P.cv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = P.group, Hkv = cv.n_kv_heads;
  const int n_entries = P.layer_count * cv.batch;

  depend_wait();
  // ---- partition of the flattened window axis
  const int total = block_prefix(cv, P.layer0, n_entries, sm.prefix);
  const int per = (total + gridDim.x - 1) / gridDim.x;
  const int pos0 = min(total, (int)blockIdx.x * per), pos1 = min(total, pos0 + per);
  const int cnt = (pos1 - pos0 + NWARP - 1) / NWARP;

  struct Where { int e, h, w0, nwin; };
  auto locate = [&](int pos) {   // (entry, head, window) of a flattened position; largest e with prefix[e] <= pos
    int lo = 0, hi = n_entries;
    while (hi - lo > 1) {
      int mid = (lo + hi) >> 1;
      if (sm.prefix[mid] <= pos) lo = mid; else hi = mid;
    }
    Where wh;
    wh.e = lo;
    wh.nwin = (sm.prefix[lo + 1] - sm.prefix[lo]) / Hkv;
    const int off = pos - sm.prefix[lo];
    wh.h = off / wh.nwin;
    wh.w0 = off % wh.nwin;
    return wh;
  };

  {
    int pos = min(pos1, pos0 + warp * cnt);
    const int pos_end = min(pos1, pos + cnt);
    while (pos < pos_end) {
      const Where wh = locate(pos);
      const int li = wh.e / cv.batch, b = wh.e % cv.batch;
      Segment sg;
      sg.rec0 = cv.unit(P.layer0 + li, b, wh.h);
      sg.mod0 = cv.modality + (size_t)b * cv.capacity;
      sg.w0 = wh.w0;
      sg.n_my = min(pos_end - pos, wh.nwin - wh.w0);
      sg.piece = P.pieces + (size_t)(wh.e * Hkv + wh.h) + ((size_t)blockIdx.x * NWARP + warp);
      const WalkEnd we = walk_segment<FMT>(sm.w[warp], sm.qlo[warp], sg, lane, [&](uint32_t (&qh)[16], float& fsc) {
        uint2 qreg[16];
        query_fragments(P.q + (((size_t)li * cv.batch + b) * cv.n_q_heads + (size_t)wh.h * G) * D, P.signs + (size_t)li * D, G,
                        P.sm_scale, lane, qreg, fsc);
#pragma unroll
        for (int r = 0; r < 16; r++) qh[r] = qreg[r].x;
#pragma unroll
        for (int kq = 0; kq < 4; kq++)   // (a lane reads back only what it wrote)
          sm.qlo[warp][kq][lane] = make_uint4(qreg[4 * kq].y, qreg[4 * kq + 1].y, qreg[4 * kq + 2].y, qreg[4 * kq + 3].y);
      });
      if ((lane & 3) == 0) { sg.piece->wm[lane >> 2] = we.m; sg.piece->wl[lane >> 2] = we.l; }
      if (lane == 0) sg.piece->mask = (int)we.held;
      pos += sg.n_my;
    }
  }
  __syncthreads();   // the pieces were written by this block's own warps: visible to the block from here on

  // ---- merge the warps' pieces into one partial per (sequence, head) of the block's range, MB_SEG
  // (sequence, head) units at a time so that the loads of many units are in flight together.  The tables
  // take the place of the record ring, which is idle by now.
  if (pos0 >= pos1) return;
  MergeSmem& mg = *reinterpret_cast<MergeSmem*>(smem_raw);
  static_assert(sizeof(MergeSmem) <= sizeof(WarpSmem<FMT>) * NWARP, "the merge tables fit the record ring");
  const Where wf = locate(pos0), wl = locate(pos1 - 1);
  const int u_first = wf.e * Hkv + wf.h, u_last = wl.e * Hkv + wl.h;
  for (int ub = u_first; ub <= u_last; ub += MB_SEG) {
    const int n_u = min(MB_SEG, u_last - ub + 1);
    // (a) the units' window ranges inside the block's slice and the warps that worked on them
    if (tid < n_u) {
      const int u = ub + tid, e = u / Hkv, h = u % Hkv;
      const int nwin = (sm.prefix[e + 1] - sm.prefix[e]) / Hkv;
      const int a0 = max(pos0, sm.prefix[e] + h * nwin), a1 = min(pos1, sm.prefix[e] + (h + 1) * nwin);
      mg.pa[tid] = a1 > a0 ? (a0 - pos0) / cnt : 0;
      mg.pb[tid] = a1 > a0 ? (a1 - 1 - pos0) / cnt : -1;   // empty: a (sequence, head) with no packed window
    }
    __syncthreads();
    // (b) the pieces' maxima and weight sums: a half-warp per (unit, warp)
    for (int j = tid >> 4; j < n_u * NWARP; j += NTHREADS / 16) {
      const int su = j / NWARP, p = j % NWARP, c = tid & 15;
      if (p < mg.pa[su] || p > mg.pb[su]) continue;
      const WarpPiece& pp = P.pieces[(size_t)(ub + su) + (size_t)blockIdx.x * NWARP + p];
      mg.meta[su + p - mg.pa[0]][c] = pp.wm[c];             // wm[GP], then wl[GP]
      if (c == 0) mg.mask[su + p - mg.pa[0]] = pp.mask;
    }
    __syncthreads();
    // (c) merged maximum, weight sum and the pieces' factors per (unit, head)
    if (tid < n_u * GP) {
      const int su = tid / GP, j = tid % GP;
      if (mg.pb[su] >= mg.pa[su]) {
        float mj = -INFINITY, L = 0.f;
        for (int p = mg.pa[su]; p <= mg.pb[su]; p++) mj = fmaxf(mj, mg.meta[su + p - mg.pa[0]][j]);
        for (int p = mg.pa[su]; p <= mg.pb[su]; p++) {
          const float f = exp2f(mg.meta[su + p - mg.pa[0]][j] - mj);
          L += mg.meta[su + p - mg.pa[0]][GP + j] * f;
          mg.fac[su + p - mg.pa[0]][j] = f;
        }
        PartialF* out = P.partials_f + (size_t)(ub + su) + blockIdx.x;
        out->m[j] = mj;
        out->l[j] = L;
      }
    }
    __syncthreads();
    // (d) the accumulators: one item = four consecutive registers of one lane of one (unit, modality); registers r and
    // r + 2 belong to head 2 (lane & 3), r + 1 and r + 3 to the next head
    constexpr int RG = 8, UNIT_ITEMS = 3 * RG * 32;
    for (int it = tid; it < n_u * UNIT_ITEMS; it += NTHREADS) {
      const int su = it / UNIT_ITEMS, idx = it % UNIT_ITEMS;
      const int L = idx & 31, rg = (idx >> 5) % RG, m = idx / (RG * 32);
      const int pa = mg.pa[su], np = mg.pb[su] - pa + 1;
      if (np <= 0) continue;
      const int inc0 = su + pa - mg.pa[0], hsel = 2 * (L & 3);
      // all the pieces' rows on their way together (they come from L2: one after another they were a third of a call with
      // few windows per warp)
      float4 x[NWARP];
#pragma unroll
      for (int q = 0; q < NWARP; q++) {
        x[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q < np && ((mg.mask[inc0 + (q < np ? q : 0)] >> m) & 1))   // (else: no such warp / no token of this modality)
          x[q] = __ldcg(&P.pieces[(size_t)(ub + su) + (size_t)blockIdx.x * NWARP + pa + q].frag[m][rg][L]);
      }
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int q = 0; q < NWARP; q++) {
        const float2 f = *reinterpret_cast<const float2*>(&mg.fac[inc0 + (q < np ? q : 0)][hsel]);
        v.x = fmaf(x[q].x, f.x, v.x); v.y = fmaf(x[q].y, f.y, v.y); v.z = fmaf(x[q].z, f.x, v.z); v.w = fmaf(x[q].w, f.y, v.w);
      }
      // in units of the bit-plane form, whose weight sums are zero here
      constexpr float F = LEVEL_UNIT / PARTIAL_ACC_SCALE;
      PartialF* out = P.partials_f + (size_t)(ub + su) + blockIdx.x;
      out->frag[m][4 * rg][L] = v.x * F; out->frag[m][4 * rg + 1][L] = v.y * F;
      out->frag[m][4 * rg + 2][L] = v.z * F; out->frag[m][4 * rg + 3][L] = v.w * F;
      if (rg == 0) out->Sp[m][L] = 0.f;
    }
    __syncthreads();
  }
}

constexpr int PARTIAL_HDR_FLOATS = 2 * GP + 3 * 32;   // m[GP], l[GP], Sp[3][32] at the start of a PartialF
constexpr int CB_SEQ_MAX = 4;             // most sequences per combine CTA (one 128-thread group each)

constexpr int MRG_MAX = 8;                // partials per (sequence, head) whose factors are precomputed
constexpr int CB_CHUNK = 16;              // rows of a rotation matrix staged per step
constexpr int CB_NBUF = 4;                // staged slices in flight (three ahead of the one in use)

// the bf16 terms of two numbers, largest first: x = sum of the low halves, y = sum of the high halves, to 24 bits
__device__ __forceinline__ void bf16_terms(float x, float y, uint32_t (&tm)[3]) {
#pragma unroll
  for (int i = 0; i < 3; i++) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;\n" : "=r"(tm[i]) : "f"(y), "f"(x));
    x -= __uint_as_float(tm[i] << 16);
    y -= __uint_as_float(tm[i] & 0xffff0000u);
  }
}
__device__ __forceinline__ void mma16816_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// CAPTION: the captioning schedule keeps up to 159 raw values (and up to 127 raw keys) per sequence, and
// the keys of the raw values' tokens may already be packed
// SEQ: sequences per CTA, one or four (combine_form below)
template <bool CAPTION, int SEQ>
struct CombineSmem {
  static constexpr int CB_SEQ = SEQ, CB_ROWS = SEQ * GP;
  static constexpr int TAIL = CAPTION ? CAPTION_V_SLOTS : W;   // most raw-value tokens of a sequence
  static constexpr bool SPLIT = SEQ == CB_SEQ_MAX;   // the product with R_m^T on the tensor cores, from three bf16 terms
  // one sequence per block: ring of 16-row slices of the rotation matrices, large enough for a quarter of the columns of all
  // three matrices, which the four-slice configuration fetches whole at the start
  __align__(16) float Rbuf[SPLIT ? 4 : 3 * D * (D / 4)];
  // per partial and head: rescale factor, weight sums of the modalities (one-sequence blocks have room for the
  // partials of a long single sequence, which is spread over many CTAs of the split-K kernel)
  static constexpr int MRG_TAB = SEQ == 1 ? 64 : MRG_MAX;
  __align__(16) float mrg[CB_SEQ][MRG_TAB][GP][4];
  __align__(16) float vec[SPLIT ? 1 : 3][SPLIT ? 1 : CB_ROWS][D];   // merged rotated-basis sums, [modality][row][rotated channel]
  // or their terms, [term][row][modality * 128 + rotated channel]: rows of 784 bytes, an odd number of 16-byte columns
  static constexpr int XP = 3 * D + 8, OUT_PITCH = D + 4;
  __align__(16) unsigned short xs[SPLIT ? 3 : 1][SPLIT ? CB_ROWS : 1][XP];
  static_assert(!SPLIT || 2 * CB_ROWS * OUT_PITCH * 4 <= (int)sizeof(xs), "the products of the two halves take the terms' place");
  __align__(16) float rawv[CB_ROWS][D];       // raw-tail contribution, [row][channel]
  // tail scores (log2 domain), then softmax numerators, [sequence][token][head]: blocks of several sequences keep
  // them behind the tail scratch, where the terms of the rotated sums are written later
  __align__(16) float tsc_own[SPLIT ? 4 : CB_SEQ * TAIL * GP];
  float Ms[CB_SEQ][GP], Ls[CB_SEQ][GP];
  float red[CB_SEQ][4][GP];   // per warp of a sequence: partial maxima / sums of the softmax bookkeeping
  // one-sequence blocks: the headers (m, l, weight sums) of the sequence's first MRG_TAB partials, fetched early
  __align__(16) float hdr[SEQ == 1 ? MRG_TAB * PARTIAL_HDR_FLOATS : 4];
  __align__(16) __half vsm[SEQ == 1 ? TAIL * D : 8];   // one-sequence blocks: the raw value rows, fetched early
  int prefix[MAX_ENTRIES + 1];
};

// NS: CTAs that share one (head, sequence group): each computes D / NS output columns (used when the grid
// would otherwise leave most SMs idle; the merge is repeated by every slice, the matrix streaming is split)
template <bool CAPTION, int NS, int SEQ>
__global__ void __launch_bounds__(SEQ * 128, SEQ == CB_SEQ_MAX ? 2 : 1) k_combine_mma(DecodeParams P, int n_cta) {
  constexpr int CB_SEQ = SEQ, CB_ROWS = SEQ * GP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CombineSmem<CAPTION, SEQ>& sm = *reinterpret_cast<CombineSmem<CAPTION, SEQ>*>(smem_raw);
  constexpr bool SPLIT = CombineSmem<CAPTION, SEQ>::SPLIT;
  constexpr int KROW = D + 8;                              // halfs per staged key row
  constexpr int KSM_FLOATS = W * KROW / 2, QSM_FLOATS = GP * D / 2;
  float* const scratch = SPLIT ? reinterpret_cast<float*>(&sm.xs[0][0][0]) : &sm.vec[0][0][0];
  float* const tsc_base = SPLIT ? scratch + CB_SEQ * (KSM_FLOATS + QSM_FLOATS) : &sm.tsc_own[0];
  static_assert(!SPLIT || 4 * (CB_SEQ * (KSM_FLOATS + QSM_FLOATS) + CB_SEQ * sm.TAIL * GP) <= (int)sizeof(sm.xs), "tail scratch and scores must fit");
  auto tsc = [&](int b_, int i_) -> float* { return tsc_base + ((size_t)b_ * sm.TAIL + i_) * GP; };   // one token's eight heads
  const CacheView& cv = P.cv;
  const int h = blockIdx.x / NS, sl = blockIdx.x % NS, li = blockIdx.z, layer = P.layer0 + li;
  const int bs = threadIdx.x >> 7, c = threadIdx.x & 127;
  const int b = blockIdx.y * CB_SEQ + bs;
  const bool live = b < cv.batch;
  const int bb = live ? b : 0;
  const int G = P.group, Hkv = cv.n_kv_heads;
  const int n_entries = P.layer_count * cv.batch;
  depend_wait();
  const int seq = live ? cv.seq_len[layer * cv.batch + bb] : 0;
  // tokens [0, v_pk) have packed values (and keys): they are in the split-K partials; tokens [v_pk, seq) have raw
  // values; of those, [v_pk, k_pk) have packed keys (captioning schedule only), the rest raw keys
  const int v_pk = cv.v_packed(seq), k_pk = cv.k_packed(seq);
  const int nwin = v_pk / W, n_tail = seq - v_pk;
  const __half* qbase = P.q + (((size_t)li * cv.batch + bb) * cv.n_q_heads + h * G) * D;
  const __half* kt = cv.k_tail + cv.k_tail_off(layer, bb, h);
  const __half* vt = cv.v_tail + cv.v_tail_off(layer, bb, h);
  // Scratch inside the array of the rotated sums or of their terms (written much later), per sequence: the raw key rows of a chunk of the
  // tail (272-byte rows: 16-byte reads of 32 different rows hit different banks) or, under the captioning
  // schedule, the key parts of the up to four packed windows among the raw-value tokens; then the group's query
  // rows.  Everything is fetched with cp.async so that all the loads are in flight together.
  constexpr int KIMG = OFF_VCODE + 144;                    // key part of a window record (+ its MXFP4 metadata bytes)
  static_assert((SPLIT || CB_SEQ * (KSM_FLOATS + QSM_FLOATS) <= 3 * CB_ROWS * D) && 4 * KIMG <= KSM_FLOATS * 4, "tail scratch must fit");
  __half* ksm = reinterpret_cast<__half*>(scratch + bs * (KSM_FLOATS + QSM_FLOATS));
  __half* qsm = ksm + W * KROW;
  unsigned char* kimg = reinterpret_cast<unsigned char*>(ksm);
  const int npc = CAPTION ? (k_pk - v_pk) / W : 0;   // packed windows among the raw-value tokens: the first chunks
  // a chunk of the tail is one 32-token window: its keys are either all packed or all raw
  auto stage_tail = [&](int chunk) {
    if (chunk == 0 && c < G * (D / 8)) cp_async16(qsm + 8 * c, qbase + 8 * c);
    if (chunk >= npc)
      for (int idx = c; idx < W * (D / 8); idx += 128) {
        const int r = idx / (D / 8), c8 = idx % (D / 8);
        if (chunk * W + r < n_tail)
          cp_async16(ksm + r * KROW + 8 * c8, kt + cv.k_slot(v_pk + chunk * W + r) * D + 8 * c8);
      }
    cp_async_commit();
  };
  if (SEQ == 1)   // the raw value rows go the same way (used after the softmax numerators are known)
    for (int idx = c; idx < n_tail * (D / 8); idx += 128) {
      const int r = idx / (D / 8), c8 = idx % (D / 8);
      cp_async16(&sm.vsm[r * D + 8 * c8], vt + cv.v_slot(v_pk + r) * D + 8 * c8);
    }
  for (int ch = 0; ch < npc; ch++) {   // key parts of the packed windows whose values are still raw
    const int win = v_pk / W + ch;
    unsigned char* img = kimg + ch * KIMG;
    if (cv.fmt == FMT_FP16) {
      const unsigned char* rec = cv.meta(layer, bb, h, win);   // the record starts with its (m, s) planes
      if (c < OFF_VCODE / 16) cp_async16(img + 16 * c, rec + 16 * c);
    } else {
      const unsigned char* body = cv.body(layer, bb, h, win);
      const unsigned char* meta = cv.meta(layer, bb, h, win);
      if (c < 4) cp_async16(img + OFF_KNORM + 16 * c, body + B_KNORM + 16 * c);
      else if (c < 4 + 64) cp_async16(img + OFF_KCODE + 16 * (c - 4), body + B_KCODE + 16 * (c - 4));
      else if (c < 4 + 64 + MX_META_BYTES / 8) cp_async8(img + OFF_VCODE + 8 * (c - 68), meta + 8 * (c - 68));
    }
  }
  if (n_tail > 0) stage_tail(0);   // on its way while the prefix is computed
  const int total = block_prefix(cv, P.layer0, n_entries, sm.prefix);
  const int per = total > 0 ? (total + n_cta - 1) / n_cta : 1;
  constexpr float ACC_SCALE = PARTIAL_ACC_SCALE;
  constexpr float LOG2E = 1.4426950408889634f;
  // Coefficient of the weight sum S: -b from the codebook identity, plus the mean of what the bit-1
  // plane loses because its relative weight (3a-b)/(2(b-a)) enters the MMA rounded to fp16 (bit 1 is
  // set for half of the codes on average); the zero-mean remainder is at the 1e-5 level.
  constexpr float DELTA_REL = (3.0f * CB_INNER - CB_OUTER) / (2.0f * (CB_OUTER - CB_INNER));
  const float S_COEF = -CB_OUTER + (CB_OUTER - CB_INNER) * (DELTA_REL - __half2float(__float2half_rn(DELTA_REL)));

  const int e = li * cv.batch + bb;
  const int unit = e * Hkv + h;
  const int start = sm.prefix[e] + h * nwin, end = start + nwin;
  const int cta_lo = nwin > 0 ? start / per : 0, cta_hi = nwin > 0 ? (end - 1) / per : -1;
  const int n_hdr = SEQ == 1 ? max(0, min(cta_hi - cta_lo + 1, sm.MRG_TAB)) : 0;   // partials whose headers are staged
  if (SEQ == 1) {
    for (int idx = c; idx < n_hdr * (PARTIAL_HDR_FLOATS / 4); idx += 128) {
      const int ci = idx / (PARTIAL_HDR_FLOATS / 4), q4 = idx % (PARTIAL_HDR_FLOATS / 4);
      cp_async16(&sm.hdr[ci * PARTIAL_HDR_FLOATS + 4 * q4],
                 reinterpret_cast<const float*>(&P.partials_f[(size_t)unit + cta_lo + ci]) + 4 * q4);
    }
    cp_async_commit();
  }
  if (CAPTION) {   // scores of the packed windows among the raw-value tokens: one warp per window, on the tensor cores
    cp_async_wait<0>();
    __syncthreads();
    const int wv = c >> 5, lane = c & 31;
    if (wv < npc) {
      uint2 qreg[16];
      float fsc;
      query_fragments(qbase, P.signs + (size_t)li * D, G, P.sm_scale, lane, qreg, fsc);
      unsigned char* st = kimg + wv * KIMG;
      if (cv.fmt == FMT_MXFP4) {   // decode the stored (m, s) into the fp16 planes of the staged image
        uint2 m4, s4;
        mx_decode_lane(st + OFF_VCODE, lane, m4, s4);
        *reinterpret_cast<uint2*>(st + OFF_KM + 8 * lane) = m4;
        *reinterpret_cast<uint2*>(st + OFF_KS + 8 * lane) = s4;
        __syncwarp();
      }
      float sc[4][2];
      window_scores_mma(st, qreg, fsc, lane, sc);
      const int g = lane >> 2, t = lane & 3;
#pragma unroll
      for (int nu = 0; nu < 4; nu++)
#pragma unroll
        for (int e2 = 0; e2 < 2; e2++)
          tsc(bs, wv * W + 8 * nu + 2 * t + e2)[g] = g < G ? sc[nu][e2] : -INFINITY;
    }
    __syncthreads();   // the images are done with: the scratch takes raw key rows next
  }
  // tail scores: thread -> (token = c & 31 of a 32-token chunk, heads (c >> 5) * 2 + {0, 1})
  for (int chunk = npc; chunk * W < n_tail; chunk++) {   // chunks of raw keys
    const int tok = chunk * W + (c & 31);
    float s2[2] = {-INFINITY, -INFINITY};
    const int j0 = (c >> 5) * 2;
    if (chunk > 0) stage_tail(chunk);
    cp_async_wait<0>();
    asm volatile("bar.sync %0, 128;\n" ::"r"(bs + 1) : "memory");   // the sequence's 128 threads
    if (tok < n_tail && j0 < G) {
      float a2[2] = {0.f, 0.f};
      {
        const __half* krow = ksm + (c & 31) * KROW;
#pragma unroll 4
        for (int k = 0; k < D; k += 8) {
          const uint4 kv = *reinterpret_cast<const uint4*>(krow + k);
          const __half2* k2 = reinterpret_cast<const __half2*>(&kv);
#pragma unroll
          for (int hh = 0; hh < 2; hh++) {
            if (j0 + hh >= G) continue;
            const uint4 qv = *reinterpret_cast<const uint4*>(qsm + (j0 + hh) * D + k);
            const __half2* q2 = reinterpret_cast<const __half2*>(&qv);
#pragma unroll
            for (int u = 0; u < 4; u++) {
              const float2 qf = __half22float2(q2[u]), kf = __half22float2(k2[u]);
              a2[hh] = fmaf(qf.x, kf.x, a2[hh]);
              a2[hh] = fmaf(qf.y, kf.y, a2[hh]);
            }
          }
        }
      }
      s2[0] = a2[0] * P.sm_scale * LOG2E;
      if (j0 + 1 < G) s2[1] = a2[1] * P.sm_scale * LOG2E;
    }
    if (tok < sm.TAIL) { tsc(bs, tok)[j0] = s2[0]; tsc(bs, tok)[j0 + 1] = s2[1]; }
    if ((chunk + 1) * W < n_tail)
      asm volatile("bar.sync %0, 128;\n" ::"r"(bs + 1) : "memory");   // before the next chunk's rows land
  }
  // Blocks of several sequences have no room to hold all raw value rows: they pass through the key-row scratch 32
  // rows at a time, the first 32 on their way from here on (used once the softmax numerators are known).
  __half* vrows = ksm;
  auto stage_values = [&](int r0) {
    for (int idx = c; idx < min(W, n_tail - r0) * (D / 8); idx += 128) {
      const int r = idx / (D / 8), c8 = idx % (D / 8);
      cp_async16(vrows + r * D + 8 * c8, vt + cv.v_slot(v_pk + r0 + r) * D + 8 * c8);
    }
    cp_async_commit();
  };
  if (SEQ != 1 && n_tail > 0) {
    asm volatile("bar.sync %0, 128;\n" ::"r"(bs + 1) : "memory");   // the last chunk's key rows have been read
    stage_values(0);
  }
  // four column slices per (head, sequence): this block's 32 columns of the three matrices (48 KB) start their way
  // into shared memory now (behind the tail's own cp.async groups, which had to be waited for) and are used at the
  // very end, after the merge
  constexpr bool PRELOAD = NS == 4;
  static_assert(!PRELOAD || SEQ == 1, "the whole-slice preload needs the one-sequence buffer");
  if (PRELOAD) {
    const float* Rsl = P.R + ((size_t)li * P.n_R + (P.n_R == 1 ? 0 : h)) * 3 * D * D + sl * (D / NS);
    for (int i = threadIdx.x; i < 3 * D * (D / NS) / 4; i += SEQ * 128) {
      const int row = i / (D / NS / 4), c4 = i % (D / NS / 4);
      cp_async16(&sm.Rbuf[row * (D / NS) + 4 * c4], Rsl + (size_t)row * D + 4 * c4);
    }
    cp_async_commit();
  }
  // the staged headers must have landed (a sequence without tail tokens has not waited yet); the matrix preload,
  // the newest group, may stay in flight
  if (SEQ == 1) { if (PRELOAD) cp_async_wait<1>(); else cp_async_wait<0>(); }
  __syncthreads();
  {
    // Softmax bookkeeping by all 128 threads of the sequence: thread = (head j, stripe); a stripe takes every 16th
    // partial and every 16th tail token (the captioning schedule has up to 159 of them); stripes are joined by two
    // shuffles inside a warp and a four-entry table across the warps.
    const int j = c & (GP - 1), stripe = c >> 3, wv = c >> 5, lane = c & 31;
    const int n_part = cta_hi - cta_lo + 1;
    auto part_m = [&](int ci) {
      return ci < n_hdr ? sm.hdr[ci * PARTIAL_HDR_FLOATS + j] : P.partials_f[(size_t)unit + cta_lo + ci].m[j];
    };
    auto part_l = [&](int ci) {
      return ci < n_hdr ? sm.hdr[ci * PARTIAL_HDR_FLOATS + GP + j] : P.partials_f[(size_t)unit + cta_lo + ci].l[j];
    };
    float M = -INFINITY;
    for (int ci = stripe; ci < n_part; ci += 16) M = fmaxf(M, part_m(ci));
    for (int i = stripe; i < n_tail; i += 16) M = fmaxf(M, tsc(bs, i)[j]);
    M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 8));
    M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 16));
    if (lane < GP) sm.red[bs][wv][j] = M;
    asm volatile("bar.sync %0, 128;\n" ::"r"(bs + 1) : "memory");
    M = fmaxf(fmaxf(sm.red[bs][0][j], sm.red[bs][1][j]), fmaxf(sm.red[bs][2][j], sm.red[bs][3][j]));
    asm volatile("bar.sync %0, 128;\n" ::"r"(bs + 1) : "memory");   // the table is reused for the sums
    float L = 0.f;
    for (int ci = stripe; ci < n_part; ci += 16) {
      const float pm = part_m(ci);
      if (pm != -INFINITY) L += part_l(ci) * exp2f(pm - M);
    }
    for (int i = stripe; i < n_tail; i += 16) {   // softmax numerators in place of the scores
      const float pnum = exp2f(tsc(bs, i)[j] - M);   // 0 for the heads beyond the group (-inf scores)
      tsc(bs, i)[j] = pnum;
      L += pnum;
    }
    L += __shfl_xor_sync(0xffffffffu, L, 8);
    L += __shfl_xor_sync(0xffffffffu, L, 16);
    if (lane < GP) sm.red[bs][wv][j] = L;
    asm volatile("bar.sync %0, 128;\n" ::"r"(bs + 1) : "memory");
    if (c < GP) {
      sm.Ms[bs][c] = M;
      sm.Ls[bs][c] = (sm.red[bs][0][c] + sm.red[bs][1][c]) + (sm.red[bs][2][c] + sm.red[bs][3][c]);
    }
  }
  __syncthreads();
  // per partial and head: the rescale factor exp2(m - M) and the weight sums S_m (the four lanes of a quad hold
  // partial sums), so that the merge below only reads accumulator fragments
  for (int idx = c; idx < min(cta_hi - cta_lo + 1, sm.MRG_TAB) * GP; idx += 128) {
    const int ci = idx / GP, j = idx % GP;
    // the partial's header: staged in shared memory (one-sequence blocks) or in global memory
    const float* ph = ci < n_hdr ? &sm.hdr[ci * PARTIAL_HDR_FLOATS]
                                 : reinterpret_cast<const float*>(&P.partials_f[(size_t)unit + cta_lo + ci]);
    const float pm = ph[j];
    float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
    if (pm != -INFINITY) {
      const float4 s0 = *reinterpret_cast<const float4*>(ph + 2 * GP + 4 * j);
      const float4 s1 = *reinterpret_cast<const float4*>(ph + 2 * GP + 32 + 4 * j);
      const float4 s2 = *reinterpret_cast<const float4*>(ph + 2 * GP + 64 + 4 * j);
      f.x = exp2f(pm - sm.Ms[bs][j]);
      f.y = s0.x + s0.y + s0.z + s0.w;
      f.z = s1.x + s1.y + s1.z + s1.w;
      f.w = s2.x + s2.y + s2.z + s2.w;
    }
    *reinterpret_cast<float4*>(sm.mrg[bs][ci][j]) = f;
  }
  __syncthreads();
  // raw-value tokens: every value row is read once for all heads
  float araw[GP];
#pragma unroll
  for (int j = 0; j < GP; j++) araw[j] = 0.f;
  constexpr int TAIL_ALL = 1 << 20;   // one-sequence blocks hold all their raw value rows: a single pass
  for (int r0 = 0; r0 < n_tail; r0 += (SEQ == 1 ? TAIL_ALL : W)) {
    const __half* rows = SEQ == 1 ? sm.vsm : vrows;
    if (SEQ != 1) {
      if (r0 > 0) {
        asm volatile("bar.sync %0, 128;\n" ::"r"(bs + 1) : "memory");   // everyone is done with the previous rows
        stage_values(r0);
      }
      cp_async_wait<0>();
      asm volatile("bar.sync %0, 128;\n" ::"r"(bs + 1) : "memory");
    }
    const int nr = SEQ == 1 ? n_tail : min(W, n_tail - r0);
#pragma unroll 8
    for (int i = 0; i < nr; i++) {
      const float x = __half2float(rows[i * D + c]);
      const float4 w0 = *reinterpret_cast<const float4*>(tsc(bs, r0 + i));
      const float4 w1 = *reinterpret_cast<const float4*>(tsc(bs, r0 + i) + 4);
      araw[0] = fmaf(w0.x, x, araw[0]); araw[1] = fmaf(w0.y, x, araw[1]);
      araw[2] = fmaf(w0.z, x, araw[2]); araw[3] = fmaf(w0.w, x, araw[3]);
      araw[4] = fmaf(w1.x, x, araw[4]); araw[5] = fmaf(w1.y, x, araw[5]);
      araw[6] = fmaf(w1.z, x, araw[6]); araw[7] = fmaf(w1.w, x, araw[7]);
    }
  }
  // (the value rows passed through scratch inside the array of the terms, which the merge below fills: a sequence
  // group must not start writing it while another still reads its rows)
  if (SEQ != 1) __syncthreads();
  // merge of the split-K partials, four heads at a time: per partial the twelve accumulator fragments of this
  // thread's channel are fetched together (independent loads), then scaled by the table's factors
#pragma unroll
  for (int jg = 0; jg < GP; jg += 4) {
    float vacc[4][3];
#pragma unroll
    for (int jj = 0; jj < 4; jj++) vacc[jj][0] = vacc[jj][1] = vacc[jj][2] = 0.f;
    if (jg < G) {
      // one-sequence blocks have registers to spare: the fragments of four partials are fetched together (a long
      // single sequence has dozens of partials per head)
      constexpr int MU4 = SEQ == 1 ? 4 : 1;
      for (int ct0 = cta_lo; ct0 <= cta_hi; ct0 += MU4) {
        float fr[MU4][4][3];
#pragma unroll
        for (int u = 0; u < MU4; u++) {
          const PartialF& pp = P.partials_f[(size_t)unit + min(ct0 + u, cta_hi)];
#pragma unroll
          for (int jj = 0; jj < 4; jj++) {
            const int j = jg + jj;
            const int r = 4 * (c >> 4) + 2 * ((c >> 3) & 1) + (j & 1), l32 = 4 * (c & 7) + (j >> 1);
#pragma unroll
            for (int m = 0; m < 3; m++) fr[u][jj][m] = pp.frag[m][r][l32];
          }
        }
#pragma unroll
        for (int u = 0; u < MU4; u++) {
          const int ct = ct0 + u;
          if (ct > cta_hi) continue;
          const PartialF& pp = P.partials_f[(size_t)unit + ct];
#pragma unroll
          for (int jj = 0; jj < 4; jj++) {
            const int j = jg + jj;
            float ef, S[3];
            if (ct - cta_lo < sm.MRG_TAB) {
              const float4 f = *reinterpret_cast<const float4*>(sm.mrg[bs][ct - cta_lo][j]);
              ef = f.x; S[0] = f.y; S[1] = f.z; S[2] = f.w;
            } else {   // more partials than the table holds (few heads over many CTAs): compute in place
              const float pm = pp.m[j];
              ef = pm == -INFINITY ? 0.f : exp2f(pm - sm.Ms[bs][j]);
#pragma unroll
              for (int m = 0; m < 3; m++) S[m] = pp.Sp[m][4 * j] + pp.Sp[m][4 * j + 1] + pp.Sp[m][4 * j + 2] + pp.Sp[m][4 * j + 3];
            }
            if (j < G && ef != 0.f) {
#pragma unroll
              for (int m = 0; m < 3; m++) vacc[jj][m] = fmaf(fmaf(ACC_SCALE, fr[u][jj][m], S_COEF * S[m]), ef, vacc[jj][m]);
            }
          }
        }
      }
    }
#pragma unroll
    for (int jj = 0; jj < 4; jj++) {
#pragma unroll
      for (int m = 0; m < 3; m++) {
        if constexpr (SPLIT) {
          uint32_t tm[3];
          bf16_terms(vacc[jj][m], 0.f, tm);
#pragma unroll
          for (int i = 0; i < 3; i++) sm.xs[i][bs * GP + jg + jj][m * D + c] = (unsigned short)tm[i];
        } else {
          sm.vec[m][bs * GP + jg + jj][c] = vacc[jj][m];
        }
      }
      sm.rawv[bs * GP + jg + jj][c] = araw[jg + jj];
    }
  }

  if constexpr (SPLIT) {
    // out[row][c] = raw[row][c] + sum_m sum_r R_m[r][c] * vec[m][row][r] on the tensor cores: both factors as three bf16 terms (24
    // bits, the exponents of fp32), the six products whose terms' orders add up to at most four.  A warp takes all 32 rows, 16
    // columns and half of the 384 rotated channels; its share of the matrices comes straight from L2, a step ahead.  The products of
    // a step of 16 channels are summed on the tensor cores, small ones first, the steps with rounded additions: the tensor cores cut
    // their sums off, and one accumulator for all 72 products was 6.6e-7 too small (error 8.1e-7 of the output's norm; 8e-8 this way,
    // 2.1e-7 a chain of fp32 multiply-adds), for 1 to 2 % of a small call.  On CUDA cores the
    // product was bound by shared memory (a 4 x 4 tile per thread: two multiply-adds per number read) at 24000 cycles a block;
    // about half now.  28 layers x 8 sequences x 4 heads at 300 tokens, the whole call: 81.9 -> 70.6 us; 28 x 16 x 8 at 64: 181 -> 142.
    __syncthreads();   // the terms are complete
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int kh = warp >> 3, n0 = 16 * (warp & 7);
    const float* Rset = P.R + ((size_t)li * P.n_R + (P.n_R == 1 ? 0 : h)) * 3 * D * D;
    constexpr int KS = 3 * D / 16 / 2;   // 16-channel steps of a half
    float acc[2][2][4];
#pragma unroll
    for (int m = 0; m < 2; m++)
#pragma unroll
      for (int n = 0; n < 2; n++)
#pragma unroll
        for (int i = 0; i < 4; i++) acc[m][n][i] = 0.f;
    float rn[2][4];
    auto fetch = [&](int ks) {
#pragma unroll
      for (int n = 0; n < 2; n++) {
        const float* p = Rset + (size_t)(16 * ks + 2 * t) * D + n0 + 8 * n + g;
        rn[n][0] = __ldg(p); rn[n][1] = __ldg(p + D); rn[n][2] = __ldg(p + 8 * D); rn[n][3] = __ldg(p + 9 * D);
      }
    };
    fetch(kh * KS);
    const unsigned short* arow = &sm.xs[0][lane & 15][8 * (lane >> 4)];
    for (int ks = kh * KS; ks < (kh + 1) * KS; ks++) {
      uint32_t b[2][2][3];
#pragma unroll
      for (int n = 0; n < 2; n++) {
        bf16_terms(rn[n][0], rn[n][1], b[n][0]);
        bf16_terms(rn[n][2], rn[n][3], b[n][1]);
      }
      if (ks + 1 < (kh + 1) * KS) fetch(ks + 1);
#pragma unroll
      for (int m = 0; m < 2; m++) {
        float part[2][4];
#pragma unroll
        for (int n = 0; n < 2; n++)
#pragma unroll
          for (int i = 0; i < 4; i++) part[n][i] = 0.f;
#pragma unroll
        for (int ta = 2; ta >= 0; ta--) {
          uint32_t a[4];
          ldsm_x4(a, arow + (ta * CB_ROWS + 16 * m) * sm.XP + 16 * ks);
#pragma unroll
          for (int tb = 2 - ta; tb >= 0; tb--)
#pragma unroll
            for (int n = 0; n < 2; n++) mma16816_bf16(part[n], a, b[n][0][tb], b[n][1][tb]);
        }
#pragma unroll
        for (int n = 0; n < 2; n++)
#pragma unroll
          for (int i = 0; i < 4; i++) acc[m][n][i] += part[n][i];
      }
    }
    __syncthreads();   // everyone has read the terms
    float* half_out = reinterpret_cast<float*>(&sm.xs[0][0][0]) + kh * CB_ROWS * sm.OUT_PITCH;
#pragma unroll
    for (int m = 0; m < 2; m++)
#pragma unroll
      for (int n = 0; n < 2; n++)
#pragma unroll
        for (int i = 0; i < 2; i++)
          *reinterpret_cast<float2*>(&half_out[(16 * m + g + 8 * i) * sm.OUT_PITCH + n0 + 8 * n + 2 * t]) = make_float2(acc[m][n][2 * i], acc[m][n][2 * i + 1]);
    __syncthreads();
    const float* sums = reinterpret_cast<const float*>(&sm.xs[0][0][0]);
    for (int i = threadIdx.x; i < CB_ROWS * D / 4; i += SEQ * 128) {
      const int row = i / (D / 4), cl = 4 * (i % (D / 4)), ob = blockIdx.y * CB_SEQ + row / GP, j = row % GP;
      if (ob >= cv.batch || j >= G) continue;
      const float L = sm.Ls[row / GP][j];
      const float inv = L > 0.f ? 1.0f / L : 0.f;
      const float4 x = *reinterpret_cast<const float4*>(&sums[row * sm.OUT_PITCH + cl]);
      const float4 y = *reinterpret_cast<const float4*>(&sums[(CB_ROWS + row) * sm.OUT_PITCH + cl]);
      const float4 rv = *reinterpret_cast<const float4*>(&sm.rawv[row][cl]);
      *reinterpret_cast<float4*>(&P.out[(((size_t)li * cv.batch + ob) * cv.n_q_heads + h * G + j) * D + cl]) =
          make_float4((x.x + y.x + rv.x) * inv, (x.y + y.y + rv.y) * inv, (x.z + y.z + rv.z) * inv, (x.w + y.w + rv.w) * inv);
    }
  } else {
    // out[row][c] = raw[row][c] + sum_m sum_r R_m[r][c] * vec[m][row][r].  The first half of the threads compute
    // a 4-row x 4-column tile each; the second half stream the matrices through shared memory in 16-row
    // slices, three slices ahead.
    // (with the matrices preloaded there is nothing to stream: both halves compute, each every other 16-row slice)
    constexpr bool PRE = NS == 4;
    const int khalf = PRE ? threadIdx.x / 64 : 0;
    const bool comp = PRE || threadIdx.x < 64;
    constexpr int CW = 4 / NS;          // output columns per compute thread
    constexpr int SW = D / NS;          // output columns of this CTA = floats per staged matrix row
    static_assert(NS == 1 || NS == 4, "column slices");
    const int rw = ((threadIdx.x & 63) >> 5) * 4, cl = (threadIdx.x & 31) * CW;   // first row / column (inside the slice) of the tile
    const float* Rset = P.R + ((size_t)li * P.n_R + (P.n_R == 1 ? 0 : h)) * 3 * D * D + sl * SW;
    constexpr int N_CHUNK = 3 * D / CB_CHUNK;
    float* rbuf = &sm.Rbuf[0];          // ring of CB_NBUF slices of CB_CHUNK x SW floats (or, preloaded, all rows)
    auto stage = [&](int chunk) {   // rows [16*chunk, 16*chunk+16) of the three stacked matrices, this CTA's columns
      const float* src = Rset + (size_t)chunk * CB_CHUNK * D;
      float* dst = rbuf + (chunk % CB_NBUF) * CB_CHUNK * SW;
      if (chunk < N_CHUNK)
        for (int i = threadIdx.x - 64; i < CB_CHUNK * SW / 4; i += 64) {
          const int row = i / (SW / 4), c4 = i % (SW / 4);
          cp_async16(dst + row * SW + 4 * c4, src + (size_t)row * D + 4 * c4);
        }
      cp_async_commit();
    };
    float o[4][CW];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int k = 0; k < CW; k++) o[i][k] = 0.f;
    if (PRELOAD) {
      cp_async_wait<0>();
      __syncthreads();   // the matrices have landed and vec is complete
    } else {
      if (!comp)
        for (int pre = 0; pre < CB_NBUF - 1; pre++) stage(pre);
    }
    for (int chunk = 0; chunk < N_CHUNK; chunk++) {
      if (!PRELOAD) {
        if (!comp) cp_async_wait<CB_NBUF - 2>();
        __syncthreads();   // slice `chunk` has landed; everyone is done with slice chunk-1 (and, first time, vec is complete)
      }
      if (!comp) {
        if (!PRELOAD) stage(chunk + CB_NBUF - 1);   // into the buffer of slice chunk-1
      } else if (!PRE || (chunk & 1) == khalf) {
        const int m = chunk / (D / CB_CHUNK), r0 = (chunk % (D / CB_CHUNK)) * CB_CHUNK;
        const float* rb = rbuf + (PRELOAD ? chunk : chunk % CB_NBUF) * CB_CHUNK * SW;
#pragma unroll 2
        for (int r = 0; r < CB_CHUNK; r += 4) {
          float4 x[4];
#pragma unroll
          for (int i = 0; i < 4; i++) x[i] = *reinterpret_cast<const float4*>(&sm.vec[m][rw + i][r0 + r]);
          if (NS == 1) {
            float4 rr[4];
#pragma unroll
            for (int k = 0; k < 4; k++) rr[k] = *reinterpret_cast<const float4*>(&rb[(r + k) * SW + cl]);
#pragma unroll
            for (int i = 0; i < 4; i++) {
              o[i][0] = fmaf(rr[0].x, x[i].x, o[i][0]); o[i][1 % CW] = fmaf(rr[0].y, x[i].x, o[i][1 % CW]);
              o[i][2 % CW] = fmaf(rr[0].z, x[i].x, o[i][2 % CW]); o[i][3 % CW] = fmaf(rr[0].w, x[i].x, o[i][3 % CW]);
              o[i][0] = fmaf(rr[1].x, x[i].y, o[i][0]); o[i][1 % CW] = fmaf(rr[1].y, x[i].y, o[i][1 % CW]);
              o[i][2 % CW] = fmaf(rr[1].z, x[i].y, o[i][2 % CW]); o[i][3 % CW] = fmaf(rr[1].w, x[i].y, o[i][3 % CW]);
              o[i][0] = fmaf(rr[2].x, x[i].z, o[i][0]); o[i][1 % CW] = fmaf(rr[2].y, x[i].z, o[i][1 % CW]);
              o[i][2 % CW] = fmaf(rr[2].z, x[i].z, o[i][2 % CW]); o[i][3 % CW] = fmaf(rr[2].w, x[i].z, o[i][3 % CW]);
              o[i][0] = fmaf(rr[3].x, x[i].w, o[i][0]); o[i][1 % CW] = fmaf(rr[3].y, x[i].w, o[i][1 % CW]);
              o[i][2 % CW] = fmaf(rr[3].z, x[i].w, o[i][2 % CW]); o[i][3 % CW] = fmaf(rr[3].w, x[i].w, o[i][3 % CW]);
            }
          } else {   // one column per thread
            const float r0v = rb[(r + 0) * SW + cl], r1v = rb[(r + 1) * SW + cl], r2v = rb[(r + 2) * SW + cl], r3v = rb[(r + 3) * SW + cl];
#pragma unroll
            for (int i = 0; i < 4; i++)
              o[i][0] = fmaf(r3v, x[i].w, fmaf(r2v, x[i].z, fmaf(r1v, x[i].y, fmaf(r0v, x[i].x, o[i][0]))));
          }
        }
      }
    }
    if (PRE) {   // the second half's sums reach the first through the tail-score array, idle by now
      float* red = &sm.tsc_own[0] + (threadIdx.x & 63) * 4 * CW;
      static_assert(!PRE || 64 * 4 * CW <= W * GP, "reduction scratch");
      if (khalf) {
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
          for (int k = 0; k < CW; k++) red[i * CW + k] = o[i][k];
      }
      __syncthreads();
      if (!khalf) {
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
          for (int k = 0; k < CW; k++) o[i][k] += red[i * CW + k];
      }
    }
    if (comp && !khalf) {
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const int row = rw + i;   // head of the group
        if (row >= G) continue;
        const float L = sm.Ls[0][row];
        const float inv = L > 0.f ? 1.0f / L : 0.f;
        float* dst = &P.out[(((size_t)li * cv.batch + b) * cv.n_q_heads + h * G + row) * D + sl * SW + cl];
        if (NS == 1) {
          const float4 rv = *reinterpret_cast<const float4*>(&sm.rawv[row][cl]);
          *reinterpret_cast<float4*>(dst) = make_float4((o[i][0] + rv.x) * inv, (o[i][1 % CW] + rv.y) * inv,
                                                        (o[i][2 % CW] + rv.z) * inv, (o[i][3 % CW] + rv.w) * inv);
        } else {
          dst[0] = (o[i][0] + sm.rawv[row][sl * SW + cl]) * inv;
        }
      }
    }
  }
}

template <bool CAPTION, int NS, int SEQ>
static cudaError_t combine_attr() {
  return cudaFuncSetAttribute(k_combine_mma<CAPTION, NS, SEQ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sizeof(CombineSmem<CAPTION, SEQ>));
}

template <bool CAPTION, int NS, int SEQ>
static void combine_launch(const DecodeParams& P, int n_cta, cudaStream_t s) {
  const dim3 grid(P.cv.n_kv_heads * NS, (P.cv.batch + SEQ - 1) / SEQ, P.layer_count);
  launch_dependent(k_combine_mma<CAPTION, NS, SEQ>, grid, SEQ * 128, sizeof(CombineSmem<CAPTION, SEQ>), s, 1, P, n_cta);
}

static int combine_form(const CacheView& cv, int layer_count, int n_cta) {
  // A block per sequence and head while they all run at once, four sequences per block, whose product is on the tensor cores, from there
  // on (30000 tokens: 132 units of 3 sequences 166 us against 175 with blocks of four, 152 units of 2, 3 and 4 sequences 196, 198 and 198
  // against 188, 194 and 197; 28 layers x 4 sequences x 4 heads at 2000 / 8192 tokens 123 / 192 against 90 / 163).  The captioning
  // schedule's long raw tails make four full sequences as slow as two waves of single ones (8192 tokens: 152 units of 4 sequences 122
  // against 125 us, 304 units 184 against 165; of 3 sequences 180 units 132 against 126).  A single sequence would leave three quarters
  // of such a block idle.  A handful of units (e.g. a single-layer call) shares four blocks each, a quarter of the output columns per
  // block.
  const int units = cv.n_kv_heads * cv.batch * layer_count, waves = cv.sched == SCHED_CAPTION && cv.batch >= CB_SEQ_MAX ? 2 : 1;
  const int n_blocks = cv.n_kv_heads * ((cv.batch + CB_SEQ_MAX - 1) / CB_SEQ_MAX) * layer_count;
  if (4 * n_blocks <= n_cta) return OKQ_PLAN_PAIR_QUARTER;
  return cv.batch < 2 || units <= waves * sm_count() ? OKQ_PLAN_PAIR_ONE : OKQ_PLAN_PAIR_FOUR;
}

template <bool CAPTION>
static void combine_dispatch(const DecodeParams& P, int form, int n_cta, cudaStream_t s) {
  switch (form) {
    case OKQ_PLAN_PAIR_QUARTER: combine_launch<CAPTION, 4, 1>(P, n_cta, s); break;
    case OKQ_PLAN_PAIR_ONE: combine_launch<CAPTION, 1, 1>(P, n_cta, s); break;
    default: combine_launch<CAPTION, 1, CB_SEQ_MAX>(P, n_cta, s);
  }
}

int g_decode_impl = 1;

int decode_plan(const DecodeParams& P, int n_cta) {
  // (the one-launch kernel: where the library chooses the grid itself)
  const int cs = P.n_splits == 0 && g_decode_impl == 1 ? decode_small_cluster(P.cv, P.layer_count, P.piece_slots) : 0;
  return cs > 0 ? cs : combine_form(P.cv, P.layer_count, n_cta);
}

okq_status launch_decode_mma(const DecodeParams& P, int n_cta, cudaStream_t s, cudaEvent_t before, cudaEvent_t after) {
  const int plan = decode_plan(P, n_cta);
  if (plan > 0) {
    if (before) cudaEventRecord(before, s);
    const okq_status st = launch_decode_small(P, plan, s);
    if (after) cudaEventRecord(after, s);
    return st;
  }
  static thread_local unsigned long long attr_mask = 0;
  int attr_dev = 0;
  if (attr_needed(attr_mask, attr_dev)) {
    cudaError_t e = cudaFuncSetAttribute(k_decode_mma<FMT_FP16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(MmaSmem<FMT_FP16>));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_decode_mma<FMT_MXFP4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)sizeof(MmaSmem<FMT_MXFP4>));
    if (e == cudaSuccess) e = combine_attr<false, 4, 1>();
    if (e == cudaSuccess) e = combine_attr<false, 1, 1>();
    if (e == cudaSuccess) e = combine_attr<false, 1, CB_SEQ_MAX>();
    if (e == cudaSuccess) e = combine_attr<true, 4, 1>();
    if (e == cudaSuccess) e = combine_attr<true, 1, 1>();
    if (e == cudaSuccess) e = combine_attr<true, 1, CB_SEQ_MAX>();
    if (e != cudaSuccess) { set_last_cuda_error((int)e); return OKQ_ERR_CUDA; }
    attr_done(attr_mask, attr_dev);
  }
  if (before) cudaEventRecord(before, s);
  if (P.cv.fmt == FMT_FP16 && g_decode_impl == 0) {
    const okq_status st = launch_decode_tc(P, n_cta, s);
    if (st != OKQ_OK) return st;
  } else if (P.cv.fmt == FMT_MXFP4) launch_dependent(k_decode_mma<FMT_MXFP4>, dim3(n_cta), NTHREADS, sizeof(MmaSmem<FMT_MXFP4>), s, 1, P);
  else launch_dependent(k_decode_mma<FMT_FP16>, dim3(n_cta), NTHREADS, sizeof(MmaSmem<FMT_FP16>), s, 1, P);
  if (after) cudaEventRecord(after, s);
  if (P.cv.sched == SCHED_CAPTION) combine_dispatch<true>(P, plan, n_cta, s);
  else combine_dispatch<false>(P, plan, n_cta, s);
  return OKQ_OK;
}

}  // namespace okq
