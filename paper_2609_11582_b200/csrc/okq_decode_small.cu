// Fused decode attention in one launch, for calls with few (layer, sequence, KV head) units: a model's per-layer call.
//
// The split-K kernel and its combine kernel are a chain of launch, prefix, partials through memory, launch, prefix,
// merge; with a handful of windows per warp that chain is the whole time (35 + 20 us for one layer of 4 sequences at
// 4096 tokens).  Here a thread-block cluster (or one block) owns one unit: its CS x 12 warps walk the unit's windows (the same code as
// the split-K kernel), leave their sums as pieces in global memory (L2), and after one cluster barrier MS of them (all; four of six)
// merge 1 / MS of the rotated channels each over all pieces.  The merged sums are pushed into those CTAs' shared memory, and after
// the second barrier each of them applies R_m^T for 1 / MS of the output columns.  The raw tail is scored by each of them (its
// rows are staged at the start) while the first barrier is on its way.
// What bounds it: latency (launch, query rotation, the first window of a warp, two cluster barriers, L2 round trips of the
// merge).  One sequence, one head group of seven, 2048 tokens: 59 -> 11.3 us per call; one layer of 4 sequences x 4 heads at
// 4111 tokens 32 -> 16.8 us against the split-K pair.
#include <cooperative_groups.h>
#include "okq_decode_walk.cuh"

namespace cg = cooperative_groups;

namespace okq {

namespace {

constexpr int KROW = D + 8;                     // halfs per staged raw key row: 16-byte reads of 32 rows over all banks
constexpr int KIMG = OFF_VCODE + 144;           // key part of a window record (+ its MXFP4 metadata bytes)
constexpr int PC_MAX = 4;                       // packed windows among the raw-value tokens (captioning schedule)

// What a CTA's block index and its sequence's length say, worked out in front of the windows' walk and read back from shared memory
// behind it: the walk needs every register there is, and what lives across it is spilled in its loop (4 % of a call with several
// windows per warp).
struct __align__(16) Place {
  int unit, rank, h, b, li, layer;
  // tokens [0, v_pk) have packed values (and keys); of the rest, [v_pk, k_pk) have packed keys (captioning schedule only)
  int v_pk, k_pk, nwin, n_tail, npc, n_rawk;
  // The windows make `used` pieces of at most cnt windows, dealt out evenly over the CTAs (this one has [piece0, piece1)): one CTA
  // filled after the other, 64 windows over 192 warps were one for every warp of five CTAs, three to a sub-partition's dispatch, and
  // nothing for the rest (13.5 -> 11.3 us).  Up to four pieces stay with the first CTA, a sub-partition each, except in a cluster of 16
  // (32 units, 64 tokens: 9.6 -> 9.3 us).  Fewer windows per piece, spread over all warps, is no better: what a warp does once, whatever
  // its windows, is dispatch of the same SM.
  int cnt, used, piece0, piece1;
};

struct PieceMeta { float m[GP], l[GP]; int held; };

template <int FMT, int CS> struct SmallSmem {
  static constexpr int MS = CS == 6 ? 4 : CS;   // CTAs that merge and write: the largest power of two
  static constexpr int C = D / MS;              // output columns (and merged channels) of one of them
  static constexpr int NP = CS * NWARP;         // pieces of a unit
  static constexpr int KS = 2 * NTHREADS / C;   // row slices of the product (a thread takes two columns)
  static constexpr int TAIL = CAPTION_V_SLOTS;
  static constexpr bool STAGED = CS >= 2;       // matrices and raw value rows in shared memory (a single block: from L2)
  // what takes the record ring's place once every warp of the CTA has walked its range
  struct After {
    __align__(16) float R[STAGED ? 3 * D : 1][C];   // this CTA's columns of the three matrices
    __align__(16) __half v[STAGED ? TAIL : 1][C];   // and of the raw value rows
    __align__(16) __half k[CAPTION_K_GROUP - W][KROW];   // raw key rows behind the first 32
    __align__(16) unsigned char img[PC_MAX][KIMG];
    __align__(16) float tsc[TAIL][GP];          // tail scores (log2 domain), then numerators
    __align__(16) float fac[NP][GP];            // per piece and head: exp2(piece maximum - maximum)
    __align__(16) float4 part[NTHREADS];        // merge: sums over a share of the pieces
    __align__(16) float vec[3 * D][GP];         // merged rotated-basis sums [modality * 128 + channel][head], each CTA's
                                                // share written by that CTA (behind the first cluster barrier)
    __align__(16) float prod[KS][GP][C];
    float red[NWARP][GP];
    float M[GP], L[GP];
  };
  union { WarpSmem<FMT> w[NWARP]; After a; };
  // written by the other CTAs of the cluster at any time
  PieceMeta meta[NP];
  __align__(16) __half k0[W][KROW], q[GP][KROW];   // staged at the start: the first 32 raw key rows, the queries
  // query fragments of the unit in mma A order, high and low parts: [kq][lane][r & 3], and the heads' scales
  __align__(16) uint32_t qhi[4][32][4], qlo[4][32][4];
  float fsc[GP];
  Place at;
};

// Rotated query of head g as fragments in shared memory, by one warp with four channels per lane: the transform of
// query_fragments with its butterflies over the lanes (every warp of the CTA needs the same fragments).
__device__ __forceinline__ void head_fragments(const __half* qrow, const float* signs, float sm_scale, int g, bool have, int lane,
                                               uint32_t (*qhi)[32][4], uint32_t (*qlo)[32][4], float* fsc) {
  float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
  if (have) {
    x = load_row4(qrow, lane);
    const float4 sv = *reinterpret_cast<const float4*>(signs + 4 * lane);
    x.x *= sv.x; x.y *= sv.y; x.z *= sv.z; x.w *= sv.w;
  }
  x = warp_fwht(x, lane);
  x.x *= RSQRT_D; x.y *= RSQRT_D; x.z *= RSQRT_D; x.w *= RSQRT_D;
  float mx = fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w)));
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
  int ex = 0;
  if (mx > 0.f) frexpf(mx, &ex);           // mx < 2^ex
  const int kh = 14 - ex, r = lane >> 1;   // |q'| * 2^kh < 2^14; channels 4 lane .. 4 lane + 3 = fragment r, t = 2 (lane & 1) + {0, 1}
  const float sc = exp2f((float)kh) / (float)(1 << (2 * (r & 3)));
  if (lane == 0) fsc[g] = exp2f((float)(24 - kh)) * sm_scale * 1.4426950408889634f;
  const float v[4] = {x.x * sc, x.y * sc, x.z * sc, x.w * sc};
#pragma unroll
  for (int i = 0; i < 2; i++) {
    const __half2 hi = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
    const float2 hf = __half22float2(hi);
    const int l = 4 * g + 2 * (lane & 1) + i;
    qhi[r >> 2][l][r & 3] = h2u(hi);
    qlo[r >> 2][l][r & 3] = h2u(__floats2half2_rn(v[2 * i] - hf.x, v[2 * i + 1] - hf.y));
  }
}

}  // namespace

// grid CS * units, clusters of CS; unit = (layer, sequence, KV head)
template <int FMT, int CS>
__global__ void __launch_bounds__(NTHREADS, 1) k_decode_small(DecodeParams P) {
  using SM = SmallSmem<FMT, CS>;
  constexpr int C = SM::C, MS = SM::MS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SM& sm = *reinterpret_cast<SM*>(smem_raw);
  typename SM::After& af = sm.a;
  const CacheView& cv = P.cv;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = P.group;
  Place at;
  at.unit = blockIdx.x / CS; at.rank = blockIdx.x % CS;
  {
    const int e = at.unit / cv.n_kv_heads;
    at.h = at.unit % cv.n_kv_heads; at.b = e % cv.batch; at.li = e / cv.batch; at.layer = P.layer0 + at.li;
  }
  depend_wait();
  const __half *kt_kept, *vt_kept;
  WarpPiece* pieces_kept;
  // Headers of as many pieces as there are, in a cluster of 16; of all places in smaller ones, warps without windows filling those behind
  // the pieces': loops of a fixed length are 0.3 us shorter there, 0.3 us longer here.
  constexpr bool COUNTED = CS > 8;
  WalkEnd we{-INFINITY, 0.f, 0u};
  // (a single block with fp16 metadata has the registers to keep addresses and all across the walk)
  constexpr bool KEEP = CS == 1 && FMT == FMT_FP16;
  auto pieces_of = [](const Place& a) { return KEEP ? (a.cnt > 0 ? (a.nwin + a.cnt - 1) / a.cnt : 0) : a.cnt > 1 ? (a.nwin + a.cnt - 1) / a.cnt : a.nwin; };
  {
    const int seq = cv.seq_len[at.layer * cv.batch + at.b];
    at.v_pk = cv.v_packed(seq); at.k_pk = cv.k_packed(seq); at.nwin = at.v_pk / W; at.n_tail = seq - at.v_pk;
    at.npc = (at.k_pk - at.v_pk) / W; at.n_rawk = seq - at.k_pk;
    at.cnt = (at.nwin + CS * NWARP - 1) / (CS * NWARP);
    at.used = CS > 1 ? pieces_of(at) : 0;   // (a single block's division can wait)
    at.piece0 = at.used * at.rank / CS; at.piece1 = CS > 1 ? at.used * (at.rank + 1) / CS : NWARP;
    if (CS > 1 && !COUNTED && at.used <= 4) { at.piece0 = at.rank ? at.used : 0; at.piece1 = at.used; }   // (a warp per sub-partition)
    if (CS > 1 && tid == 0) sm.at = at;
    const __half* qbase = P.q + (((size_t)at.li * cv.batch + at.b) * cv.n_q_heads + (size_t)at.h * G) * D;
    const float* signs = P.signs + (size_t)at.li * D;
    const __half* kt = cv.k_tail + cv.k_tail_off(at.layer, at.b, at.h);
    kt_kept = kt; vt_kept = cv.v_tail + cv.v_tail_off(at.layer, at.b, at.h);
    pieces_kept = P.pieces + (size_t)at.unit * (CS * NWARP);

    // ---- on their way from the start: queries and the first raw keys
    for (int i = tid; i < G * (D / 8); i += NTHREADS) cp_async16(&sm.q[i / (D / 8)][8 * (i % (D / 8))], qbase + 8 * i);
    for (int i = tid; i < min(W, at.n_rawk) * (D / 8); i += NTHREADS)
      cp_async16(&sm.k0[i / (D / 8)][8 * (i % (D / 8))], kt + cv.k_slot(at.k_pk + i / (D / 8)) * D + 8 * (i % (D / 8)));
    cp_async_commit();

    cluster.barrier_arrive();   // every CTA of the cluster runs before its shared memory is written from outside
    // ---- this warp's windows
    auto queries = [&]() {   // the CTA's first eight warps, then everyone waits
      if (warp < GP) head_fragments(qbase + warp * D, signs, P.sm_scale, warp, warp < G, lane, sm.qhi, sm.qlo, sm.fsc);
      asm volatile("bar.sync 1, %0;\n" ::"n"(NTHREADS) : "memory");
    };
    const int piece = at.piece0 + warp;
    if (CS > 1 ? piece < at.piece1 : piece * at.cnt < at.nwin) {
      Segment sg;
      sg.rec0 = cv.unit(at.layer, at.b, at.h);
      sg.mod0 = cv.modality + (size_t)at.b * cv.capacity;
      sg.w0 = piece * at.cnt;
      sg.n_my = min(at.cnt, at.nwin - sg.w0);
      sg.piece = P.pieces + (size_t)at.unit * (CS * NWARP) + piece;
      we = walk_segment<FMT>(sm.w[warp], reinterpret_cast<const uint4(*)[32]>(sm.qlo), sg, lane, [&](uint32_t (&qh)[16], float& fsc) {
        queries();
        fsc = sm.fsc[lane >> 2];
#pragma unroll
        for (int kq = 0; kq < 4; kq++) {
          const uint4 x = *reinterpret_cast<const uint4*>(sm.qhi[kq][lane]);
          qh[4 * kq] = x.x; qh[4 * kq + 1] = x.y; qh[4 * kq + 2] = x.z; qh[4 * kq + 3] = x.w;
        }
      });
    } else {
      queries();
    }
  }
  if (CS > 1) {                    // (a single block, with less to keep: as they are)
    asm volatile("" ::: "memory");   // (written in front of the warps' common barrier for the queries)
    at = sm.at;
  }
  cluster.barrier_wait();
  // ---- the piece's header goes to every merging CTA of the cluster
  const bool held = CS == 1 || warp < at.piece1 - at.piece0;
  if (!COUNTED || held) {
    const int slot = held ? at.piece0 + warp : at.used + at.rank * NWARP + warp - at.piece1;
    for (int r = 0; r < MS; r++) {
      PieceMeta* pm = cluster.map_shared_rank(&sm.meta[slot], r);
      if ((lane & 3) == 0) { pm->m[lane >> 2] = we.m; pm->l[lane >> 2] = we.l; }
      if (lane == 0) pm->held = (int)we.held;
    }
  }
  cluster.barrier_arrive();   // (release: the pieces and their headers)
  if (MS < CS && at.rank >= MS) {   // the rest is the merging CTAs'
    cp_async_wait<0>();
    cluster.barrier_wait();
    cluster.sync();
    return;
  }
  cp_async_wait<0>();
  __syncthreads();            // the record rings are idle: their space holds the rest from here on

  const int rank = at.rank, h = at.h, b = at.b, li = at.li, layer = at.layer;
  const int v_pk = at.v_pk, k_pk = at.k_pk, nwin = at.nwin, n_tail = at.n_tail, npc = at.npc, n_rawk = at.n_rawk, n_meta = COUNTED ? at.used : SM::NP;
  const __half* kt = KEEP ? kt_kept : cv.k_tail + cv.k_tail_off(layer, b, h);
  const __half* vt = KEEP ? vt_kept : cv.v_tail + cv.v_tail_off(layer, b, h);
  WarpPiece* const pieces = KEEP ? pieces_kept : P.pieces + (size_t)at.unit * (CS * NWARP);
  // ---- rest of the tail, value rows and matrices
  for (int i = tid; i < (n_rawk - W) * (D / 8); i += NTHREADS)
    cp_async16(&af.k[i / (D / 8)][8 * (i % (D / 8))], kt + cv.k_slot(k_pk + W + i / (D / 8)) * D + 8 * (i % (D / 8)));
  for (int w = 0; w < npc; w++) {
    const int win = nwin + w;
    unsigned char* img = af.img[w];
    if (FMT == FMT_FP16) {
      const unsigned char* rec = cv.meta(layer, b, h, win);   // the record starts with its (m, s) planes
      if (tid < OFF_VCODE / 16) cp_async16(img + 16 * tid, rec + 16 * tid);
    } else {
      const unsigned char* body = cv.body(layer, b, h, win);
      const unsigned char* meta = cv.meta(layer, b, h, win);
      if (tid < 4) cp_async16(img + OFF_KNORM + 16 * tid, body + B_KNORM + 16 * tid);
      else if (tid < 4 + 64) cp_async16(img + OFF_KCODE + 16 * (tid - 4), body + B_KCODE + 16 * (tid - 4));
      else if (tid < 4 + 64 + MX_META_BYTES / 8) cp_async8(img + OFF_VCODE + 8 * (tid - 68), meta + 8 * (tid - 68));
    }
  }
  cp_async_commit();
  const float* Rsl = P.R + ((size_t)li * P.n_R + (P.n_R == 1 ? 0 : h)) * 3 * D * D + rank * C;
  if (SM::STAGED)
    for (int i = tid; i < n_tail * (C / 8); i += NTHREADS)
      cp_async16(&af.v[i / (C / 8)][8 * (i % (C / 8))], vt + cv.v_slot(v_pk + i / (C / 8)) * D + rank * C + 8 * (i % (C / 8)));
  for (int i = tid; i < 3 * D * (C / 4); i += NTHREADS) {
    if (SM::STAGED) cp_async16(&af.R[i / (C / 4)][4 * (i % (C / 4))], Rsl + (size_t)(i / (C / 4)) * D + 4 * (i % (C / 4)));
    else if (i % 8 == 0) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(Rsl + 4 * i));
  }
  cp_async_commit();

  // ---- tail scores (log2 domain)
  constexpr float LOG2E = 1.4426950408889634f;
  if (n_tail > 0) {
    if (npc > 0 || n_rawk > W) { cp_async_wait<1>(); __syncthreads(); }
    if (warp < npc) {   // packed keys: one warp per window, on the tensor cores
      uint2 qreg[16];
#pragma unroll
      for (int r = 0; r < 16; r++) qreg[r] = make_uint2(sm.qhi[r >> 2][lane][r & 3], sm.qlo[r >> 2][lane][r & 3]);
      const float fsc = sm.fsc[lane >> 2];
      unsigned char* st = af.img[warp];
      if (FMT == FMT_MXFP4) {
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
        for (int e2 = 0; e2 < 2; e2++) af.tsc[warp * W + 8 * nu + 2 * t + e2][g] = g < G ? sc[nu][e2] : -INFINITY;
    }
    for (int i = tid; i < n_rawk * GP; i += NTHREADS) {   // raw keys: a token and a head per thread, four sums
      const int tok = i / GP, j = i % GP;
      float s = -INFINITY;
      if (j < G) {
        const __half* krow = tok < W ? sm.k0[tok] : af.k[tok - W];
        float a4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int k = 0; k < D; k += 8) {
          const uint4 kv = *reinterpret_cast<const uint4*>(krow + k), qv = *reinterpret_cast<const uint4*>(&sm.q[j][k]);
          const uint32_t kx[4] = {kv.x, kv.y, kv.z, kv.w}, qx[4] = {qv.x, qv.y, qv.z, qv.w};
#pragma unroll
          for (int u = 0; u < 4; u++) {
            const float2 kf = __half22float2(u2h(kx[u])), qf = __half22float2(u2h(qx[u]));
            a4[u] = fmaf(qf.x, kf.x, a4[u]);
            a4[u] = fmaf(qf.y, kf.y, a4[u]);
          }
        }
        s = ((a4[0] + a4[1]) + (a4[2] + a4[3])) * P.sm_scale * LOG2E;
      }
      af.tsc[npc * W + tok][j] = s;
    }
  }
  cluster.barrier_wait();     // (acquire) all pieces of the unit and their headers are there
  __syncthreads();            // (and the tail scores)

  // ---- softmax bookkeeping: thread = (head j, stripe of 48)
  {
    const int j = tid & (GP - 1), stripe = tid / GP;
    float M = -INFINITY;
    for (int p = stripe; p < n_meta; p += NTHREADS / GP) M = fmaxf(M, sm.meta[p].m[j]);
    for (int i = stripe; i < n_tail; i += NTHREADS / GP) M = fmaxf(M, af.tsc[i][j]);
    M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 8));
    M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, 16));
    if (lane < GP) af.red[warp][j] = M;
    __syncthreads();
    M = af.red[0][j];
#pragma unroll
    for (int w = 1; w < NWARP; w++) M = fmaxf(M, af.red[w][j]);
    __syncthreads();
    float L = 0.f;
    for (int p = stripe; p < n_meta; p += NTHREADS / GP) {
      const float pm = sm.meta[p].m[j];
      const float f = pm == -INFINITY ? 0.f : exp2f(pm - M);
      af.fac[p][j] = f;
      L += sm.meta[p].l[j] * f;
    }
    for (int i = stripe; i < n_tail; i += NTHREADS / GP) {
      const float x = exp2f(af.tsc[i][j] - M);   // 0 for the heads beyond the group (-inf scores)
      af.tsc[i][j] = x;
      L += x;
    }
    L += __shfl_xor_sync(0xffffffffu, L, 8);
    L += __shfl_xor_sync(0xffffffffu, L, 16);
    if (lane < GP) af.red[warp][j] = L;
    __syncthreads();
    if (tid < GP) {
      float s = 0.f;
      for (int w = 0; w < NWARP; w++) s += af.red[w][tid];
      af.L[tid] = s;
    }
  }
  // ---- merge of the pieces for channels [rank * C, rank * C + C): item = (modality, m-tile, lane), a float4 of the piece
  // = channels g and g + 8 of the tile for heads 2 t and 2 t + 1 (clusters of 16: half a tile, one of the two channels)
  {
    constexpr int MT = C >= 16 ? C / 16 : 1, ITEMS = 3 * MT * 32, SHARES = ITEMS < NTHREADS ? NTHREADS / ITEMS : 1;
    static_assert(NTHREADS % ITEMS == 0 || ITEMS % NTHREADS == 0, "whole shares");
    const int share = tid / ITEMS;
    const int used = CS == 1 ? pieces_of(at) : at.used;
#pragma unroll
    for (int it0 = 0; it0 < ITEMS; it0 += NTHREADS) {        // (one round, two for a single block)
      const int it = ITEMS < NTHREADS ? tid % ITEMS : tid + it0;
      const int L32 = it & 31, mt = (it >> 5) % MT, m = it / (32 * MT);
      const int mu = C >= 16 ? rank * MT + mt : rank / 2;
      const int j0 = 2 * (L32 & 3);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      constexpr int IN_FLIGHT = 12;   // loads of a thread fetched together: the pieces come from L2
      for (int p0 = share; p0 < used; p0 += IN_FLIGHT * SHARES) {
        float4 x[IN_FLIGHT];
#pragma unroll
        for (int i = 0; i < IN_FLIGHT; i++) {
          const int p = p0 + i * SHARES;
          const bool have = p < used && ((sm.meta[p < used ? p : 0].held >> m) & 1);
          x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (have) x[i] = __ldcg(&pieces[p].frag[m][mu][L32]);
        }
#pragma unroll
        for (int i = 0; i < IN_FLIGHT; i++) {
          const int p = min(p0 + i * SHARES, used - 1);
          const float2 f = *reinterpret_cast<const float2*>(&af.fac[p][j0]);
          v.x = fmaf(x[i].x, f.x, v.x); v.y = fmaf(x[i].y, f.y, v.y); v.z = fmaf(x[i].z, f.x, v.z); v.w = fmaf(x[i].w, f.y, v.w);
        }
      }
      if (SHARES > 1) {
        af.part[tid] = v;
        __syncthreads();
        if (tid < ITEMS)
          for (int q = 1; q < SHARES; q++) {
            const float4 x = af.part[q * ITEMS + tid];
            v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
          }
      }
      if (SHARES == 1 || tid < ITEMS) {
        constexpr float F = LEVEL_UNIT;
        const int ch = 16 * mu + (L32 >> 2);
        for (int r = 0; r < MS; r++) {   // to every merging CTA of the cluster
          float* dst = CS == 1 ? &af.vec[0][0] : cluster.map_shared_rank(&af.vec[0][0], r);
          if (C >= 16 || (rank & 1) == 0) *reinterpret_cast<float2*>(dst + (m * D + ch) * GP + j0) = make_float2(v.x * F, v.y * F);
          if (C >= 16 || (rank & 1) == 1) *reinterpret_cast<float2*>(dst + (m * D + ch + 8) * GP + j0) = make_float2(v.z * F, v.w * F);
        }
      }
    }
  }
  cluster.sync();
  cp_async_wait<0>();
  __syncthreads();   // matrices and value rows have landed

  // ---- out[j][c] = (raw[j][c] + sum_r R[r][c] vec[r][j]) / L: thread = (two columns, slice of rows), all heads
  {
    constexpr int KS = SM::KS, ROWS = 3 * D / KS;
    static_assert(KS * ROWS == 3 * D, "whole slices");
    const int c = 2 * (tid % (C / 2)), ks = tid / (C / 2);
    float2 o[GP];
#pragma unroll
    for (int j = 0; j < GP; j++) o[j] = make_float2(0.f, 0.f);
    auto add_row = [&](float2 x, const float* w) {
      const float4 a = *reinterpret_cast<const float4*>(w), bq = *reinterpret_cast<const float4*>(w + 4);
      const float wj[GP] = {a.x, a.y, a.z, a.w, bq.x, bq.y, bq.z, bq.w};
#pragma unroll
      for (int j = 0; j < GP; j++) { o[j].x = fmaf(x.x, wj[j], o[j].x); o[j].y = fmaf(x.y, wj[j], o[j].y); }
    };
    if (SM::STAGED) {
#pragma unroll 8
      for (int r = ks * ROWS; r < (ks + 1) * ROWS; r++) add_row(*reinterpret_cast<const float2*>(&af.R[r][c]), af.vec[r]);
      for (int i = ks; i < n_tail; i += KS)   // raw value rows
        add_row(__half22float2(*reinterpret_cast<const __half2*>(&af.v[i][c])), af.tsc[i]);
    } else {
#pragma unroll 16
      for (int r = ks * ROWS; r < (ks + 1) * ROWS; r++) add_row(__ldg(reinterpret_cast<const float2*>(Rsl + (size_t)r * D + c)), af.vec[r]);
#pragma unroll 4
      for (int i = ks; i < n_tail; i += KS)
        add_row(__half22float2(*reinterpret_cast<const __half2*>(vt + cv.v_slot(v_pk + i) * D + c)), af.tsc[i]);
    }
#pragma unroll
    for (int j = 0; j < GP; j++) *reinterpret_cast<float2*>(&af.prod[ks][j][c]) = o[j];
    __syncthreads();
    for (int i = tid; i < G * C; i += NTHREADS) {
      const int j = i / C, cc = i % C;
      float s = 0.f;
#pragma unroll 8
      for (int k = 0; k < KS; k++) s += af.prod[k][j][cc];
      const float L = af.L[j];
      P.out[(((size_t)li * cv.batch + b) * cv.n_q_heads + h * G + j) * D + rank * C + cc] = L > 0.f ? s / L : 0.f;
    }
  }
}

template <int FMT, int CS>
static void small_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& at, int units) {
  cfg = {};
  cfg.gridDim = dim3(units * CS);
  cfg.blockDim = dim3(NTHREADS);
  cfg.dynamicSmemBytes = sizeof(SmallSmem<FMT, CS>);
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = CS; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
}

// clusters of this size the current device runs at once (0 if it cannot run them); looked up once per device and thread
template <int FMT, int CS>
static int small_clusters() {
  static_assert(sizeof(SmallSmem<FMT, CS>) <= 227 * 1024, "shared memory of one CTA");
  static thread_local int cached_dev = -1, cached = 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (dev == cached_dev) return cached;
  cudaError_t e = cudaFuncSetAttribute(k_decode_small<FMT, CS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem<FMT, CS>));
  if (e == cudaSuccess && CS > 8) e = cudaFuncSetAttribute(k_decode_small<FMT, CS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  int n = 0;
  if (e == cudaSuccess) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    small_config<FMT, CS>(cfg, at, 1);
    e = cudaOccupancyMaxActiveClusters(&n, k_decode_small<FMT, CS>, &cfg);
  }
  if (e != cudaSuccess) { (void)cudaGetLastError(); n = 0; }   // the split-K kernel takes the call
  cached = n;
  cached_dev = dev;
  return n;
}

template <int FMT, int CS>
static cudaError_t small_launch(const DecodeParams& P, int units, cudaStream_t s) {
  return launch_dependent(k_decode_small<FMT, CS>, dim3(units * CS), NTHREADS, sizeof(SmallSmem<FMT, CS>), s, CS, P);
}

// Cluster size for a call, 0 if the split-K pair should take it: whichever of the estimates below is least.  A cluster per
// unit, in waves of as many as run at once (on this GPU 7 clusters of 16, 15 of 8, 22 of 6, 33 of 4, 74 of 2, 148 blocks: a cluster
// stays inside one of eight groups of SMs): 11.5 us a wave and 2.1 us per window of a warp.  The pair: 31 us, 2 us per window
// of a warp with the windows balanced over all warps, 0.04 us per unit in the combine kernel.  Fitted to calls of 1 to 28
// layers, 1 to 16 sequences, 1 to 8 heads and 200 to 32768 tokens with the pieces not yet dealt out and the combine kernel's product
// on CUDA cores; both ways have become faster since (the smallest call takes 11.3 us of the 13.6 that this says) and the
// constants have not been fitted again.  Where a unit's windows spread over many blocks the pair costs
// more than this says, its combine kernel merging that many partials per unit (one unit of 131072 tokens: 36 us estimated, 214
// measured; four units: 50 and 75).  The host knows the capacity, not the lengths, and takes sequences to be full: a cache mostly
// empty goes the way it would go full.
// Clusters of six are for the 16 units of a layer of 4 sequences x 4 heads and a few more, one too many for clusters of eight: all six
// blocks walk, four of them merge.  Of up to four windows, which one block walks, four blocks make 0.4 us less.
template <int FMT>
static int small_cluster(long long units, long long windows, long long piece_slots) {
  constexpr int SIZES = 6;
  const int size[SIZES] = {1, 2, 4, 6, 8, 16};
  const int fit[SIZES] = {small_clusters<FMT, 1>(), small_clusters<FMT, 2>(), small_clusters<FMT, 4>(), small_clusters<FMT, 6>(), small_clusters<FMT, 8>(), small_clusters<FMT, 16>()};
  int best = 0;
  double best_cost = 31.0 + 2.0 * (double)units * (double)windows / ((double)sm_count() * NWARP) + 0.04 * (double)units;
  for (int i = SIZES - 1; i >= 0; i--) {   // (of equals the largest cluster)
    if (fit[i] <= 0 || units * size[i] * NWARP > piece_slots) continue;   // the warps' pieces have to fit the scratch
    if (size[i] == 6 && windows <= 4) continue;
    const double waves = (double)((units + fit[i] - 1) / fit[i]), walk = (double)((windows + NWARP * size[i] - 1) / (NWARP * size[i]));
    const double cost = waves * (11.5 + 2.1 * walk);
    if (cost < best_cost) { best_cost = cost; best = size[i]; }
  }
  return best;
}

int decode_small_cluster(const CacheView& cv, int layer_count, long long piece_slots) {
  const long long units = (long long)layer_count * cv.batch * cv.n_kv_heads, windows = cv.capacity / W;
  return cv.fmt == FMT_MXFP4 ? small_cluster<FMT_MXFP4>(units, windows, piece_slots) : small_cluster<FMT_FP16>(units, windows, piece_slots);
}

template <int CS>
static cudaError_t small_format(const DecodeParams& P, int units, cudaStream_t s) {
  return P.cv.fmt == FMT_MXFP4 ? small_launch<FMT_MXFP4, CS>(P, units, s) : small_launch<FMT_FP16, CS>(P, units, s);
}

okq_status launch_decode_small(const DecodeParams& P, int cs, cudaStream_t s) {
  const int units = P.layer_count * P.cv.batch * P.cv.n_kv_heads;
  const cudaError_t e = cs == 16 ? small_format<16>(P, units, s) : cs == 8 ? small_format<8>(P, units, s) : cs == 6 ? small_format<6>(P, units, s)
                      : cs == 4 ? small_format<4>(P, units, s) : cs == 2 ? small_format<2>(P, units, s) : small_format<1>(P, units, s);
  if (e != cudaSuccess) { set_last_cuda_error((int)e); return OKQ_ERR_CUDA; }
  return OKQ_OK;
}

}  // namespace okq
