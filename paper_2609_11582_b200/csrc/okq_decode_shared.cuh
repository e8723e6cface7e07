// Types shared by the two decode implementations (CUDA-core and tensor-core).
#pragma once
#include "okq_common.cuh"

namespace okq {

constexpr int GP = OKQ_MAX_GROUP;   // padded GQA group
constexpr int NACC = 4;             // 3 modality accumulators + 1 raw (tail) accumulator
constexpr int MAX_ENTRIES = 1024;   // (layer, sequence) pairs one launch can cover

// CUDA-core kernel: one per (sequence, head, split)
struct Partial {
  float m[GP];
  float l[GP];
  float acc[NACC][GP][D];
};

// tensor-core kernel: one per (CTA, (sequence, head)) overlap; accumulators stay in
// mma fragment order [modality][register][lane]
struct PartialF {
  float m[GP];          // running maximum per head (log2 domain)
  float l[GP];          // sum of exp2(score - m)
  float Sp[3][32];      // per modality: sum of p * vnorm, four lane-partials per head
  float frag[3][32][32];
};

// unit of PartialF's accumulators: a value sum is PARTIAL_ACC_SCALE * frag + (codebook offset) * (sum of Sp)
constexpr float PARTIAL_ACC_SCALE = (CB_OUTER - CB_INNER) * 262144.0f;  // (b - a) * 2^18

// mma.sync kernel: what one warp accumulated over its part of one (sequence, head); the CTA merges its warps'
// pieces into the PartialF records at the end of the launch
constexpr int DECODE_WARPS = 12;    // warps per CTA
struct WarpPiece {
  float4 frag[3][8][32];   // [modality][m-tile][lane]: the tile's four accumulator registers
  float wm[GP], wl[GP];    // reference (log2 domain) of everything in the piece, sum of exp2(score - reference)
  int mask;                // modalities the piece holds (bit m); the other modalities' sums are not written
  int pad[3];
};

struct DecodeParams {
  CacheView cv;
  int layer0, layer_count, n_splits, group;
  const __half* q;     // [layer_count][batch][n_q_heads][128]
  const float* signs;  // [layer_count][128]
  const float* R;      // [layer_count][n_R][3][128][128]
  int n_R;
  float sm_scale;
  Partial* partials;   // CUDA-core path: [layer_count*batch*n_kv_heads][n_splits]
  PartialF* partials_f;  // tensor-core path: [n_units + n_cta]
  WarpPiece* pieces;     // tensor-core path: [n_units + DECODE_WARPS * n_cta] at least
  long long piece_slots; // how many there is room for
  float* out;          // [layer_count][batch][n_q_heads][128]
};

// prefix[e] = number of windows (all KV heads) of the (layer, sequence) entries before e,
// entries ordered layer-major; returns the total.  Called by every thread of the block.
__device__ inline int block_prefix(const CacheView& cv, int layer0, int n_entries, int* prefix) {
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    const int chunk = (n_entries + 31) / 32;
    const int e0 = min(n_entries, lane * chunk), e1 = min(n_entries, e0 + chunk);
    int sum = 0;
    for (int e = e0; e < e1; e++) sum += (cv.v_packed(cv.seq_len[(size_t)layer0 * cv.batch + e]) / W) * cv.n_kv_heads;
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      int v = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += v;
    }
    int run = incl - sum;
    for (int e = e0; e < e1; e++) {
      prefix[e] = run;
      run += (cv.v_packed(cv.seq_len[(size_t)layer0 * cv.batch + e]) / W) * cv.n_kv_heads;
    }
    if (lane == 31) prefix[n_entries] = incl;
  }
  __syncthreads();
  return prefix[n_entries];
}

// tcgen05 split-K kernel (fp16 metadata): fills partials_f exactly where launch_decode_mma's own split kernel would
okq_status launch_decode_tc(const DecodeParams& P, int n_cta, cudaStream_t s);
// which split-K kernel launch_decode_mma uses: 0 = the tcgen05 kernel (fp16 metadata), 1 = the mma.sync kernel
extern int g_decode_impl;

// one-launch form for few (sequence, head) units: cluster size it would use for a call (0: the split-K pair), launch
int decode_small_cluster(const CacheView& cv, int layer_count, long long piece_slots);
okq_status launch_decode_small(const DecodeParams& P, int cs, cudaStream_t s);

// how launch_decode_mma takes a call: blocks of a cluster of the one-launch kernel, or the pair's OKQ_PLAN_PAIR_*
int decode_plan(const DecodeParams& P, int n_cta);
// launches the tensor-core split kernel (bracketed by the optional events) and its combine kernel
okq_status launch_decode_mma(const DecodeParams& P, int n_cta, cudaStream_t s, cudaEvent_t before, cudaEvent_t after);

}  // namespace okq
