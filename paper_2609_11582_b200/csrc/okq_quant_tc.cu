// Bulk value quantiser with the per-modality rotation on the 5th-generation tensor cores
// (Eq. 6 then Eq. 3 for whole prefill chunks).
//
// z = R_m v is a dense [tokens x 128] x [128 x 128] contraction.  A CTA takes tiles of 128
// consecutive tokens (four windows) of one (sequence, KV head):
// three roles that meet only at mbarriers:
//   * a loader warp brings each tile of fp16 values with two TMA tensor copies (64 channels x 128
//     tokens, 128-byte swizzle: the K-major layout tcgen05.mma reads) plus the tile's modality bytes
//     (two tile buffers, "full" / "empty" barriers); the values are the B operand as they are (exact);
//   * an MMA warp issues the tensor-core work of a tile as soon as it has landed and one of the two
//     accumulator sets in tensor memory is free ("mma_done" / "acc_free" barriers);
//   * sixteen worker warps compute the norms and turn accumulators into packed codes.
// In detail:
//   * R_m (fp32) is split into two fp16 matrices R_hi + R_lo (the A operand), kept in shared memory
//     while the modality does not change; 16 tcgen05.mma (M = 128, K = 16, N = the windows of the
//     tile that hold the modality) accumulate z^T = R_hi v^T + R_lo v^T in fp32 in tensor memory:
//     lane = output channel, column = token;
//   * in the epilogue a thread owns one channel and reads the 32 tokens of one window with one
//     tcgen05.ld: exactly the (channel, 8 tokens) groups a word of the decode kernel's value-code
//     layout holds, so the words are built in registers (one lane exchange joins the two channels
//     of a word).  The code, the number of thresholds {-T, 0, T} below z / norm, is taken
//     arithmetically: v = sat(2/3 - z / (3 T norm)), k = floor(3 v) with a round-down fused
//     multiply-add against 1.5 * 2^23, code = 3 - k: three full-rate instructions per element.
// The split leaves a relative error of about 2^-22 on z and the tensor cores' accumulation about
// 1e-6, so the arithmetic code is only trusted where z / norm is further than 2^-18 from every
// threshold (the code is taken twice, with the coordinate moved down and up by that band); the few
// coordinates in the band (about 1e-4 of them) are listed and recomputed at the end of the kernel, one per warp at
// a time, with the exact fused-multiply-add chain of the reference arithmetic over the value row, read again from
// global memory; the code in the record is then patched.  Codes and norms (exact summation tree) are therefore bit-identical to the exact path.
// The band is good for rotations.  If a matrix row is longer than 2 (the errors grow with it, and entries may not even fit fp16)
// or a value longer than fp16 can say, the block takes all its coordinates through the exact chain at the end.
//
// The same kernel writes the value codes of the bit-width ladder (BITS = 2, 3 or 4: token-major bit streams): a table of 32
// bins over the coordinate, each with at most one threshold of the codebook, gives (threshold, code below it) in one
// look-up, the coordinates within the band go the same way as above, and a warp transposes its 32 x 32 codes through
// shared memory and stores 4 BITS bytes per token.  8 sequences x 4 heads x 8192 tokens at 3 bits, keys and values:
// 1282 us with one block per window evaluating the exact chain, 146 us now.
//
// Every wait on an mbarrier is bounded; on a timeout the kernel records OKQ_ERR_TIMEOUT in the
// cache's status word (the ladder, which has none: NaN in the value norms of the block's tokens, which decode hands on), stops
// issuing work, frees its tensor memory and returns.
#include "okq_common.cuh"
#include "okq_device.cuh"
#include "okq_ladder.cuh"
#include "okq_quant_tail.cuh"
#include "okq_tc.cuh"

namespace okq {

namespace {

constexpr int TILE = 128;                 // tokens per tile
constexpr int NT = 512;                   // worker threads per CTA: 16 warps, four per tensor-memory lane quarter
constexpr int NT_ALL = NT + 64;           // + the MMA warp (16) and the loader warp (17)
constexpr int TILE_BYTES = TILE * D * 2;  // 32 KB: one fp16 operand tile
constexpr float NEG_INV_3T = -1.0f / (3.0f * CB_THRESH);
constexpr float TWO_THIRDS = 2.0f / 3.0f;          // rounds up: a zero coordinate gives floor(3 v) = 2, code 1
// The code is taken twice, with the coordinate moved down and up by BAND (in units of z / norm: far above the
// rounding noise of the tensor-core product, about 1e-6); where the two disagree the coordinate lies that close to a
// threshold and is recomputed with the exact fused-multiply-add chain of the reference arithmetic.
constexpr float BAND = 0x1p-18f;
constexpr float BAND_V = BAND / (3.0f * CB_THRESH);
constexpr float NORM_MAX = 65504.0f;               // of a stored norm; the value itself may be sqrt(128) times as long
constexpr float ROW_SQ_MAX = 4.0f;                 // squared length of the matrix rows that BAND is good for
constexpr float FLOOR_MAGIC = 12582912.0f;         // 1.5 * 2^23: unit in the last place 1, bits 0x4B400000
// sum over the eight fields (bit 16*e + 2*j) of a word of the magic bits shifted to the field, modulo 2^32
constexpr uint32_t magic_sum() {
  uint32_t s = 0;
  for (int e = 0; e < 2; e++)
    for (int j = 0; j < 4; j++) s += 0x4B400000u << (16 * e + 2 * j);
  return s;
}
constexpr uint32_t MAGIC_SUM = magic_sum();

// A coordinate too close to a threshold for the tensor-core product to decide: recomputed with the reference
// arithmetic at the end of the kernel (its code is patched in the record), so that the tile pipeline never waits for
// the two rows this needs from global memory.
struct FixItem {
  uint32_t* word;        // code word of the record
  const __half* xrow;    // the token's value row (128 fp16)
  const float* rrow;     // row of the rotation matrix (128 fp32): output channel of the coordinate
  float inv;             // 1 / norm
  int bit;               // bit position of the field in the word
};

// bins of the code table: bin i covers [(i - 16.5) w, (i - 15.5) w); every width keeps all thresholds at least 0.13 w away
// from the edges, so a coordinate within the band of a threshold is always looked up in that threshold's bin
constexpr int BINS = 32;
__host__ __device__ constexpr float bin_width(int bits) { return bits == 2 ? 0.0078875f : bits == 3 ? 0.0152875f : 0.02097845f; }

template <int BITS> struct LadderSmem {
  float2 bin[BINS];                                  // threshold in the bin (+inf: none), code below it (integer bits)
  __align__(4) unsigned char code[16][W][36];        // per worker warp: [token][channel of its 32], 9-word rows
};
template <> struct LadderSmem<0> {};

template <int BITS> struct TcSmem {
  static constexpr int FIX_MAX = BITS ? 128 : 256;
  LadderSmem<BITS> lad;
  __align__(1024) unsigned char a[2][TILE_BYTES];      // value tiles (double buffered)
  __align__(1024) unsigned char b[2][2][TILE_BYTES];   // two resident matrices, each as R_hi, R_lo
  __align__(16) float part[2][4][TILE];                // per token: sum of squares of channels [32 q, 32 q + 32)
  __align__(16) float c3[16][W];                       // per worker warp: -1 / (3 T norm) of its window's tokens
  __align__(16) float inv[16][W];                      // per worker warp: 1 / norm of its window's tokens (0 for a zero vector)
  __align__(4) unsigned char mod[2][TILE];             // modality per token of a tile (255 = no token)
  __align__(8) unsigned long long full[2];             // 1 arrival + 32 KB of TMA bytes: tile and modality bytes are in
  __align__(8) unsigned long long empty[2];            // 16 arrivals: every worker warp is done with the buffer
  __align__(8) unsigned long long mma_done[2];         // 1 arrival (tcgen05.commit): accumulator set complete
  __align__(8) unsigned long long acc_free[2];         // 16 arrivals: every worker warp has read the accumulator set
  __align__(8) unsigned long long part_ready[2][4];    // 4 arrivals: a window's four warps have written its partial norms
  __align__(8) unsigned long long slot_ready;          // 16 arrivals: every worker warp has written its share of a rotation matrix
  uint32_t tmem_slot;
  FixItem fix[FIX_MAX];
  int fix_count;
  int redo;                                            // BAND was not good for one of the block's matrices or values
  long long limit;                                     // SM clocks a wait may take
  volatile int abort;                                  // set by a role whose bounded wait ran out
  volatile int tmem_busy;                              // set if products may still be in flight at the end (tensor memory is then not released)
};

// shared-memory matrix descriptor: no swizzle, K-major; core matrices of 8 rows x 16 bytes,
// `lbo` bytes between the two 8-element K chunks of one MMA, `sbo` bytes between 8-row groups
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3fff) | ((uint64_t)((lbo >> 4) & 0x3fff) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3fff) << 32) | ((uint64_t)1 << 46);
}

// byte offset of element (row r, column k) of a 128 x 128 fp16 operand tile
__device__ __forceinline__ uint32_t tile_off(int r, int k) {
  return (uint32_t)((k >> 3) * 2048 + (r >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// byte offset of the 16-byte chunk holding channels [8 kc, 8 kc + 8) of token row r in a TMA-written value
// tile: two halves of 64 channels, 128 bytes per row, chunk index xor-ed with the row inside its 8-row group
__device__ __forceinline__ uint32_t vtile_off(int r, int kc) {
  return (uint32_t)((kc >> 3) * (TILE_BYTES / 2) + r * 128 + (((kc & 7) ^ (r & 7)) << 4));
}

// the reference arithmetic: one fused-multiply-add chain, input index ascending
__device__ __noinline__ float exact_chain(const float* rrow, const __half* xrow) {
  float a = 0.0f;
#pragma unroll 4
  for (int kc = 0; kc < 16; kc++) {
    const uint4 raw = __ldg(reinterpret_cast<const uint4*>(xrow) + kc);
    const __half2* h2 = reinterpret_cast<const __half2*>(&raw);
    const float4 r0 = __ldg(reinterpret_cast<const float4*>(rrow) + 2 * kc), r1 = __ldg(reinterpret_cast<const float4*>(rrow) + 2 * kc + 1);
    const float2 x0 = __half22float2(h2[0]), x1 = __half22float2(h2[1]), x2 = __half22float2(h2[2]), x3 = __half22float2(h2[3]);
    a = __fmaf_rn(r0.x, x0.x, a); a = __fmaf_rn(r0.y, x0.y, a); a = __fmaf_rn(r0.z, x1.x, a); a = __fmaf_rn(r0.w, x1.y, a);
    a = __fmaf_rn(r1.x, x2.x, a); a = __fmaf_rn(r1.y, x2.y, a); a = __fmaf_rn(r1.z, x3.x, a); a = __fmaf_rn(r1.w, x3.y, a);
  }
  return a;
}

// R_m (fp32) as two fp16 operand tiles in slot `slot`, by the NT worker threads: all of a thread's loads in flight together.
// A warp takes 8 rows, 32 columns at a time: 128-byte pieces of a row in global memory, eight consecutive 16-byte rows of a core
// matrix per quarter-warp in shared memory (lanes along a row instead put eight stores on the same banks: 6000 cycles).
template <int BITS>
__device__ __forceinline__ void write_matrix(TcSmem<BITS>& sm, const float* Rm, int slot, int tid) {
  constexpr int N = D * D / 8 / NT;
  float4 x[N][2];
#pragma unroll
  for (int i = 0; i < N; i++) {
    const int n = 8 * (tid >> 5) + (tid & 7), kc = 4 * i + ((tid >> 3) & 3);
    const float* src = Rm + n * D + kc * 8;
    x[i][0] = __ldg(reinterpret_cast<const float4*>(src));
    x[i][1] = __ldg(reinterpret_cast<const float4*>(src) + 1);
  }
  static_assert(N == 4 && NT / 32 == D / 8, "a warp has whole rows");
  float sq = 0.0f;
#pragma unroll
  for (int i = 0; i < N; i++) {
    const int n = 8 * (tid >> 5) + (tid & 7), kc = 4 * i + ((tid >> 3) & 3);
    const float xs[8] = {x[i][0].x, x[i][0].y, x[i][0].z, x[i][0].w, x[i][1].x, x[i][1].y, x[i][1].z, x[i][1].w};
    __align__(16) __half hi[8], lo[8];
#pragma unroll
    for (int u = 0; u < 8; u++) {
      sq = fmaf(xs[u], xs[u], sq);
      hi[u] = __float2half_rn(xs[u]);
      lo[u] = __float2half_rn(xs[u] - __half2float(hi[u]));
    }
    const uint32_t off = tile_off(n, kc * 8);
    *reinterpret_cast<uint4*>(sm.b[slot][0] + off) = *reinterpret_cast<const uint4*>(hi);
    *reinterpret_cast<uint4*>(sm.b[slot][1] + off) = *reinterpret_cast<const uint4*>(lo);
  }
  sq += __shfl_xor_sync(0xffffffffu, sq, 8);
  sq += __shfl_xor_sync(0xffffffffu, sq, 16);
  if (!(sq <= ROW_SQ_MAX)) sm.redo = 1;   // (not a number either)
}

// The jobs of a tile, derived identically by the MMA warp and every worker warp from the tile's modality
// bytes: `present` = modalities in the tile (bit m); a job takes at most two of them, so a tile with all
// three needs two jobs.  winmask[m] = windows of the tile (bit w) that hold modality m.
struct TileMods {
  unsigned present;
  unsigned winmask[3];
};
__device__ __forceinline__ TileMods tile_mods(uint32_t m4) {   // 4 tokens per lane, window lane >> 3
  TileMods t;
  t.present = 0;
#pragma unroll
  for (int mm = 0; mm < 3; mm++) {
    const bool has = ((m4 & 0xffu) == mm) | (((m4 >> 8) & 0xffu) == mm) | (((m4 >> 16) & 0xffu) == mm) | ((m4 >> 24) == mm);
    const unsigned bal = __ballot_sync(0xffffffffu, has);
    t.winmask[mm] = ((bal & 0xffu) ? 1u : 0u) | ((bal & 0xff00u) ? 2u : 0u) | ((bal & 0xff0000u) ? 4u : 0u) | ((bal >> 24) ? 8u : 0u);
    if (bal) t.present |= 1u << mm;
  }
  return t;
}
__device__ __forceinline__ TileMods tile_mods(const unsigned char* mod, int lane) {
  return tile_mods(reinterpret_cast<const uint32_t*>(mod)[lane]);
}
// The tile's jobs in scalars (arrays indexed by a run-time value would live in local memory: 1000 cycles per tile and warp):
// job 0 takes the first two modalities, job 1 the third one, if there is one.
struct TileJobs {
  int n_jobs, n0, m0, m1;
  __device__ __forceinline__ explicit TileJobs(unsigned present) {
    const unsigned rest = present & (present - 1u);
    n_jobs = present == 0u ? 0 : (present == 7u ? 2 : 1);
    n0 = rest ? 2 : 1;
    m0 = __ffs(present) - 1;
    m1 = __ffs(rest) - 1;
  }
  __device__ __forceinline__ int count(int jt) const { return jt ? 1 : n0; }
  __device__ __forceinline__ int mod(int jt, int mi) const { return jt ? 2 : (mi ? m1 : m0); }
};

// The two resident rotation matrices (hi/lo pairs), tracked identically by the MMA warp and the worker warps.
// plan() assigns the job's matrices to slots and says which have to be written first; a matrix goes to the
// slot the job's other matrix does not use, else to the one that was not used last.
struct Slots {
  int k0 = -1, k1 = -1;   // (rotation set * 3 + modality) held by each slot
  int last = 0;
  int sa = 0, sb = 0;     // slots of the planned job's matrices
  bool na = false, nb = false;   // whether they have to be written
  __device__ __forceinline__ bool plan(int nm, int ka, int kb) {
    sa = k0 == ka ? 0 : (k1 == ka ? 1 : -1);
    sb = nm == 2 ? (k0 == kb ? 0 : (k1 == kb ? 1 : -1)) : -1;
    na = sa < 0;
    nb = nm == 2 && sb < 0;
    if (na) {
      sa = (sb >= 0 ? sb : last) ^ 1;
      if (sa) k1 = ka; else k0 = ka;
    }
    if (nb) {
      sb = sa ^ 1;
      if (sb) k1 = kb; else k0 = kb;
    }
    last = nm == 2 ? sb : sa;
    return na || nb;
  }
};

}  // namespace

// persistent grid, NT_ALL threads.  Tiles are numbered (b, h, tile-in-sequence), tile = 4 windows; a CTA
// owns a contiguous range of them.  A "job" is one tile and at most two of the modalities present in it
// (one accumulator of 128 columns each); jobs alternate between two accumulator sets in tensor memory.
// BITS = 0: window records of `cv` (2 bits); 2, 3, 4: the canonical arrays of `lv` (cv: shape and modality only).
template <int BITS>
__global__ void __launch_bounds__(NT_ALL, 1) k_quantize_values_tc(const __grid_constant__ CUtensorMap vmap, CacheView cv, LadderView lv, int layer,
                                                             const unsigned char* __restrict__ modality, int n_tokens,
                                                             int n_win, const float* __restrict__ R, int n_R,
                                                             const __half* __restrict__ vrows, long long vs_b, long long vs_h,
                                                             long long vs_t, long long wait_limit, int skip_tile) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  using SM = TcSmem<BITS>;
  constexpr int FIX_MAX = SM::FIX_MAX;
  SM& sm = *reinterpret_cast<SM*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if constexpr (BITS != 0) {
    if (tid < BINS) {
      const float lo = ((float)tid - 16.5f) * bin_width(BITS), hi = lo + bin_width(BITS);
      float th = INFINITY;
      int below = 0;
      for (int j = 0; j < (1 << BITS) - 1; j++) {
        const float x = c_thresholds[BITS - 2][j];
        if (x < lo) below++;
        else if (x < hi) th = x;
      }
      sm.lad.bin[tid] = make_float2(th, __int_as_float(below));
    }
  }
  const int tiles_per_unit = (n_win + 3) / 4;   // n_win: windows to pack (the schedule may keep recent tokens raw)
  const int n_tiles_all = tiles_per_unit * cv.n_kv_heads * cv.batch;
  // contiguous tile range of this CTA
  const int per_cta = (n_tiles_all + gridDim.x - 1) / gridDim.x;
  const int tile_begin = min(n_tiles_all, (int)blockIdx.x * per_cta);
  const int my_tiles = min(n_tiles_all, tile_begin + per_cta) - tile_begin;

  if (tid == 0) {
    for (int i = 0; i < 2; i++) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&sm.full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 16;\n" ::"r"(smem_u32(&sm.empty[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&sm.mma_done[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 16;\n" ::"r"(smem_u32(&sm.acc_free[i])));
      for (int w = 0; w < 4; w++) asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;\n" ::"r"(smem_u32(&sm.part_ready[i][w])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 16;\n" ::"r"(smem_u32(&sm.slot_ready)));
    sm.abort = 0;
    sm.tmem_busy = 0;
    sm.fix_count = 0;
    sm.redo = 0;
    sm.limit = wait_limit;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_u32(&sm.tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = sm.tmem_slot;
  depend_wait();

  // coordinates of the first tile; every role steps them without divisions afterwards
  int cb = 0, ch = 0, cwin0 = 0;
  if (my_tiles > 0) {
    cb = tile_begin / (tiles_per_unit * cv.n_kv_heads);
    const int rem = tile_begin - cb * tiles_per_unit * cv.n_kv_heads;
    ch = rem / tiles_per_unit;
    cwin0 = (rem - ch * tiles_per_unit) * 4;
  }
  auto step_coords = [&]() {
    cwin0 += 4;
    if (cwin0 >= tiles_per_unit * 4) { cwin0 = 0; if (++ch == cv.n_kv_heads) { ch = 0; cb++; } }
  };

  // modality bytes of the current tile's tokens 4 lane .. 4 lane + 3 (255: no token)
  auto tile_modality = [&]() -> uint32_t {
    const int rows = min(TILE, (n_win - cwin0) * W);
    uint32_t packed = 0;
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const int tok = 4 * lane + u;
      unsigned m = 255;
      if (tok < rows) { m = modality[(size_t)cb * n_tokens + (size_t)cwin0 * W + tok]; m = m > 2 ? 0 : m; }
      packed |= m << (8 * u);
    }
    return packed;
  };

  if (warp == 17) {
    // ------------------------------------------------------------------ loader warp
    // tile i of the range goes to buffer i & 1 once the buffer's previous tile (i - 2) has been released.
    // A lane carries the modality bytes of the tokens 4*lane .. 4*lane+3, fetched one tile ahead.
    auto fetch_mod = [&](int i) -> uint32_t { return i < my_tiles ? tile_modality() : 0xffffffffu; };
    uint32_t mod_cur = fetch_mod(0);
    int armed = 0;   // tiles whose copies have been issued
    for (int i = 0; i < my_tiles; i++) {
      const int buf = i & 1, fill = i >> 1;
      if (tile_begin + i == skip_tile) {   // testing aid: this tile never arrives, so that every role's wait runs out
        step_coords();
        mod_cur = fetch_mod(i + 1);
        continue;
      }
      if (fill >= 1 && !mbar_wait(sm, &sm.empty[buf], (uint32_t)(fill - 1) & 1u)) break;
      reinterpret_cast<uint32_t*>(sm.mod[buf])[lane] = mod_cur;
      __syncwarp();
      if (lane == 0) {
        // the arrival (release) publishes sm.mod; the phase completes when the 32 KB have landed.  Rows past
        // the end of the sequence are filled with zeros by the copy engine.
        const uint32_t bar = smem_u32(&sm.full[buf]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"((uint32_t)TILE_BYTES) : "memory");
#pragma unroll
        for (int half = 0; half < 2; half++)
          asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];\n"
                       ::"r"(smem_u32(sm.a[buf]) + half * (TILE_BYTES / 2)), "l"(reinterpret_cast<uint64_t>(&vmap)),
                         "r"(64 * half), "r"(cwin0 * W), "r"(ch), "r"(cb), "r"(bar) : "memory");
      }
      armed = i + 1;
      step_coords();
      mod_cur = fetch_mod(i + 1);
    }
    // with its tiles on their way: this CTA's share of the modality bytes and of the raw tail rows
    for (int bb = 0; bb < cv.batch; bb++) bulk_modality(cv, bb, modality, n_tokens, blockIdx.x * 32 + lane, gridDim.x * 32);
    if (BITS == 0)
      for (int u = blockIdx.x; u < cv.batch * cv.n_kv_heads; u += gridDim.x)
        bulk_tail_rows(cv, layer, u / cv.n_kv_heads, u % cv.n_kv_heads, vrows, vs_b, vs_h, vs_t, n_tokens, true, lane, 32);
    // after a timeout somewhere: no copy of this warp may still be landing when the block ends
    if (sm.abort)
      for (int i = max(0, armed - 2); i < armed; i++) mbar_drain(&sm.full[i & 1], (uint32_t)(i >> 1) & 1u);
  } else if (warp == 16) {
    // ------------------------------------------------------------------ MMA warp
    Slots slots;
    uint32_t jobidx = 0, refills = 0;
    bool dead = false;
    for (int i = 0; i < my_tiles && !dead; i++) {
      const int buf = i & 1;
      if (!mbar_wait(sm, &sm.full[buf], (uint32_t)(i >> 1) & 1u)) break;
      const TileMods tm = tile_mods(sm.mod[buf], lane);
      const TileJobs jobs(tm.present);
      for (int jt = 0; jt < jobs.n_jobs; jt++) {
        const int nm = jobs.count(jt);
        const uint32_t a = jobidx & 1u;
        if (jobidx >= 2 && !mbar_wait(sm, &sm.acc_free[a], ((jobidx >> 1) - 1u) & 1u)) { dead = true; break; }
        // resident rotation matrices: the worker warps write a missing one and report on slot_ready
        const int key0 = (n_R == 1 ? 0 : ch) * 3;
        if (slots.plan(nm, key0 + jobs.mod(jt, 0), key0 + jobs.mod(jt, 1))) {
          if (!mbar_wait(sm, &sm.slot_ready, refills & 1u)) { dead = true; break; }
          refills++;
        }
        if (elect_one()) {   // one thread of the converged warp: the compiler keeps the operands in uniform registers
          asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // the landed copies -> tensor-core reads
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          for (int mi = 0; mi < nm; mi++) {
            // the windows [w_lo, w_hi] of the tile that hold this modality are the N extent of the MMAs
            const int mod = jobs.mod(jt, mi), slot = mi ? slots.sb : slots.sa;
            const unsigned wm = mod == 0 ? tm.winmask[0] : (mod == 1 ? tm.winmask[1] : tm.winmask[2]);
            const int w_lo = __ffs(wm) - 1, w_hi = 31 - __clz(wm);
            const uint32_t n_ext = 32u * (uint32_t)(w_hi - w_lo + 1);
            const uint32_t idesc = (1u << 4) | ((n_ext >> 3) << 17) | ((128u >> 4) << 24);   // D fp32, A/B fp16 K-major, M = 128
            const uint32_t dcol = tmem + a * 256u + (uint32_t)mi * 128u + 32u * (uint32_t)w_lo;
            const uint64_t da0 = make_desc(smem_u32(sm.b[slot][0]), 2048, 128);                   // R: M = output channel
            const uint64_t da1 = make_desc(smem_u32(sm.b[slot][1]), 2048, 128);
            const uint64_t db0 = make_desc_sw128(smem_u32(sm.a[buf]) + 4096u * (uint32_t)w_lo);       // values: N = token
#pragma unroll
            for (int k = 0; k < 16; k++) {
              // next 16 input channels: 4096 bytes further in R; 32 bytes further inside a value row, the second
              // 64 channels in the tile's second half
              const uint64_t da = (k < 8 ? da0 : da1) + (uint64_t)((k & 7) * (4096 >> 4));
              const uint64_t db = db0 + (uint64_t)(((k & 3) * 32 + ((k >> 2) & 1) * (TILE_BYTES / 2)) >> 4);
              asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                           "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5}, p;\n\t}\n"
                           ::"r"(dcol), "l"(da), "l"(db), "r"(idesc), "r"(k ? 1u : 0u), "r"(0u) : "memory");
            }
          }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(&sm.mma_done[a])) : "memory");
        }
        __syncwarp();
        jobidx++;
      }
      step_coords();
    }
    // nothing may be in flight when tensor memory is released: the last committed job is waited for whatever the
    // abort flag says (every issued product belongs to a committed job); if even that does not answer, tensor
    // memory stays allocated
    if (jobidx >= 1 && !mbar_drain(&sm.mma_done[(jobidx - 1u) & 1u], ((jobidx - 1u) >> 1) & 1u)) sm.tmem_busy = 1;
  } else {
    // ------------------------------------------------------------------ worker warps
    // window ewq of every tile, together with the three other warps of the window and nobody else: norm role: its token
    // rows, channels [32 eq, 32 eq + 32); epilogue role: channels 32*eq + lane (the warp's tensor-memory lane quarter)
    const int eq = warp & 3, ewq = warp >> 2;
    // the rotation matrices on their way to L2 before the first tile says which one it needs
    for (int i = blockIdx.x * NT + tid; i < n_R * 3 * D * D / 32; i += gridDim.x * NT)
      asm volatile("prefetch.global.L2 [%0];\n" ::"l"(R + (size_t)i * 32));
    Slots slots;
    uint32_t jobidx = 0;
    bool dead = false;
    // A rotation matrix that a job needs is not resident: split R_m into fp16 hi + lo, laid out as the A
    // operand (row = output channel, K = input channel).  Every MMA issued so far has completed (this warp
    // has waited for each), and the job's own MMAs wait for slot_ready.
    auto bring_matrices = [&](const TileJobs& jobs, int jt) {
      const int key0 = (n_R == 1 ? 0 : ch) * 3;
      if (slots.plan(jobs.count(jt), key0 + jobs.mod(jt, 0), key0 + jobs.mod(jt, 1))) {
        if (slots.na) write_matrix<BITS>(sm, R + (size_t)(key0 + jobs.mod(jt, 0)) * D * D, slots.sa, tid);
        if (slots.nb) write_matrix<BITS>(sm, R + (size_t)(key0 + jobs.mod(jt, 1)) * D * D, slots.sb, tid);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // generic-proxy writes -> tensor-core reads
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.slot_ready);
      }
    };
    // the first job's matrices before anything else: they are the longest way of a block's start (15000 of 70000 cycles for seven
    // tiles), and behind the first tile's arrival and norms they came 5000 cycles later
    if (my_tiles > 0) bring_matrices(TileJobs(tile_mods(tile_modality()).present), 0);
    for (int i = 0; i < my_tiles && !dead; i++) {
      const int buf = i & 1;
      const uint32_t par = (uint32_t)(i >> 1) & 1u;
      if (!mbar_wait(sm, &sm.full[buf], par)) break;
      const TileMods tm = tile_mods(sm.mod[buf], lane);
      const TileJobs jobs(tm.present);
      const unsigned mymod = sm.mod[buf][32 * ewq + lane];   // token `lane` of this warp's window
      const int wins = min(4, n_win - cwin0);
      {
        // Sum of squares with the exact adjacent-pair tree, split so that shared-memory reads are free of bank
        // conflicts: a 16-byte chunk (8 channels) is three levels of the tree, the warp's four chunks two more;
        // the last two levels (p0 + p1) + (p2 + p3) follow below.
        const int row = 32 * ewq + lane, q = eq;
        float part[4];
#pragma unroll
        for (int c = 0; c < 4; c++) {
          const uint4 raw = *reinterpret_cast<const uint4*>(sm.a[buf] + vtile_off(row, 4 * q + c));
          const __half2* h2 = reinterpret_cast<const __half2*>(&raw);
          float2 x0 = __half22float2(h2[0]), x1 = __half22float2(h2[1]), x2 = __half22float2(h2[2]), x3 = __half22float2(h2[3]);
          float s0 = __fadd_rn(__fmul_rn(x0.x, x0.x), __fmul_rn(x0.y, x0.y));
          float s1 = __fadd_rn(__fmul_rn(x1.x, x1.x), __fmul_rn(x1.y, x1.y));
          float s2 = __fadd_rn(__fmul_rn(x2.x, x2.x), __fmul_rn(x2.y, x2.y));
          float s3 = __fadd_rn(__fmul_rn(x3.x, x3.x), __fmul_rn(x3.y, x3.y));
          part[c] = __fadd_rn(__fadd_rn(s0, s1), __fadd_rn(s2, s3));
        }
        sm.part[buf][q][row] = __fadd_rn(__fadd_rn(part[0], part[1]), __fadd_rn(part[2], part[3]));
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.part_ready[buf][ewq]);
      }
      if (!mbar_wait(sm, &sm.part_ready[buf][ewq], par)) break;
      [[maybe_unused]] unsigned nonzero = 0;   // tokens of the window that are not zero vectors
      if (ewq < wins) {
        // lane: norm of token `lane` of the window; the warp needs all 32 factors -1 / (3 T norm)
        const int tok = 32 * ewq + lane;
        const float sum = __fadd_rn(__fadd_rn(sm.part[buf][0][tok], sm.part[buf][1][tok]),
                                    __fadd_rn(sm.part[buf][2][tok], sm.part[buf][3][tok]));
        float n = __fsqrt_rn(sum);
        if (n > NORM_MAX) { n = NORM_MAX; sm.redo = 1; }
        const __half nh16 = __float2half_rn(n);
        const float nf = __half2float(nh16);
        if (eq == 0) {
          if (BITS == 0) reinterpret_cast<__half*>(cv.body(layer, cb, ch, cwin0 + ewq) + B_VNORM)[norm_pos(lane)] = nh16;
          else lv.v_norm[lv.unit(cb, ch) * lv.capacity + (size_t)(cwin0 + ewq) * W + lane] = nh16;
        }
        const float inv = nf != 0.0f ? __fdiv_rn(1.0f, nf) : 0.0f;
        sm.inv[warp][lane] = inv;
        sm.c3[warp][lane] = BITS == 0 ? __fmul_rn(inv, NEG_INV_3T) : inv * (1.0f / (BINS * bin_width(BITS)));
        nonzero = __ballot_sync(0xffffffffu, nf != 0.0f);
      }
      __syncwarp();
      uint32_t wacc[4] = {0u, 0u, 0u, 0u};   // this channel's codes of the window, one word per t (sh = 0 position)
      for (int jt = 0; jt < jobs.n_jobs; jt++) {
        const int nm = jobs.count(jt);
        const uint32_t a = jobidx & 1u;
        if (i > 0 || jt > 0) bring_matrices(jobs, jt);
        if (!mbar_wait(sm, &sm.mma_done[a], (jobidx >> 1) & 1u)) { dead = true; break; }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const bool last_job = jt + 1 == jobs.n_jobs;
        // the tile's MMAs are complete and this warp keeps what it needs of the buffer in registers (the rare exact
        // recomputation below reads its value row from global memory)
        if (last_job && lane == 0) mbar_arrive(&sm.empty[buf]);
        if (ewq < wins) {
#pragma unroll 1
          for (int mi = 0; mi < nm; mi++) {
            const int mod = jobs.mod(jt, mi);
            const unsigned keep = __ballot_sync(0xffffffffu, mymod == (unsigned)mod);   // bit i: token i
            if (!keep) continue;
            uint32_t r[32];
            const uint32_t taddr = tmem + ((uint32_t)(eq * 32) << 16) + a * 256u + (uint32_t)mi * 128u + (uint32_t)ewq * 32u;
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
                         : "=r"(r[0]),"=r"(r[1]),"=r"(r[2]),"=r"(r[3]),"=r"(r[4]),"=r"(r[5]),"=r"(r[6]),"=r"(r[7]),"=r"(r[8]),"=r"(r[9]),"=r"(r[10]),"=r"(r[11]),"=r"(r[12]),"=r"(r[13]),"=r"(r[14]),"=r"(r[15]),
                           "=r"(r[16]),"=r"(r[17]),"=r"(r[18]),"=r"(r[19]),"=r"(r[20]),"=r"(r[21]),"=r"(r[22]),"=r"(r[23]),"=r"(r[24]),"=r"(r[25]),"=r"(r[26]),"=r"(r[27]),"=r"(r[28]),"=r"(r[29]),"=r"(r[30]),"=r"(r[31])
                         : "r"(taddr) : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
            if constexpr (BITS != 0) {
              unsigned close = 0;   // tokens whose coordinate lies within the band of a threshold
              unsigned char* codes = &sm.lad.code[warp][0][lane];
              const float4* c3p = reinterpret_cast<const float4*>(sm.c3[warp]);
              const float4* ivp = reinterpret_cast<const float4*>(sm.inv[warp]);
#pragma unroll
              for (int i4 = 0; i4 < 8; i4++) {
                const float4 c4 = c3p[i4], v4 = ivp[i4];
                const float cs[4] = {c4.x, c4.y, c4.z, c4.w}, iv[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
                for (int u = 0; u < 4; u++) {
                  const int tok = 4 * i4 + u;
                  const float zr = __uint_as_float(r[tok]);
                  float x, f;
                  asm("fma.rn.sat.f32 %0, %1, %2, %3;\n" : "=f"(x) : "f"(zr), "f"(cs[u]), "f"(16.5f / BINS));
                  asm("fma.rm.f32 %0, %1, %2, %3;\n" : "=f"(f) : "f"(x), "f"((float)BINS - 0.0001f), "f"(FLOOR_MAGIC));
                  const float2 bin = sm.lad.bin[__float_as_uint(f) & (BINS - 1)];
                  const float d = fmaf(zr, iv[u], -bin.x);
                  const int code = __float_as_int(bin.y) + (d > 0.0f ? 1 : 0);
                  if (fabsf(d) <= BAND) close |= 1u << tok;
                  if (keep == 0xffffffffu || ((keep >> tok) & 1u)) codes[tok * 36] = (unsigned char)code;
                }
              }
              close &= keep & nonzero;   // (a zero vector's coordinates are exactly zero)
              while (close) {
                const int tok = __ffs(close) - 1, c = 32 * eq + lane;
                close &= close - 1;
                const __half* xrow = vrows + cb * vs_b + ch * vs_h + (long long)((cwin0 + ewq) * W + tok) * vs_t;
                const float* rrow = R + (size_t)((n_R == 1 ? 0 : ch) * 3 + mod) * D * D + (size_t)c * D;
                const int slot_i = atomicAdd(&sm.fix_count, 1);
                if (slot_i < FIX_MAX) {
                  FixItem& it = sm.fix[slot_i];
                  it.word = reinterpret_cast<uint32_t*>(lv.v_codes + (lv.unit(cb, ch) * lv.capacity + (size_t)(cwin0 + ewq) * W + tok) * (16 * BITS)) +
                            ((BITS * c) >> 5);
                  it.xrow = xrow; it.rrow = rrow; it.inv = sm.inv[warp][tok]; it.bit = (BITS * c) & 31;
                } else {
                  const float z = __fmul_rn(exact_chain(rrow, xrow), sm.inv[warp][tok]);
                  int code = 0;
                  for (int j = 0; j < (1 << BITS) - 1; j++) code += z > c_thresholds[BITS - 2][j];
                  codes[tok * 36] = (unsigned char)code;
                }
              }
            } else {
                        // token i = 8*j + 2*t + e sits in word t at bit 16*e + 2*j (+ 8 for the second channel of the word)
            uint32_t kaccA[4] = {0u, 0u, 0u, 0u}, kaccB[4] = {0u, 0u, 0u, 0u};
            const float4* c3p = reinterpret_cast<const float4*>(sm.c3[warp]);
#pragma unroll
            for (int i4 = 0; i4 < 8; i4++) {
              const float4 c4 = c3p[i4];
              const float cs[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
              for (int u = 0; u < 4; u++) {
                const int t4 = 4 * i4 + u;
                float va, vb, ka, kb;
                asm("fma.rn.sat.f32 %0, %1, %2, %3;\n" : "=f"(va) : "f"(__uint_as_float(r[t4])), "f"(cs[u]), "f"(TWO_THIRDS - BAND_V));
                asm("fma.rn.sat.f32 %0, %1, %2, %3;\n" : "=f"(vb) : "f"(__uint_as_float(r[t4])), "f"(cs[u]), "f"(TWO_THIRDS + BAND_V));
                asm("fma.rm.f32 %0, %1, %2, %3;\n" : "=f"(ka) : "f"(va), "f"(3.0f), "f"(FLOOR_MAGIC));
                asm("fma.rm.f32 %0, %1, %2, %3;\n" : "=f"(kb) : "f"(vb), "f"(3.0f), "f"(FLOOR_MAGIC));
                kaccA[(t4 & 7) >> 1] += __float_as_uint(ka) << (16 * (t4 & 1) + 2 * (t4 >> 3));
                kaccB[(t4 & 7) >> 1] += __float_as_uint(kb) << (16 * (t4 & 1) + 2 * (t4 >> 3));
              }
            }
#pragma unroll
            for (int t = 0; t < 4; t++) {
              // kacc = sum of (magic bits + k) << pos over the word's eight tokens; codes = 3 - k per field
              uint32_t codes = 0x00ff00ffu - (kaccA[t] - MAGIC_SUM);
              uint32_t differ = codes ^ (0x00ff00ffu - (kaccB[t] - MAGIC_SUM));
              uint32_t km = 0x00ff00ffu;
              if (keep != 0xffffffffu) {   // mixed-modality window: only this modality's tokens
                km = 0;
#pragma unroll
                for (int j = 0; j < 4; j++)
#pragma unroll
                  for (int e = 0; e < 2; e++) km |= ((keep >> (8 * j + 2 * t + e)) & 1u) * (3u << (16 * e + 2 * j));
              }
              codes &= km;
              differ &= km;
              while (differ) {   // rare: a coordinate within BAND of a threshold takes the reference arithmetic
                const int pos = (__ffs(differ) - 1) & ~1;               // bit 16 e + 2 j of the field
                const int tok = 8 * ((pos & 15) >> 1) + 2 * t + (pos >> 4);
                const int c = 32 * eq + lane, mu = c >> 4, sh = (c >> 3) & 1, g = c & 7;
                const __half* xrow = vrows + cb * vs_b + ch * vs_h + (long long)((cwin0 + ewq) * W + tok) * vs_t;
                const float* rrow = R + (size_t)((n_R == 1 ? 0 : ch) * 3 + mod) * D * D + (size_t)c * D;
                const int slot_i = atomicAdd(&sm.fix_count, 1);
                if (slot_i < FIX_MAX) {   // later, by a whole warp (the code written now is one of the two neighbouring levels)
                  FixItem& it = sm.fix[slot_i];
                  it.word = reinterpret_cast<uint32_t*>(cv.body(layer, cb, ch, cwin0 + ewq) + B_VCODE) +
                            vword_index((mu >> 2) * 128 + (4 * g + t) * 4 + (mu & 3));
                  it.xrow = xrow; it.rrow = rrow; it.inv = sm.inv[warp][tok]; it.bit = pos + 8 * sh;
                } else {                  // the list is full: here and now
                  const float z = __fmul_rn(exact_chain(rrow, xrow), sm.inv[warp][tok]);
                  const uint32_t code = (uint32_t)((z > -CB_THRESH) + (z > 0.0f) + (z > CB_THRESH));
                  codes = (codes & ~(3u << pos)) | (code << pos);
                }
                differ &= ~(3u << pos);
              }
              wacc[t] |= codes;
            }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.acc_free[a]);
        jobidx++;
      }
      if (dead) break;
      if (BITS != 0 && ewq < wins) {
        if constexpr (BITS != 0) {
          // lane = token: its 32 codes of this warp's channels are 4 BITS bytes of the token's row
          __syncwarp();
          const uint32_t* row = reinterpret_cast<const uint32_t*>(&sm.lad.code[warp][lane][0]);
          uint32_t q4[8];
#pragma unroll
          for (int i = 0; i < 8; i++) {   // four codes of a byte each -> 4 BITS bits
            const uint32_t x = row[i];
            const uint32_t y = (x & 0x00ff00ffu) | ((x & 0xff00ff00u) >> (8 - BITS));
            q4[i] = (y & 0xffffu) | (y >> (16 - 2 * BITS));
          }
          uint32_t* dst = reinterpret_cast<uint32_t*>(lv.v_codes + (lv.unit(cb, ch) * lv.capacity + (size_t)(cwin0 + ewq) * W + lane) * (16 * BITS) +
                                                      4 * BITS * eq);
          if constexpr (BITS == 4)
            *reinterpret_cast<uint4*>(dst) = make_uint4(q4[0] | q4[1] << 16, q4[2] | q4[3] << 16, q4[4] | q4[5] << 16, q4[6] | q4[7] << 16);
          else if constexpr (BITS == 2)
            *reinterpret_cast<uint2*>(dst) = make_uint2(q4[0] | q4[1] << 8 | q4[2] << 16 | q4[3] << 24, q4[4] | q4[5] << 8 | q4[6] << 16 | q4[7] << 24);
          else {
            dst[0] = q4[0] | q4[1] << 12 | q4[2] << 24;
            dst[1] = q4[2] >> 8 | q4[3] << 4 | q4[4] << 16 | q4[5] << 28;
            dst[2] = q4[5] >> 4 | q4[6] << 8 | q4[7] << 20;
          }
        }
      } else if (ewq < wins) {
        // join the two channels of each word (c and c ^ 8 are eight lanes apart) and store: channel
        // c = 16*mu + 8*sh + g writes the words t = 2*sh, 2*sh + 1 of (mu, g)
        const int c = 32 * eq + lane, mu = c >> 4, sh = (c >> 3) & 1, g = c & 7;
        uint32_t* words = reinterpret_cast<uint32_t*>(cv.body(layer, cb, ch, cwin0 + ewq) + B_VCODE);
#pragma unroll
        for (int t = 0; t < 4; t++) {
          const uint32_t own = wacc[t] << (8 * sh);
          const uint32_t full = own | __shfl_xor_sync(0xffffffffu, own, 8);
          if ((t >> 1) == sh) words[vword_index((mu >> 2) * 128 + (4 * g + t) * 4 + (mu & 3))] = full;
        }
      }
      __syncwarp();   // sm.c3[warp] is rewritten for the next tile
      step_coords();
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  // ---- the listed coordinates, one per warp at a time: the two rows go through the warp's corner of the (idle) first
  // tile buffer, every lane evaluates the same chain (input index ascending, one rounding per step), lane 0 patches
  auto patch = [&](uint32_t* word, int bit, float z) {   // the code of coordinate z in place of what is there
    if constexpr (BITS == 0) {
      const uint32_t code = (uint32_t)((z > -CB_THRESH) + (z > 0.0f) + (z > CB_THRESH));
      atomicAnd(word, ~(3u << bit));
      atomicOr(word, code << bit);
    } else {
      uint32_t code = 0;
      for (int j = 0; j < (1 << BITS) - 1; j++) code += z > c_thresholds[BITS - 2][j];
      const unsigned long long field = (unsigned long long)((1u << BITS) - 1u) << bit, val = (unsigned long long)code << bit;
      atomicAnd(word, ~(uint32_t)field);
      atomicOr(word, (uint32_t)val);
      if (field >> 32) {   // a 3-bit code across two words
        atomicAnd(word + 1, ~(uint32_t)(field >> 32));
        atomicOr(word + 1, (uint32_t)(val >> 32));
      }
    }
  };
  {
    const int n_fix = sm.redo ? 0 : min(sm.fix_count, FIX_MAX);
    unsigned char* scr = sm.a[0] + warp * 1024;
    for (int i = warp; i < n_fix && !sm.abort; i += NT_ALL / 32) {
      const FixItem it = sm.fix[i];
      *reinterpret_cast<float4*>(scr + 16 * lane) = __ldg(reinterpret_cast<const float4*>(it.rrow) + lane);
      if (lane < 16) *reinterpret_cast<uint4*>(scr + 512 + 16 * lane) = __ldg(reinterpret_cast<const uint4*>(it.xrow) + lane);
      __syncwarp();
      float a = 0.0f;
#pragma unroll 4
      for (int kc = 0; kc < 16; kc++) {
        const uint4 raw = *reinterpret_cast<const uint4*>(scr + 512 + 16 * kc);
        const __half2* h2 = reinterpret_cast<const __half2*>(&raw);
        const float4 r0 = *reinterpret_cast<const float4*>(scr + 32 * kc), r1 = *reinterpret_cast<const float4*>(scr + 32 * kc + 16);
        const float2 x0 = __half22float2(h2[0]), x1 = __half22float2(h2[1]), x2 = __half22float2(h2[2]), x3 = __half22float2(h2[3]);
        a = __fmaf_rn(r0.x, x0.x, a); a = __fmaf_rn(r0.y, x0.y, a); a = __fmaf_rn(r0.z, x1.x, a); a = __fmaf_rn(r0.w, x1.y, a);
        a = __fmaf_rn(r1.x, x2.x, a); a = __fmaf_rn(r1.y, x2.y, a); a = __fmaf_rn(r1.z, x3.x, a); a = __fmaf_rn(r1.w, x3.y, a);
      }
      const float z = __fmul_rn(a, it.inv);
      if (lane == 0) patch(it.word, it.bit, z);
      __syncwarp();
    }
  }
  // ---- or all of the block's coordinates, one per thread: a warp has 32 channels of a token
  if (sm.redo && !sm.abort) {
    for (int i = 0; i < my_tiles; i++) {
      const int tile = tile_begin + i, b = tile / (tiles_per_unit * cv.n_kv_heads), h = tile / tiles_per_unit % cv.n_kv_heads;
      const int win0 = tile % tiles_per_unit * 4, n_tok = min(TILE, (n_win - win0) * W);
      for (int idx = tid; idx < n_tok * D; idx += NT_ALL) {
        const int tok = win0 * W + idx / D, c = idx % D;
        unsigned m = modality[(size_t)b * n_tokens + tok];
        m = m > 2 ? 0 : m;
        float nf;
        uint32_t* word;
        int bit;
        if constexpr (BITS == 0) {
          unsigned char* body = cv.body(layer, b, h, tok / W);
          nf = __half2float(reinterpret_cast<const __half*>(body + B_VNORM)[norm_pos(tok % W)]);
          int w;
          vcode_pos(tok % W, c, w, bit);
          word = reinterpret_cast<uint32_t*>(body + B_VCODE) + w;
        } else {
          const size_t t = lv.unit(b, h) * lv.capacity + tok;
          nf = __half2float(lv.v_norm[t]);
          word = reinterpret_cast<uint32_t*>(lv.v_codes + t * (16 * BITS)) + ((BITS * c) >> 5);
          bit = (BITS * c) & 31;
        }
        const float a = exact_chain(R + ((size_t)((n_R == 1 ? 0 : h) * 3 + m) * D + c) * D, vrows + b * vs_b + h * vs_h + (long long)tok * vs_t);
        patch(word, bit, __fmul_rn(a, nf != 0.0f ? __fdiv_rn(1.0f, nf) : 0.0f));
      }
    }
  }
  if (BITS != 0 && sm.abort) {   // the ladder's calls have no status word: the tokens of the block's tiles get norms that are no numbers
    for (int i = tid; i < my_tiles * TILE; i += NT_ALL) {
      const int tile = tile_begin + i / TILE, tok = tile % tiles_per_unit * TILE + i % TILE;
      if (tok < n_win * W) lv.v_norm[(size_t)(tile / tiles_per_unit) * lv.capacity + tok] = __ushort_as_half(0x7fff);
    }
  }
  if (tid == 0 && sm.abort && cv.status) atomicCAS(cv.status, 0, (int)OKQ_ERR_TIMEOUT);
  if (warp == 0 && !sm.tmem_busy) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem) : "memory");
}

template <int BITS>
static okq_status launch_values_tc(const CacheView& cv, const LadderView& lv, int layer, const __half* v, const int64_t strides[3],
                                     const unsigned char* modality, int n_tokens, int n_win, const float* R, int n_R,
                                     int n_sm, cudaStream_t s, long long wait_limit, int skip_tile) {
  static_assert(sizeof(TcSmem<BITS>) + 1024 <= 227 * 1024, "shared memory of one block");
  static thread_local unsigned long long attr_mask = 0;
  int attr_dev = 0;
  if (attr_needed(attr_mask, attr_dev)) {
    cudaError_t e = cudaFuncSetAttribute(k_quantize_values_tc<BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(TcSmem<BITS>) + 1024);
    if (e != cudaSuccess) { set_last_cuda_error((int)e); return OKQ_ERR_CUDA; }
    attr_done(attr_mask, attr_dev);
  }
  const long long n_tiles = (long long)((n_win + 3) / 4) * cv.n_kv_heads * cv.batch;
  if (n_tiles == 0) return OKQ_OK;
  // the values as a 4-d tensor [batch][head][token][channel] for the copy engine; a box is 64 channels x 128 tokens
  EncodeTiledFn enc = encode_tiled();
  if (!enc) { set_last_cuda_error((int)cudaErrorNotSupported); return OKQ_ERR_CUDA; }
  CUtensorMap vmap;
  const cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)n_tokens, (cuuint64_t)cv.n_kv_heads, (cuuint64_t)cv.batch};
  // a dimension of extent 1 is never stepped: give it any legal stride
  const cuuint64_t gstr[3] = {(cuuint64_t)(n_tokens > 1 ? strides[2] : D) * 2, (cuuint64_t)(cv.n_kv_heads > 1 ? strides[1] : D) * 2,
                              (cuuint64_t)(cv.batch > 1 ? strides[0] : D) * 2};
  const cuuint32_t box[4] = {64, (cuuint32_t)TILE, 1, 1}, estr[4] = {1, 1, 1, 1};
  for (int i = 0; i < 3; i++)
    if (gstr[i] == 0 || gstr[i] % 16 || gstr[i] >= (1ull << 40)) return OKQ_ERR_UNSUPPORTED;
  const CUresult cr = enc(&vmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<__half*>(v), dims, gstr, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (cr != CUDA_SUCCESS) { set_last_cuda_error((int)cudaErrorInvalidValue); return OKQ_ERR_CUDA; }
  const int grid = (int)(n_tiles < n_sm ? n_tiles : n_sm);
  const cudaError_t le = launch_dependent(k_quantize_values_tc<BITS>, dim3(grid), NT_ALL, sizeof(TcSmem<BITS>) + 1024, s, 1, vmap, cv, lv, layer,
                                          modality, n_tokens, n_win, R, n_R, v, (long long)strides[0], (long long)strides[1], (long long)strides[2],
                                          wait_limit > 0 ? wait_limit : WAIT_LIMIT_CLOCKS, skip_tile);
  if (le != cudaSuccess) { set_last_cuda_error((int)le); return OKQ_ERR_CUDA; }
  return OKQ_OK;
}

okq_status launch_quantize_values_tc(const CacheView& cv, int layer, const __half* v, const int64_t strides[3],
                                     const unsigned char* modality, int n_tokens, int n_win, const float* R, int n_R,
                                     int n_sm, cudaStream_t s, long long wait_limit, int skip_tile) {
  return launch_values_tc<0>(cv, LadderView{}, layer, v, strides, modality, n_tokens, n_win, R, n_R, n_sm, s, wait_limit, skip_tile);
}

okq_status launch_ladder_values_tc(const LadderView& lv, const __half* v, const int64_t strides[3], const unsigned char* modality,
                                   int n_tokens, const float* R, int n_R, int n_sm, cudaStream_t s, long long wait_limit, int skip_tile) {
  CacheView cv{};   // shape and modality bytes; no status word: the ladder calls have none
  cv.n_layers = 1; cv.batch = lv.batch; cv.n_kv_heads = lv.n_kv_heads; cv.n_q_heads = lv.n_q_heads; cv.capacity = lv.capacity;
  cv.modality = lv.modality;
  const int n_win = n_tokens / W;
  return lv.bits == 2 ? launch_values_tc<2>(cv, lv, 0, v, strides, modality, n_tokens, n_win, R, n_R, n_sm, s, wait_limit, skip_tile)
       : lv.bits == 3 ? launch_values_tc<3>(cv, lv, 0, v, strides, modality, n_tokens, n_win, R, n_R, n_sm, s, wait_limit, skip_tile)
                      : launch_values_tc<4>(cv, lv, 0, v, strides, modality, n_tokens, n_win, R, n_R, n_sm, s, wait_limit, skip_tile);
}

}  // namespace okq
