// Attention weights of a calibration sequence on the 5th-generation tensor cores: w_j = sum over heads g and queries i of
// alpha[g, i, j]^2, alpha = softmax(q k^T * scale), in two passes over the score tiles.
//
//   pass 0   every query's maximum m_i and normaliser l_i = sum_j 2^(s_ij - m_i)   (log2 domain, s = (q . k) * scale2)
//   pass 1   column sums of alpha^2 = 2^(2 s_ij - 2 m_i) / l_i^2
//
// A tile is 128 queries x 128 keys of one head, the product of two TMA-fetched operands in tensor memory: lane = query,
// column = key, in both passes.  Pass 0 keeps a tile of queries and walks the keys, so that a thread has one query's
// maximum and sum; pass 1 keeps a tile of keys and walks the queries of all heads, so that a thread adds up 32 columns in
// registers and lanes only meet when the key tile changes.  Neither pass reads anything per score from shared memory.
//
// Roles: a loader warp (ring of NS walked tiles, two kept ones), an MMA warp (four accumulators of 128 columns), sixteen
// worker warps, four to each quarter of the lanes, 32 columns each.  The (tile, head) steps of a pass are numbered and cut
// into equal ranges, one per block; what a range holds of a query or key tile is a piece, pieces are put together in order.
//
// What bounds it: one exponential per score and pass (16 per cycle and SM; 8192 tokens x 7 heads, causal: 51 us a pass), the units
// for which are busy 73 % of the time; the tensor pipe is a third busy.  8192 tokens x 7 heads 578 -> 195 us against the mma.sync
// kernels of okq_calib.cu, 512 x 7 34 -> 20 (most of it the four launches).
#include "okq_calib_scores.cuh"
#include "okq_device.cuh"
#include "okq_tc.cuh"

namespace okq {

namespace {

constexpr int TS = SCORE_TILE;            // queries and keys per tile
constexpr int NT = 512;                   // worker threads
constexpr int NT_ALL = NT + 64;           // + the MMA warp (16) and the loader warp (17)
constexpr int OP_BYTES = TS * D * 2;      // one operand tile
constexpr int NS = 4;                     // ring of walked tiles

struct ScoreSmem {
  __align__(1024) unsigned char ring[NS][OP_BYTES];
  __align__(1024) unsigned char kept[2][OP_BYTES];
  __align__(16) float2 row[2][4][TS];     // pass 0: (m, l) of a query over the columns of a warp's quarter, two items
  __align__(16) float col[2][4][TS];      // pass 1: column sums over a quarter of the lanes, two items
  __align__(8) unsigned long long full[NS], empty[NS];           // ring: landed / read by the products
  __align__(8) unsigned long long kept_full[2], kept_empty[2];   // kept tiles
  __align__(8) unsigned long long acc_full[4], acc_free[4];      // accumulators: complete / read by the 16 worker warps
  uint32_t tmem_slot;
  long long limit;                        // SM clocks a wait may take
  volatile int abort;                     // set by a role whose bounded wait ran out
  volatile int tmem_busy;
};

// The steps of a pass in order.  Pass 0: items (query tile t, head), an item walks the key tiles it sees.  Pass 1: items = key
// tiles t, an item walks the query tiles that see it, all heads of one before the next.
template <int PASS> struct Steps {
  int n_t, G, causal;
  __host__ __device__ long long start(int t, int head) const {   // number of the item's first step
    if (PASS == 0) return causal ? (long long)G * t * (t + 1) / 2 + (long long)head * (t + 1) : ((long long)t * G + head) * n_t;
    return causal ? (long long)G * ((long long)t * n_t - (long long)t * (t - 1) / 2) : (long long)t * G * n_t;
  }
  __host__ __device__ int size(int t) const { return PASS == 0 ? (causal ? t + 1 : n_t) : G * (causal ? n_t - t : n_t); }
  __host__ __device__ long long total() const { return start(n_t, 0); }
};

template <int PASS> struct Cursor {
  Steps<PASS> st;
  int t, head, pos, size;     // item (pass 1: head of the walked tile), step inside it
  int q;                      // pass 1: walked query tile
  int piece;                  // number of the piece of this item that this range holds
  __device__ Cursor(const Steps<PASS>& s, long long c0, long long per) : st(s) {
    t = 0; head = 0;
    while (t + 1 < st.n_t && st.start(t + 1, 0) <= c0) t++;
    if (PASS == 0) { head = (int)((c0 - st.start(t, 0)) / st.size(t)); }
    const long long s0 = st.start(t, PASS == 0 ? head : 0);
    pos = (int)(c0 - s0);
    size = st.size(t);
    piece = (int)(c0 / per - s0 / per);
    if (PASS == 1) { q = (st.causal ? t : 0) + pos / st.G; head = pos % st.G; }
  }
  __device__ bool first() const { return pos == 0; }
  __device__ bool last() const { return pos + 1 == size; }
  __device__ void next() {
    if (PASS == 1 && ++head == st.G) { head = 0; q++; }
    if (++pos < size) return;
    pos = 0; piece = 0;
    if (PASS == 0) { if (++head == st.G) { head = 0; t++; } }
    else { t++; q = st.causal ? t : 0; }
    size = st.size(t);
  }
  __device__ int qtile() const { return PASS == 0 ? t : q; }
  __device__ int ktile() const { return PASS == 0 ? pos : t; }
};

__device__ __forceinline__ void tma_tile(const CUtensorMap* map, void* dst, int row, int slab, uint32_t bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"((uint32_t)OP_BYTES) : "memory");
#pragma unroll
  for (int half = 0; half < 2; half++)   // 64 channels x 128 rows; rows past the end are filled with zeros
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n"
                 ::"r"(smem_u32(dst) + half * (OP_BYTES / 2)), "l"(reinterpret_cast<uint64_t>(map)), "r"(64 * half), "r"(row), "r"(slab),
                   "r"(bar) : "memory");
}

// stat: pass 0 writes the pieces' (m, l), [piece][head][query]; pass 1 reads (-2 m, 1 / l^2), [head][query].
// partial: pass 1 writes [piece][key].
template <int PASS>
__global__ void __launch_bounds__(NT_ALL, 1) k_calib_scores(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap,
                                                           int G, int n, float scale2, int causal, long long per, float2* __restrict__ stat,
                                                           float* __restrict__ partial, long long wait_limit, int skip_step) {
  extern __shared__ unsigned char raw_smem[];
  ScoreSmem& sm = *reinterpret_cast<ScoreSmem*>((reinterpret_cast<uintptr_t>(raw_smem) + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    auto init = [](unsigned long long* b, int count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(b)), "r"(count)); };
    for (int i = 0; i < NS; i++) { init(&sm.full[i], 1); init(&sm.empty[i], 1); }
    for (int i = 0; i < 2; i++) { init(&sm.kept_full[i], 1); init(&sm.kept_empty[i], 1); }
    for (int i = 0; i < 4; i++) { init(&sm.acc_full[i], 1); init(&sm.acc_free[i], 16); }
    sm.abort = 0;
    sm.tmem_busy = 0;
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

  const Steps<PASS> steps{(n + TS - 1) / TS, G, causal};
  const long long total = steps.total(), c0 = min(total, (long long)blockIdx.x * per);
  const int n_my = (int)(min(total, c0 + per) - c0);
  Cursor<PASS> cur(steps, min(c0, total - 1), per);

  if (warp == 17) {
    // ------------------------------------------------------------------ loader warp
    int armed = 0, items = 0;
    for (int i = 0; i < n_my; i++, cur.next()) {
      const int s = i % NS;
      if (i == skip_step) break;   // testing aid: the tile never arrives, so that every role's wait runs out
      if (i == 0 || cur.first()) {
        if (items >= 2 && !mbar_wait(sm, &sm.kept_empty[items & 1], (uint32_t)((items >> 1) - 1) & 1u)) break;
        if (lane == 0) {
          if (PASS == 0) tma_tile(&qmap, sm.kept[items & 1], cur.t * TS, cur.head, smem_u32(&sm.kept_full[items & 1]));
          else tma_tile(&kmap, sm.kept[items & 1], cur.t * TS, 0, smem_u32(&sm.kept_full[items & 1]));
        }
        items++;
      }
      if (i >= NS && !mbar_wait(sm, &sm.empty[s], (uint32_t)(i / NS - 1) & 1u)) break;
      if (lane == 0) {
        if (PASS == 0) tma_tile(&kmap, sm.ring[s], cur.ktile() * TS, 0, smem_u32(&sm.full[s]));
        else tma_tile(&qmap, sm.ring[s], cur.qtile() * TS, cur.head, smem_u32(&sm.full[s]));
      }
      armed = i + 1;
    }
    if (sm.abort || armed < n_my) {   // no copy of this warp may still be landing when the block ends
      for (int i = max(0, armed - NS); i < armed; i++) mbar_drain(&sm.full[i % NS], (uint32_t)(i / NS) & 1u);
      for (int i = max(0, items - 2); i < items; i++) mbar_drain(&sm.kept_full[i & 1], (uint32_t)(i >> 1) & 1u);
    }
  } else if (warp == 16) {
    // ------------------------------------------------------------------ MMA warp
    int done = 0, items = 0;
    for (int i = 0; i < n_my; i++, cur.next()) {
      const int s = i % NS, a = i & 3;
      if (i == 0 || cur.first()) {
        if (!mbar_wait(sm, &sm.kept_full[items & 1], (uint32_t)(items >> 1) & 1u)) break;
        items++;
      }
      if (!mbar_wait(sm, &sm.full[s], (uint32_t)(i / NS) & 1u)) break;
      if (i >= 4 && !mbar_wait(sm, &sm.acc_free[a], (uint32_t)((i >> 2) - 1) & 1u)) break;
      const int kb = (items - 1) & 1;
      const bool give_back = cur.last() || i + 1 == n_my;
      if (elect_one()) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(TS >> 3) << 17) | ((uint32_t)(TS >> 4) << 24);   // D fp32, A/B fp16 K-major
        const uint64_t walked = make_desc_sw128(smem_u32(sm.ring[s])), kept = make_desc_sw128(smem_u32(sm.kept[kb]));
        const uint64_t da0 = PASS == 0 ? kept : walked, db0 = PASS == 0 ? walked : kept;   // A: queries, B: keys
#pragma unroll
        for (int k = 0; k < 8; k++) {   // 16 channels: 32 bytes further inside a row, the second 64 in the tile's second half
          const uint64_t off = (uint64_t)(((k & 3) * 32 + (k >> 2) * (OP_BYTES / 2)) >> 4);
          asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                       "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5}, p;\n\t}\n"
                       ::"r"(tmem + (uint32_t)a * TS), "l"(da0 + off), "l"(db0 + off), "r"(idesc), "r"(k ? 1u : 0u), "r"(0u) : "memory");
        }
        auto commit = [](unsigned long long* b) {
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(b)) : "memory");
        };
        commit(&sm.empty[s]);
        if (give_back) commit(&sm.kept_empty[kb]);
        commit(&sm.acc_full[a]);
      }
      __syncwarp();
      done = i + 1;
    }
    // nothing may be in flight when tensor memory is released; if the last products do not answer, it stays allocated
    if (done >= 1 && !mbar_drain(&sm.acc_full[(done - 1) & 3], (uint32_t)((done - 1) >> 2) & 1u)) sm.tmem_busy = 1;
  } else {
    // ------------------------------------------------------------------ worker warps (after a timeout they run on, waits failing at once)
    const int eq = warp & 3, wq = warp >> 2;   // quarter of the lanes, quarter of the columns
    const uint32_t taddr = tmem + ((uint32_t)(eq * 32) << 16) + 32u * (uint32_t)wq;
    const F2 two2 = f2(2.0f * scale2, 2.0f * scale2), one2 = f2(scale2, scale2);
    float m = -INFINITY, l = 0.f;              // pass 0: this thread's query over its columns
    F2 acc[16];                                // pass 1: sums of this thread's columns over the lane's queries
#pragma unroll
    for (int i = 0; i < 16; i++) acc[i] = f2(0.f, 0.f);
    float tot = 0.f;                           // ... of earlier steps, one column per lane
    int items = 0;
    const int ragged = n % TS ? n / TS : -1;   // the tile that is not full
    auto row_stat = [&]() -> float2 {          // pass 1: of this lane's query in the current step
      const int i = cur.qtile() * TS + 32 * eq + lane;
      return i < n ? __ldcg(&stat[(size_t)cur.head * n + i]) : make_float2(0.f, 0.f);
    };
    float2 rs_next = make_float2(0.f, 0.f);
    if (PASS == 1 && n_my > 0) rs_next = row_stat();
    for (int i = 0; i < n_my; i++) {
      const int a = i & 3, t = cur.t, head = cur.head, piece = cur.piece, qt = cur.qtile(), kt = cur.ktile();
      const bool last = cur.last() || i + 1 == n_my;
      const float2 rs = rs_next;
      cur.next();
      if (PASS == 1 && i + 1 < n_my) rs_next = row_stat();
      mbar_wait(sm, &sm.acc_full[a], (uint32_t)(i >> 2) & 1u);
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      uint32_t r[32];
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
                   : "=r"(r[0]),"=r"(r[1]),"=r"(r[2]),"=r"(r[3]),"=r"(r[4]),"=r"(r[5]),"=r"(r[6]),"=r"(r[7]),"=r"(r[8]),"=r"(r[9]),"=r"(r[10]),"=r"(r[11]),"=r"(r[12]),"=r"(r[13]),"=r"(r[14]),"=r"(r[15]),
                     "=r"(r[16]),"=r"(r[17]),"=r"(r[18]),"=r"(r[19]),"=r"(r[20]),"=r"(r[21]),"=r"(r[22]),"=r"(r[23]),"=r"(r[24]),"=r"(r[25]),"=r"(r[26]),"=r"(r[27]),"=r"(r[28]),"=r"(r[29]),"=r"(r[30]),"=r"(r[31])
                   : "r"(taddr + (uint32_t)a * TS) : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.acc_free[a]);
      // scores that do not count: keys after the query, rows of no token (zero queries, whose products with infinite keys are NaN)
      const bool edge = (causal && qt == kt) || (PASS == 0 ? kt : qt) == ragged;
      if (edge) {
        const int row = qt * TS + 32 * eq + lane, j0 = kt * TS + 32 * wq;
        const int seen = (row < n ? (causal ? row + 1 : n) : 0) - j0;
#pragma unroll
        for (int c = 0; c < 32; c++)
          if (c >= seen) r[c] = 0xff800000u;   // -inf
      }
      if (PASS == 0) {
        float mx[4];
#pragma unroll
        for (int q = 0; q < 4; q++) mx[q] = __uint_as_float(r[q]);
#pragma unroll
        for (int c = 4; c < 32; c++) mx[c & 3] = fmaxf(mx[c & 3], __uint_as_float(r[c]));
        const float mn = fmaxf(m, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * scale2);
        if (!edge || mn != -INFINITY) {
          const float at = mn == -INFINITY ? 0.f : mn;   // (whole tiles of infinite keys: every term is 0)
          const F2 neg = f2(-at, -at);
          F2 s[2] = {f2(0.f, 0.f), f2(0.f, 0.f)};   // (on their own: a long sum takes one rounding per tile)
#pragma unroll
          for (int c = 0; c < 16; c++) {
            const float2 x = un2(fma2(f2(__uint_as_float(r[2 * c]), __uint_as_float(r[2 * c + 1])), one2, neg));
            s[c & 1] = add2(s[c & 1], f2(ex2(x.x), ex2(x.y)));
          }
          const float2 u = un2(add2(s[0], s[1]));
          l = fmaf(l, ex2(m - at), u.x + u.y);     // (a factor 0 for the first finite maximum)
          m = mn;
        }
        if (last) {
          sm.row[items & 1][wq][32 * eq + lane] = make_float2(m, l);
          asm volatile("bar.sync 1, %0;\n" ::"n"(NT) : "memory");
          const int row = t * TS + 32 * eq + lane;
          if (wq == 0 && row < n) {
            float2 p[4];
            float M = -INFINITY, L = 0.f;
#pragma unroll
            for (int q = 0; q < 4; q++) { p[q] = sm.row[items & 1][q][32 * eq + lane]; M = fmaxf(M, p[q].x); }
#pragma unroll
            for (int q = 0; q < 4; q++) L += p[q].x == -INFINITY ? 0.f : p[q].y * ex2(p[q].x - M);
            stat[((size_t)piece * G + head) * n + row] = sm.abort ? make_float2(NAN, NAN) : make_float2(M, L);
          }
          items++;
          m = -INFINITY;
          l = 0.f;
        }
      } else {
        const F2 m2 = f2(rs.x, rs.x), c2 = f2(rs.y, rs.y);
#pragma unroll
        for (int c = 0; c < 16; c++) {
          const float2 x = un2(fma2(f2(__uint_as_float(r[2 * c]), __uint_as_float(r[2 * c + 1])), two2, m2));
          acc[c] = fma2(f2(ex2(x.x), ex2(x.y)), c2, acc[c]);
        }
        // over the lanes, each ending with one column: bits 4..0 of the column by lane bits 4..0.  Every 16 steps: the exchange is
        // hidden behind the exponentials, and sums of 98 terms in one register cost a factor two in the error.
        if (last || (i & 15) == 15) {
          float v[32];
#pragma unroll
          for (int c = 0; c < 16; c++) { const float2 x = un2(acc[c]); v[2 * c] = x.x; v[2 * c + 1] = x.y; acc[c] = f2(0.f, 0.f); }
#pragma unroll
          for (int w = 16; w >= 1; w >>= 1) {
            const bool upper = (lane & w) != 0;
#pragma unroll
            for (int c = 0; c < 16; c++)
              if (c < w) {
                const float give = upper ? v[c] : v[c + w], keep = upper ? v[c + w] : v[c];
                v[c] = keep + __shfl_xor_sync(0xffffffffu, give, w);
              }
          }
          tot += v[0];
        }
        if (last) {
          sm.col[items & 1][eq][32 * wq + lane] = tot;
          tot = 0.f;
          asm volatile("bar.sync 1, %0;\n" ::"n"(NT) : "memory");
          const int c = 32 * wq + lane, j = t * TS + c;
          if (eq == 0 && j < n) {
            const float (*p)[TS] = sm.col[items & 1];
            partial[(size_t)piece * n + j] = sm.abort ? NAN : (p[0][c] + p[1][c]) + (p[2][c] + p[3][c]);
          }
          items++;
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0 && !sm.tmem_busy) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem) : "memory");
}

// the pieces of a query's (m, l) put together, as pass 1 uses them: (-2 m, 1 / l^2), in the first piece's place
__global__ void __launch_bounds__(256) k_calib_rows(int G, int n, int causal, long long per, float2* __restrict__ stat) {
  depend_wait();
  const int id = blockIdx.x * 256 + threadIdx.x;
  if (id >= G * n) return;
  const int head = id / n, i = id % n, t = i / TS;
  const Steps<0> steps{(n + TS - 1) / TS, G, causal};
  const long long s0 = steps.start(t, head);
  const int pieces = (int)((s0 + steps.size(t) - 1) / per - s0 / per) + 1;
  float2* p = stat + (size_t)head * n + i;
  float M = -INFINITY, L = 0.f;
  for (int q = 0; q < pieces; q++) {
    const float2 x = p[(size_t)q * G * n];
    const float mn = fmaxf(M, x.x);
    L = (M == -INFINITY ? 0.f : L * ex2(M - mn)) + (x.x == -INFINITY ? 0.f : x.y * ex2(x.x - mn));
    M = mn;
  }
  *p = make_float2(-2.0f * M, 1.0f / (L * L));
}

// w_j = the pieces' sums in order
__global__ void __launch_bounds__(256) k_calib_pieces(const float* __restrict__ partial, int G, int n, int causal, long long per, float* __restrict__ w) {
  depend_wait();
  const int j = blockIdx.x * 256 + threadIdx.x;
  if (j >= n) return;
  const Steps<1> steps{(n + TS - 1) / TS, G, causal};
  const long long s0 = steps.start(j / TS, 0);
  const int pieces = (int)((s0 + steps.size(j / TS) - 1) / per - s0 / per) + 1;
  float s = 0.f;
  for (int q = 0; q < pieces; q++) s += partial[(size_t)q * n + j];
  w[j] = s;
}

bool make_map(CUtensorMap* map, const __half* x, int n, int slabs) {
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)n, (cuuint64_t)slabs};
  const cuuint64_t str[2] = {(cuuint64_t)D * 2, (cuuint64_t)n * D * 2};
  const cuuint32_t box[3] = {64, (cuuint32_t)TS, 1}, estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half*>(x), dims, str, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int PASS>
cudaError_t launch_pass(const CUtensorMap& qmap, const CUtensorMap& kmap, int G, int n, float scale2, int causal, long long per, int grid,
                        float2* stat, float* partial, long long wait_limit, int skip_step, cudaStream_t s) {
  static thread_local unsigned long long attr_mask = 0;
  int dev = 0;
  constexpr int SMEM = (int)sizeof(ScoreSmem) + 1024;
  static_assert(SMEM <= 227 * 1024, "shared memory of one block");
  if (attr_needed(attr_mask, dev)) {
    const cudaError_t e = cudaFuncSetAttribute(k_calib_scores<PASS>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    if (e != cudaSuccess) return e;
    attr_done(attr_mask, dev);
  }
  return launch_dependent(k_calib_scores<PASS>, dim3(grid), NT_ALL, SMEM, s, 1, qmap, kmap, G, n, scale2, causal, per, stat, partial,
                          wait_limit > 0 ? wait_limit : WAIT_LIMIT_CLOCKS, skip_step);
}

}  // namespace

cudaError_t launch_calib_scores(const __half* q, const __half* k, int G, int n, float scale2, int causal, int n_sm, void* ws, float* w_out,
                                long long wait_limit, int skip_step, cudaStream_t s) {
  const Steps<0> s0{(n + TS - 1) / TS, G, causal};
  const Steps<1> s1{s0.n_t, G, causal};
  const long long total = s0.total(), even = (total + n_sm - 1) / n_sm, per = even > SCORE_MIN_STEPS ? even : SCORE_MIN_STEPS;
  const int grid = (int)((total + per - 1) / per);
  const long long row_pieces = (s0.size(s0.n_t - 1) + per - 2) / per + 1;
  float2* stat = static_cast<float2*>(ws);
  float* partial = reinterpret_cast<float*>(stat + (size_t)row_pieces * G * n);
  CUtensorMap qmap, kmap;
  if (!make_map(&qmap, q, n, G) || !make_map(&kmap, k, n, 1)) return cudaErrorInvalidValue;
  cudaError_t e = launch_pass<0>(qmap, kmap, G, n, scale2, causal, per, grid, stat, partial, wait_limit, skip_step, s);
  if (e == cudaSuccess) e = launch_dependent(k_calib_rows, dim3((unsigned)(((long long)G * n + 255) / 256)), 256, 0, s, 1, G, n, causal, per, stat);
  if (e == cudaSuccess) e = launch_pass<1>(qmap, kmap, G, n, scale2, causal, per, grid, stat, partial, wait_limit, skip_step, s);
  if (e == cudaSuccess) e = launch_dependent(k_calib_pieces, dim3((n + 255) / 256), 256, 0, s, 1, partial, G, n, causal, per, w_out);
  return e;
}

}  // namespace okq
