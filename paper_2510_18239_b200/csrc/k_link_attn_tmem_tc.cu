// Links attend over the history on the 5th-generation tensor cores, probabilities kept in tensor memory (bf16 storage,
// rows LayerNorm-ed already; d = 128 and d = 256):
//
//   O[T]_h = phi( Q[T]_h K[S]_h^T * scale ) V[S]_h,  K[S] = X W_K,  V[S] = X W_V,  X = LN(S)                (Eq. 3 / Eq. 7)
//
// Same algebra as k_link_attn_tc.cu (which serves rows that still need their LayerNorm): W_K is folded into the link
// queries (Q2, k_link_prep.cu; scores arrive in the log2 domain) and W_V is applied after the attention, so both
// contractions run against the stored history rows X, streamed once by TMA and used as keys and as values:
//   scores [128 x TILE]  = Q2_block [128 x d] . X_tile^T          (one block of 128 stacked (head, link) rows per work item)
//   acc    [128 x d]    += P [128 x TILE] . X_tile
// Online softmax in the log2 domain with lazy rescale, or SiLU(s) / N(U) with `silu` (Algorithms 1-2).
//
// What bounds it: a tile is a chain - scores, TMEM load, row maximum, exponentials, probabilities, value contraction -
// whose latency is several times its tensor time, so the design is about keeping several tiles in the chain at once and
// each link of it short.
//  * P overwrites its own scores in TMEM as bf16 (half the columns) and is the A operand of the value contraction from
//    there: no shared memory for P, no proxy fence, and the contraction's shared-memory reads halve.
//  * Scores and values are issued by two warps.  The scores of tile g + SBUFS are ordered behind the value contraction of
//    tile g in the pipe (its completion is not waited for), across the ends of items too.
//  * 64-token tiles waste the tensor pipe: with N = 64 the A operand's shared-memory reads take twice the time of the
//    products.  d = 128 takes 128 tokens, five stages, three score buffers; at d = 256 a stage of 128 tokens is 64 KB and
//    only two fit beside the 64 KB of queries, which exposes the copy of every tile: 96 tokens, three stages, two buffers.
//  * d = 128, three score buffers: two groups of softmax warps take alternate tiles, one thread per row.  d = 256, two
//    buffers: the chain of a buffer is what repeats, so all eight warps take every tile, two threads per row.
// Measured: d = 256, 64 links (1024 users of 1024..4096 tokens) 1.51 -> 1.04 ms a launch (0.61 of the tensor peak at the
// clock it runs at; 64-token tiles with P in shared memory and one issuing thread before); d = 128, 64 links, 32 users x 32768
// tokens 172 -> 128 us and, with the items fitted to the CTAs (k_misc.cu), 110; 256 users x 512 tokens, 32 links 20 -> 16 us.
// A tile of d = 128 takes 1490 cycles, 1024 of them the exponentials' (16 a cycle and SM), and an item 3100 to 8800 besides.
// Dropped: 16 softmax warps at d = 128 (two threads per row and two groups: 200 us, the polling takes the issue slots),
// prefetching token tiles into L2 (no change), a quarter to a half of the exponentials as polynomials on the FMA pipes (no
// change to 15 % slower: the chain is what repeats, not the unit).
#include "lime_common.cuh"
#include "tc_common.cuh"

namespace lime {

// Geometry: D features per row, TILE tokens per tile, XSTAGES token stages, SBUFS score buffers in TMEM, QBUFS buffers of
// folded queries.  STRIDED: the CTA walks items blockIdx / RB, + gridDim / RB, ..; otherwise the dealt lists.
template <int D_, int TILE_, int XSTAGES_, int SBUFS_, int QBUFS_, int GROUPS_, int PARTS_, bool STRIDED_>
struct LtCfg {
  static constexpr int D = D_, TILE = TILE_, XSTAGES = XSTAGES_, SBUFS = SBUFS_, QBUFS = QBUFS_;
  static constexpr bool STRIDED = STRIDED_;
  static constexpr int GROUPS = GROUPS_;                        // softmax groups: tile g belongs to group g % GROUPS
  static constexpr int PARTS = PARTS_, COLS = TILE / PARTS;     // threads per row in a group, token columns of each
  static constexpr int OUT = D / (GROUPS * PARTS);              // accumulator columns a thread reads out
  static constexpr int GROUP_WARPS = 4 * PARTS, SOFTMAX_WARPS = GROUPS * GROUP_WARPS, THREADS = 128 + 32 * SOFTMAX_WARPS;
  // registers a thread at launch and after the split (a softmax thread holds its scores of the tile)
  static constexpr int REGS_LAUNCH = SOFTMAX_WARPS == 8 ? 168 : 96;
  static constexpr int REGS_CONTROL = SOFTMAX_WARPS == 8 ? 88 : 64, REGS_SOFTMAX = SOFTMAX_WARPS == 8 ? 208 : 104;
  static_assert(128 * REGS_CONTROL + 32 * SOFTMAX_WARPS * REGS_SOFTMAX <= THREADS * REGS_LAUNCH, "register split");
  static constexpr uint32_t XSUB = TILE * 128;                  // [TILE tokens x 64 features]
  static constexpr uint32_t X_STAGE = (D / 64) * XSUB;
  static constexpr uint32_t QSUB = 128 * 128;                   // [128 rows x 64 features]
  static constexpr uint32_t Q_BUF = (D / 64) * QSUB;
  static constexpr uint32_t OFF_X = 0;
  static constexpr uint32_t OFF_Q2 = XSTAGES * X_STAGE;
  // exchange area (floats): published reference maxima [2 tile parities][128] (two groups), row sums
  // [2 item parities][GROUPS * PARTS][128], row maxima of a tile's parts [GROUPS][2 tile parities][PARTS][128] (PARTS > 1)
  static constexpr uint32_t OFF_EXCH = OFF_Q2 + QBUFS * Q_BUF;
  static constexpr uint32_t EXCH_FLOATS = ((GROUPS > 1 ? 2 : 0) + 2 * GROUPS * PARTS + (PARTS > 1 ? 2 * GROUPS * PARTS : 0)) * 128;
  static constexpr uint32_t OFF_BAR = OFF_EXCH + EXCH_FLOATS * 4;
  static constexpr uint32_t SMEM = OFF_BAR + 384;
  static constexpr uint32_t COL_O = 512 - D;                    // scores: SBUFS x 128 columns from 0; accumulator: D columns
  static constexpr uint32_t TMEM_COLS = 512;
  static_assert(SBUFS * 128 <= 512 - D && COLS % 16 == 0 && TILE <= 128 && GROUPS <= 2 && OUT % 32 == 0 && XSTAGES <= 5 && SBUFS <= 3 && QBUFS <= 2, "layout");
  static_assert(X_STAGE % 1024 == 0 && SMEM <= 232448, "shared memory budget of one CTA");
};
constexpr float LT_RESCALE_THRESHOLD = 8.0f;                  // in log2 units

struct LinkAttnTmemParams {
  const int32_t* off;
  const int32_t* chunk_start;     // [B+1] prefix of per-user chunk counts
  const int32_t* chunk_user;      // [chunk items] user of each (user, chunk) item
  const int32_t* group_start;     // [groups + 1] the items of a group of CTAs (one CTA per row block) are
  const int32_t* group_items;     //              group_items[group_start[j] .. group_start[j + 1]); unused when strided
  const int32_t* chunk;           // tokens per chunk
  int B, shared, ell, H;
  int silu;
  int HL, RB;                     // stacked (head, link) rows in all, and 128-row blocks of them (one per work item)
  float *part_m, *part_s, *part_acc;   // [items x HL], [items x HL], [items x HL x d]
  __nv_bfloat16* Ohat;                 // [B*ell x H*d]: final rows of single-chunk users
  int* err;
};

__device__ __forceinline__ uint32_t lt_pack(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float lt_silu(float x) {
  const float hx = 0.5f * x;
  float th;
  asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(hx));
  return fmaf(hx, th, hx);
}
__device__ __forceinline__ float lt_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// p = 2^(s - m_ref) (or SiLU(s)) for the thread's token columns, stored as bf16 pairs over its own scores: columns 2j and
// 2j + 1 in TMEM column j.  Columns past the end of a ragged last tile were set to -inf (0 for SiLU) by the caller and give
// 0.  Returns the sum.
template <bool SILU, int COLS>
__device__ __forceinline__ float lt_probabilities(const float (&v)[COLS], float m_ref, uint32_t taddr) {
  constexpr int STEP = COLS % 32 == 0 ? 32 : 16;
  float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll
  for (int c = 0; c < COLS; c += STEP) {
    float packed[STEP / 2];
#pragma unroll
    for (int j = 0; j < STEP / 2; ++j) {
      float2 e = make_float2(v[c + 2 * j], v[c + 2 * j + 1]);
      if (SILU) {
        e = make_float2(lt_silu(e.x), lt_silu(e.y));
      } else {
        e = __fadd2_rn(e, make_float2(-m_ref, -m_ref));
        e = make_float2(lt_ex2(e.x), lt_ex2(e.y));
        if (j & 1) s1 = __fadd2_rn(s1, e); else s0 = __fadd2_rn(s0, e);
      }
      packed[j] = __uint_as_float(lt_pack(e.x, e.y));
    }
    if constexpr (STEP == 32) tc::tmem_st_32x16(taddr + (uint32_t)(c >> 1), packed);
    else tc::tmem_st_32x8(taddr + (uint32_t)(c >> 1), packed);
  }
  s0 = __fadd2_rn(s0, s1);
  return s0.x + s0.y;
}

// Walk over the (user, chunk) items of a CTA's group.  The index arrays stay in global memory; the items and users of the
// next two steps and the token range of the next item are fetched an item ahead.
template <bool STRIDED>
struct LtItemWalk {
  int pos, end, step;       // position of the current item (STRIDED: the item itself), end, step
  int ci, ci1, ci2;         // (user, chunk) index of the current item, the next, and the one after
  int b0, b1, b2;           // their users (-1: none)
  int tok0, tok1, single;   // token range of the current item; 1 if its user has this chunk only
  int nc0, nc1, no0, no1;   // next item: its user's first chunk, first chunk of the user after, same for the rows (not combined
                            // before they are needed: the reads stay in flight)
  const int32_t* items; const int32_t* chunk_user; const int32_t* chunk_start; const int32_t* off;
  int chunk;
  __device__ __forceinline__ void fetch(int b) {
    nc0 = __ldg(chunk_start + b); nc1 = __ldg(chunk_start + b + 1); no0 = __ldg(off + b); no1 = __ldg(off + b + 1);
  }
  __device__ __forceinline__ void take() {
    tok0 = no0 + (ci - nc0) * chunk;
    tok1 = min(no1, tok0 + chunk);
    single = (nc1 - nc0 == 1) ? 1 : 0;
  }
  __device__ __forceinline__ int item(int ps) const { return ps < end ? (STRIDED ? ps : __ldg(items + ps)) : -1; }
  __device__ __forceinline__ void init(const LinkAttnTmemParams& p, int first, int last, int step_) {
    items = p.group_items; chunk_user = p.chunk_user; chunk_start = p.chunk_start; off = p.off; chunk = __ldg(p.chunk);
    pos = first; end = last; step = step_;
    ci = item(pos);
    ci1 = item(pos + step);
    ci2 = -1;
    b0 = ci >= 0 ? __ldg(chunk_user + ci) : -1;
    b1 = ci1 >= 0 ? __ldg(chunk_user + ci1) : -1;
    b2 = -1;
    tok0 = tok1 = single = nc0 = nc1 = no0 = no1 = 0;
    if (b0 >= 0) { fetch(b0); take(); }
    if (b1 >= 0) fetch(b1);
  }
  __device__ __forceinline__ bool valid() const { return pos < end; }
  __device__ __forceinline__ void prefetch() {
    ci2 = item(pos + 2 * step);
    b2 = ci2 >= 0 ? __ldg(chunk_user + ci2) : -1;
  }
  __device__ __forceinline__ void advance() {
    pos += step; ci = ci1; ci1 = ci2; b0 = b1; b1 = b2;
    take();
    if (b1 >= 0) fetch(b1);
  }
};

template <class G>
__global__ void __launch_bounds__(G::THREADS, 1)
k_link_attn_tmem_tc(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmQ2, const LinkAttnTmemParams p) {
  using namespace tc;
  constexpr int D = G::D, TILE = G::TILE, COLS = G::COLS, PARTS = G::PARTS, OUT = G::OUT, XSTAGES = G::XSTAGES, SBUFS = G::SBUFS, QBUFS = G::QBUFS;
  using Walk = LtItemWalk<G::STRIDED>;
  extern __shared__ __align__(1024) uint8_t smem[];
  if ((smem_u32(smem) & 1023u) != 0) {                     // the swizzled tiles need a 1024-byte aligned base
    pdl_wait();                                               // nobody leaves ahead of it (lime_common.cuh)
    if (threadIdx.x == 0) atomicCAS(p.err, 0, 97);
    return;
  }
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + G::OFF_BAR);
  uint64_t* x_full = bars;             // [5]
  uint64_t* x_empty = bars + 5;        // [5]  value contraction of the tile done (its tokens, its P, the accumulator)
  uint64_t* s_full = bars + 10;         // [3]  score tile in TMEM
  uint64_t* p_ready = bars + 13;       // [3]  P in TMEM over those scores (the four warps of the tile's group)
  uint64_t* q_full = bars + 16;        // [2]  folded queries of a user landed
  uint64_t* q_empty = bars + 18;       // [2]  every score MMA that reads them has run
  uint64_t* o_free = bars + 20;        //      accumulator of the item read out (all softmax warps)
  uint64_t* row_bar = bars + 21;       // [4]  rendezvous of the warps that share a TMEM lane quarter (end of an item)
  uint64_t* mref_bar = bars + 25;      // [2 tile parities][4 quarters]  reference maxima after the tile published (and the
                                       //                                previous ones read) by the handling group's warps
  uint64_t* part_bar = bars + 33;      // [2 groups][4 quarters]  row maxima of the parts written
  uint64_t* s_free = bars + 41;        // [3]  the buffer's probabilities are in use by a contraction issued already
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 44);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < XSTAGES; ++s) { mbar_init(&x_full[s], 1); mbar_init(&x_empty[s], 1); }
    for (int i = 0; i < SBUFS; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_ready[i], G::GROUP_WARPS); mbar_init(&s_free[i], 1); }
    for (int i = 0; i < QBUFS; ++i) { mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 1); }
    mbar_init(o_free, G::SOFTMAX_WARPS);
    for (int i = 0; i < 4; ++i) mbar_init(&row_bar[i], G::GROUPS * PARTS);
    for (int i = 0; i < 8; ++i) { mbar_init(&mref_bar[i], PARTS); mbar_init(&part_bar[i], PARTS); }
    fence_barrier_init();
    prefetch_tmap(&tmX); prefetch_tmap(&tmQ2);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, G::TMEM_COLS); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // set-up done: the next kernel's CTAs may become resident; nothing an earlier kernel wrote is read before this wait
  pdl_launch_dependents();
  pdl_wait();

  // gridDim % RB == 0: a CTA keeps one row block for its whole life, and the RB CTAs of a group walk the same items, so
  // the history rows they share meet in L2
  const int rb = (int)blockIdx.x % p.RB, grp_idx = (int)blockIdx.x / p.RB;
  const int it_first = G::STRIDED ? grp_idx : __ldg(p.group_start + grp_idx);
  const int it_end = G::STRIDED ? __ldg(p.chunk_start + p.B) : __ldg(p.group_start + grp_idx + 1);
  const int it_step = G::STRIDED ? (int)gridDim.x / p.RB : 1;
  const bool active = it_first < it_end;

  if (warp < 4) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(G::REGS_CONTROL));
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0 && active) {
      const uint64_t pol_stream = policy_evict_first(), pol_keep = policy_evict_last();
      bool ok = true;
      int g = 0, qn = 0, prev_user = -1;
      Walk w;
      for (w.init(p, it_first, it_end, it_step); w.valid() && ok; w.advance()) {
        w.prefetch();
        const int b = w.b0;
        const bool load_q = p.shared ? (qn == 0) : (b != prev_user);
        prev_user = b;
        if (load_q) {
          const int qb = qn % QBUFS;
          if (!mbar_wait(&q_empty[qb], ((uint32_t)(qn / QBUFS) & 1u) ^ 1u, p.err, 42)) { ok = false; break; }
          mbar_arrive_expect_tx(&q_full[qb], G::Q_BUF);
          for (int kb = 0; kb < D / 64; ++kb)
            tma_load_2d_hint(smem + G::OFF_Q2 + qb * G::Q_BUF + kb * G::QSUB, &tmQ2, kb * 64, (p.shared ? 0 : b) * p.HL + rb * 128,
                             &q_full[qb], pol_keep);
          ++qn;
        }
        const int n_tiles = (w.tok1 - w.tok0 + TILE - 1) / TILE;
        for (int t = 0; t < n_tiles; ++t, ++g) {
          const int s = g % XSTAGES;
          if (!mbar_wait(&x_empty[s], ((uint32_t)(g / XSTAGES) & 1u) ^ 1u, p.err, 41)) { ok = false; break; }
          mbar_arrive_expect_tx(&x_full[s], G::X_STAGE);
          for (int kb = 0; kb < D / 64; ++kb)
            tma_load_2d_hint(smem + G::OFF_X + s * G::X_STAGE + kb * G::XSUB, &tmX, kb * 64, w.tok0 + t * TILE, &x_full[s], pol_stream);
        }
      }
      if (!ok || *(volatile int*)p.err != 0) {
        // giving up: let the copies already issued land (bounded) before this CTA's shared memory goes away
        for (int j = 0; j < g && j < XSTAGES; ++j)
          mbar_wait_quiet(&x_full[(g - 1 - j) % XSTAGES], (uint32_t)((g - 1 - j) / XSTAGES) & 1u);
        for (int j = 0; j < qn && j < QBUFS; ++j)
          mbar_wait_quiet(&q_full[(qn - 1 - j) % QBUFS], (uint32_t)((qn - 1 - j) / QBUFS) & 1u);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuers: scores here, values in the next warp
    // Two warps, because one cannot feed the pipe: between two batches it alone is at work, one dependent instruction
    // after the other (400 cycles each way, measured with the clock, for batches of 500).  In both the whole warp runs the
    // code and one elected lane issues, so that descriptors and TMEM addresses are warp-uniform values: inside a one-lane
    // branch every instruction's operands are first moved to uniform registers, and a 64-cycle MMA took 90 to issue.
    if (active) {
      constexpr uint32_t idesc_s = make_idesc_bf16(128, TILE);               // Q2 . X^T  : both K-major
      const uint32_t sbase = smem_u32(smem);
      const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
      const uint64_t dq0 = make_sdesc_k_sw128(sbase + G::OFF_Q2), dx0 = make_sdesc_k_sw128(sbase + G::OFF_X);
      uint64_t dq = dq0, dx = dx0;
      int xs = 0, ss = 0, qs = 0, prev_user = -1;                   // token stage, score buffer, next query buffer
      uint32_t xs_ph = 0, ss_ph = 0, qs_ph = 0;
      bool ok = true, first = true;
      Walk w;
      for (w.init(p, it_first, it_end, it_step); w.valid() && ok; w.advance()) {
        w.prefetch();
        const bool new_q = p.shared ? first : w.b0 != prev_user;
        prev_user = w.b0;
        first = false;
        if (new_q) {
          if (!__all_sync(0xffffffffu, mbar_wait(&q_full[qs], qs_ph, p.err, 50))) { ok = false; break; }
          dq = dq0 + (uint64_t)((uint32_t)qs * G::Q_BUF >> 4);
          if (++qs == QBUFS) { qs = 0; qs_ph ^= 1u; }
        }
        // will the producer replace the queries after this item?
        const bool replaced = !p.shared && w.b1 >= 0 && w.b1 != w.b0;
        const int n_tiles = (w.tok1 - w.tok0 + TILE - 1) / TILE;
        for (int t = 0; t < n_tiles; ++t) {
          // the buffer's last probabilities have been handed to the pipe (nothing to wait for in the first round)
          if (!__all_sync(0xffffffffu, mbar_wait(&s_free[ss], ss_ph ^ 1u, p.err, 54))) { ok = false; break; }
          if (!__all_sync(0xffffffffu, mbar_wait(&x_full[xs], xs_ph, p.err, 51))) { ok = false; break; }
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
              mma_bf16_ss(tmem_u + (uint32_t)ss * 128, dq + (((kk >> 2) * G::QSUB + (kk & 3) * 32) >> 4),
                          dx + (((kk >> 2) * G::XSUB + (kk & 3) * 32) >> 4), idesc_s, kk != 0);
            mma_commit(&s_full[ss]);
            if (replaced && t + 1 == n_tiles) mma_commit(&q_empty[QBUFS == 1 ? 0 : qs ^ 1]);        // the buffer taken last
          }
          __syncwarp();
          dx += G::X_STAGE >> 4;
          if (++xs == XSTAGES) { xs = 0; xs_ph ^= 1u; dx = dx0; }
          if (++ss == SBUFS) { ss = 0; ss_ph ^= 1u; }
        }
      }
    }
  } else if (warp == 2) {
    if (active) {
      constexpr uint32_t idesc_o = make_idesc_bf16(128, D, false, true);     // P . X     : B is MN-major
      const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
      const uint64_t dx0 = make_sdesc_mn_sw128(smem_u32(smem) + G::OFF_X, G::XSUB);
      uint64_t dx = dx0;
      int xv = 0, sv = 0;
      uint32_t sv_ph = 0, o_ph = 1u;
      bool ok = true;
      Walk w;
      for (w.init(p, it_first, it_end, it_step); w.valid() && ok; w.advance()) {
        w.prefetch();
        const int n_tiles = (w.tok1 - w.tok0 + TILE - 1) / TILE;
        // the first tile of an item overwrites the accumulator: the previous item must have been read out (the very
        // first wait asks for the phase before the first, which counts as passed)
        if (!__all_sync(0xffffffffu, mbar_wait(o_free, o_ph, p.err, 53))) { ok = false; break; }
        o_ph ^= 1u;
        for (int t = 0; t < n_tiles; ++t) {
          if (!__all_sync(0xffffffffu, mbar_wait(&p_ready[sv], sv_ph, p.err, 52))) { ok = false; break; }
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < TILE / 16; ++kk)      // contraction over the tile's tokens, 16 per instruction
              mma_bf16_ts(tmem_u + G::COL_O, tmem_u + (uint32_t)sv * 128 + kk * 16 / COLS * COLS + kk * 16 % COLS / 2, dx + ((kk * 2048) >> 4), idesc_o,
                          kk != 0 ? 1u : (t != 0 ? 1u : 0u));
            mma_commit(&x_empty[xv]);
            // the next scores may be issued over these probabilities: the fence orders them behind this contraction in the
            // pipe, so its completion is not waited for
            tc_fence_before();
            mbar_arrive(&s_free[sv]);
          }
          __syncwarp();
          dx += G::X_STAGE >> 4;
          if (++xv == XSTAGES) { xv = 0; dx = dx0; }
          if (++sv == SBUFS) { sv = 0; sv_ph ^= 1u; }
        }
      }
    }
  }
  } else {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(G::REGS_SOFTMAX));
  if (active) {
    // ------------------------------------------------------------------ softmax warps (4..)
    const int q = warp & 3;                                    // TMEM lane quarter of this warp
    const int sub = (warp - 4) >> 2, part = sub % PARTS;       // which of the threads of its row this is,
    const int grp = sub / PARTS;                               // which tiles it takes (g % GROUPS == grp)
    const uint32_t r = (uint32_t)(q * 32 + lane);              // (head, link) row == TMEM lane
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    float* exch_sums = reinterpret_cast<float*>(smem + G::OFF_EXCH);         // [2 item parities][GROUPS * PARTS][128]
    float* exch_max = exch_sums + 2 * G::GROUPS * PARTS * 128 + grp * 2 * PARTS * 128;    // [2][PARTS][128] of this group
    float* mref = exch_sums + (PARTS > 1 ? 4 : 2) * G::GROUPS * PARTS * 128;              // [2 tile parities][128]
    const int R = rb * 128 + (int)r;                            // row among all H * ell
    // rows are stored after a 4 x 4 transpose of 16-byte chunks inside each group of four lanes: lane 4j+i then holds
    // chunk i of rows 4j..4j+3, so every store instruction writes whole 64-byte row parts.  Four consecutive rows share
    // a head (ell is a multiple of 4), so they are H * d elements apart.
    const int R4 = rb * 128 + q * 32 + (lane & ~3);
    const int64_t ohat_off = (int64_t)(R4 % p.ell) * (p.H * D) + (R4 / p.ell) * D + sub * OUT + (lane & 3) * 8;
    auto xchg = [&](uint4& keep_lo, uint4& keep_hi, bool upper, int dist) {
      // lanes with `upper` clear give away keep_hi and receive into it; lanes with it set give away keep_lo
      uint4 send = upper ? keep_lo : keep_hi, recv;
      recv.x = __shfl_xor_sync(0xffffffffu, send.x, dist); recv.y = __shfl_xor_sync(0xffffffffu, send.y, dist);
      recv.z = __shfl_xor_sync(0xffffffffu, send.z, dist); recv.w = __shfl_xor_sync(0xffffffffu, send.w, dist);
      if (upper) keep_lo = recv; else keep_hi = recv;
    };
    auto transpose4 = [&](uint4 (&t)[4]) {
      xchg(t[0], t[1], (lane & 1) != 0, 1);
      xchg(t[2], t[3], (lane & 1) != 0, 1);
      xchg(t[0], t[2], (lane & 2) != 0, 2);
      xchg(t[1], t[3], (lane & 2) != 0, 2);
    };
    bool ok = true;
    int g = 0;
    uint32_t row_uses = 0, part_uses = 0;
    int sb = 0;                                                // score buffer of the tile, and how often the ring came round
    uint32_t sb_ph = 0;
    Walk w;
    for (w.init(p, it_first, it_end, it_step); w.valid() && ok; w.advance()) {
      w.prefetch();
      const int b = w.b0, tok0 = w.tok0, tok1 = w.tok1;
      const int n_tiles = (tok1 - tok0 + TILE - 1) / TILE;
      // m_own: the reference maximum this thread's row sum is relative to; l_sum: sum over its columns and tiles
      float m_own = -INFINITY, l_sum = 0.f;
      for (int t = 0; t < n_tiles && ok; ++t, ++g) {
        const int buf = sb;
        const uint32_t buf_ph = sb_ph;
        if (++sb == SBUFS) { sb = 0; sb_ph ^= 1u; }
        if (G::GROUPS > 1 && (g & 1) != grp) continue;         // the other group's tile
        const uint32_t s_addr = lane_addr + (uint32_t)buf * 128 + (uint32_t)(part * COLS);
        const int nvalid = tok1 - tok0 - t * TILE - part * COLS;          // of this thread's columns
        if (!mbar_wait(&s_full[buf], buf_ph, p.err, 63)) { ok = false; break; }
        tc_fence_after();
        float v[COLS];
#pragma unroll
        for (int c = 0; c < COLS / 32 * 32; c += 32) tmem_ld_32x32(s_addr + c, *reinterpret_cast<float(*)[32]>(&v[c]));
        if constexpr (COLS % 32 != 0) tmem_ld_32x16(s_addr + COLS / 32 * 32, *reinterpret_cast<float(*)[16]>(&v[COLS / 32 * 32]));
        tmem_wait_ld();
        if (nvalid < COLS) {
          // ragged last tile of the item: the columns past its end (rows of the next user, or the fill value) drop out
          const float dead = p.silu ? 0.f : -INFINITY;
#pragma unroll
          for (int j = 0; j < COLS; ++j)
            if (j >= nvalid) v[j] = dead;
        }
        if (p.silu) {
          // SiLU(s) / N(U) needs neither a reference maximum nor row sums: one pass, nothing shared between threads
          lt_probabilities<true, COLS>(v, 0.f, s_addr);
        } else {
          // four independent chains for the row maximum (a ragged tile's dead columns hold -inf)
          float mx0 = v[0], mx1 = v[1], mx2 = v[2], mx3 = v[3];
#pragma unroll
          for (int j = 4; j < COLS; j += 4) {
            mx0 = fmaxf(mx0, v[j]); mx1 = fmaxf(mx1, v[j + 1]); mx2 = fmaxf(mx2, v[j + 2]); mx3 = fmaxf(mx3, v[j + 3]);
          }
          float mx = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3));
          if (PARTS > 1) {
            float* slot = exch_max + (part_uses & 1u) * PARTS * 128;
            slot[part * 128 + r] = mx;
            __syncwarp();
            if (lane == 0) mbar_arrive(&part_bar[grp * 4 + q]);
            if (!mbar_wait(&part_bar[grp * 4 + q], part_uses & 1u, p.err, 67)) { ok = false; break; }
            ++part_uses;
#pragma unroll
            for (int i = 1; i < PARTS; ++i) mx = fmaxf(mx, slot[((part + i) % PARTS) * 128 + r]);
          }
          float m_prev = m_own;
          if (G::GROUPS > 1) {
            // the reference the other group left after the previous tile (every tile but the very first waits, whether or
            // not it uses the value: the two groups then never drift more than one tile apart)
            m_prev = -INFINITY;
            if (g > 0) {
              if (!mbar_wait(&mref_bar[((g - 1) & 1) * 4 + q], (uint32_t)((g - 1) >> 1) & 1u, p.err, 69)) { ok = false; break; }
              if (t > 0) m_prev = mref[((g - 1) & 1) * 128 + r];
            }
            if (m_prev != m_own && l_sum != 0.f) l_sum *= lt_ex2(m_own - m_prev);     // bring this group's sum up to date
          }
          // raise the reference maximum only when it is exceeded by more than the threshold (or unset)
          const bool need = mx > m_prev + LT_RESCALE_THRESHOLD;
          const float m_new = need ? mx : m_prev;
          const float factor = (need && m_prev != -INFINITY) ? lt_ex2(m_prev - m_new) : 1.0f;
          if (G::GROUPS > 1) {
            if (part == 0) mref[(g & 1) * 128 + r] = m_new;
            __syncwarp();
            if (lane == 0) mbar_arrive(&mref_bar[(g & 1) * 4 + q]);
          }
          if (__any_sync(0xffffffffu, need && t > 0)) {
            // the accumulator must be quiescent: wait for the previous tile's value contraction (no later one is issued
            // before this tile's P exists), then scale this thread's columns of the row (of all tiles' sums: the parts of
            // the group that handles the tile share them)
            if (!mbar_wait(&x_empty[(g - 1) % XSTAGES], (uint32_t)((g - 1) / XSTAGES) & 1u, p.err, 64)) { ok = false; break; }
            tc_fence_after();
#pragma unroll 1
            for (int c = part * (D / PARTS); c < (part + 1) * (D / PARTS); c += 32) {
              float a[32];
              tmem_ld_32x32(lane_addr + G::COL_O + c, a);
              tmem_wait_ld();
#pragma unroll
              for (int j = 0; j < 32; ++j) a[j] *= factor;
              tmem_st_32x32(lane_addr + G::COL_O + c, a);
            }
          }
          l_sum *= factor;
          m_own = m_new;
          l_sum += lt_probabilities<false, COLS>(v, m_own, s_addr);
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_ready[buf]);
      }
      if (!ok) break;
      // item result: the final reference (published with the last tile), the two partial sums, then the accumulator
      const int gl = g - 1;
      float* exch_sum = exch_sums + (row_uses & 1u) * G::GROUPS * PARTS * 128;
      if (!p.silu) {
        if (G::GROUPS > 1 && (gl & 1) != grp) {
          if (!mbar_wait(&mref_bar[(gl & 1) * 4 + q], (uint32_t)(gl >> 1) & 1u, p.err, 70)) { ok = false; break; }
          const float m_fin = mref[(gl & 1) * 128 + r];
          if (m_fin != m_own && l_sum != 0.f) l_sum *= lt_ex2(m_own - m_fin);
          m_own = m_fin;
        }
        exch_sum[sub * 128 + r] = l_sum;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&row_bar[q]);
      if (!mbar_wait(&row_bar[q], row_uses & 1u, p.err, 68)) { ok = false; break; }
      ++row_uses;
      // SiLU mode normalises by the number of keys (Algorithm 1): this chunk's tokens, summed over the chunks by the merge
      float l_tot = (float)(tok1 - tok0);
      if (!p.silu) {
        l_tot = 0.f;
#pragma unroll
        for (int i = 0; i < G::GROUPS * PARTS; ++i) l_tot += exch_sum[i * 128 + r];
      }
      if (!mbar_wait(&x_empty[gl % XSTAGES], (uint32_t)(gl / XSTAGES) & 1u, p.err, 66)) { ok = false; break; }
      tc_fence_after();
      float a[OUT];
#pragma unroll
      for (int c = 0; c < OUT; c += 32) tmem_ld_32x32(lane_addr + G::COL_O + sub * OUT + c, *reinterpret_cast<float(*)[32]>(&a[c]));
      tmem_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(o_free);
      if (w.single != 0) {
        // the whole history of this user was one chunk: normalise and write the attention rows directly
        const float inv = 1.0f / l_tot;
        __nv_bfloat16* dst = p.Ohat + (int64_t)b * p.ell * (p.H * D) + ohat_off;
#pragma unroll
        for (int c = 0; c < OUT; c += 32) {
          uint4 tch[4];
#pragma unroll
          for (int c8 = 0; c8 < 4; ++c8) {
            const int j = c + c8 * 8;
            tch[c8] = make_uint4(lt_pack(a[j] * inv, a[j + 1] * inv), lt_pack(a[j + 2] * inv, a[j + 3] * inv),
                                 lt_pack(a[j + 4] * inv, a[j + 5] * inv), lt_pack(a[j + 6] * inv, a[j + 7] * inv));
          }
          transpose4(tch);
#pragma unroll
          for (int m = 0; m < 4; ++m) *reinterpret_cast<uint4*>(dst + (int64_t)m * (p.H * D) + c) = tch[m];
        }
      } else {
        // fp32 partial accumulator: runs of four 16-byte chunks, transposed the same way
        float* dst = p.part_acc + ((int64_t)w.ci * p.HL + R4) * D + sub * OUT + (lane & 3) * 4;
#pragma unroll
        for (int c = 0; c < OUT; c += 16) {
          uint4 tch[4];
#pragma unroll
          for (int c4 = 0; c4 < 4; ++c4) {
            const int j = c + c4 * 4;
            tch[c4] = make_uint4(__float_as_uint(a[j]), __float_as_uint(a[j + 1]), __float_as_uint(a[j + 2]), __float_as_uint(a[j + 3]));
          }
          transpose4(tch);
#pragma unroll
          for (int m = 0; m < 4; ++m) *reinterpret_cast<uint4*>(dst + (int64_t)m * D + c) = tch[m];
        }
        if (sub == 0) {
          const int64_t prow = (int64_t)w.ci * p.HL + R;
          p.part_m[prow] = p.silu ? 0.f : m_own;        // log2 domain; equal weights for the chunks in SiLU mode
          p.part_s[prow] = l_tot;
        }
      }
    }
  }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, G::TMEM_COLS);
  }
}

using LtD128 = LtCfg<128, 128, 5, 3, 1, 2, 1, true>;
using LtD256 = LtCfg<256, 96, 3, 2, 1, 1, 2, false>;

bool link_attn_d256_tc_supported(int dtype, int d, int H, int ell, int phi) {
  return dtype == LIME_BF16 && d == 256 && (H * ell) % 128 == 0 && H * ell <= 512 && ell % 4 == 0 &&
         (phi == LIME_PHI_SOFTMAX || phi == LIME_PHI_SILU);
}

int link_attn_d256_groups(int n_chunk_upper, int H, int ell) {
  const int RB = H * ell / 128;
  if (RB < 1) return 0;
  const int grid = n_chunk_upper * RB < kSMs ? n_chunk_upper * RB : kSMs;
  return grid / RB;
}

template <class G>
static lime_status launch_link_attn_tmem(const LinkAttnArgs& a, cudaStream_t st, bool (&smem_set)[kMaxDeviceOrdinals]) {
  if (a.n_chunk_upper <= 0 || a.total == 0) return LIME_OK;   // no history: the merge step writes zeros
  if (a.ln) return LIME_INVALID_ARG;                           // rows must arrive LayerNorm-ed
  CUtensorMap tmX, tmQ2;
  const uint64_t users = a.shared ? 1 : (uint64_t)a.B;
  if (!make_tmap_bf16_sw128(&tmX, a.hist, (uint64_t)a.total, G::D, G::D, G::TILE) ||
      !make_tmap_bf16_sw128(&tmQ2, a.Q2, users * (uint64_t)(a.H * a.ell), G::D, G::D, 128))
    return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
  if (!G::STRIDED && (a.group_start == nullptr || a.group_items == nullptr)) return LIME_INVALID_ARG;
  LinkAttnTmemParams p;
  p.group_start = a.group_start; p.group_items = a.group_items;
  p.off = a.off; p.chunk_start = a.chunk_start; p.chunk_user = a.chunk_user; p.silu = a.silu; p.B = a.B; p.chunk = a.chunk; p.shared = a.shared;
  p.ell = a.ell; p.H = a.H; p.HL = a.H * a.ell; p.RB = p.HL / 128; p.part_m = a.part_m; p.part_s = a.part_s; p.part_acc = a.part_acc;
  p.Ohat = (__nv_bfloat16*)a.Ohat; p.err = a.err;
  const int grid = link_attn_d256_groups(a.n_chunk_upper, a.H, a.ell) * p.RB;
  if (!G::STRIDED && a.n_groups * p.RB != grid) return LIME_INVALID_ARG;      // the schedule was dealt for another grid
  lime_status es = ensure_dynamic_smem((const void*)k_link_attn_tmem_tc<G>, (int)G::SMEM, smem_set);
  if (es != LIME_OK) return es;
  ProfScope _p("k_link_attn_tmem_tc", st);
  launch_pdl(k_link_attn_tmem_tc<G>, dim3(grid), dim3(G::THREADS), G::SMEM, st, tmX, tmQ2, p);
  LIME_LAUNCH_CHECK("k_link_attn_tmem_tc");
  return LIME_OK;
}

lime_status launch_link_attn_d128_tmem(const LinkAttnArgs& a, cudaStream_t st) {
  static bool smem_set[kMaxDeviceOrdinals] = {};
  return launch_link_attn_tmem<LtD128>(a, st, smem_set);
}
lime_status launch_link_attn_d256_tc(const LinkAttnArgs& a, cudaStream_t st) {
  static bool smem_set[kMaxDeviceOrdinals] = {};
  return launch_link_attn_tmem<LtD256>(a, st, smem_set);
}

}  // namespace lime
