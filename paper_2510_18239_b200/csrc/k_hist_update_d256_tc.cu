// History update of one XOR layer on tcgen05 at d = d_ff = 256 with 64 links and 2, 4 or 8 heads or 32 links and 4 or 8
// heads (bf16 storage, rows LayerNorm-ed already):
//
//   S'[t,:] = GatedMLP( O[S]_t ),   O[S]_t = concat_h phi( Q[S]_{t,h} K[T]_{l,h}^T * scale ) V[T]_{l,h}          (Eq. 7, Eq. 5)
//   GatedMLP(A) = ( SiLU(A W_g) * (A W_u) ) W_o
//
// Per 128-token tile the chain of contractions never leaves the SM.  Scores are taken against the folded link keys K2
// (k_link_prep.cu: Q[S] is never formed), the value mix is done head by head against the plain link values V[T], and
// the GatedMLP weights follow unfolded - at this width folding W_V W_g into the link side (as the d = 128 kernels do)
// would cost twice the tensor work and twice the operand traffic:
//   scores [128 x H*ell] = X . K2^T, 256 stacked (head, link) rows per contraction
//   per-head softmax over the links, unnormalised (or SiLU(s) / ell) -> P (bf16)
//   O[:, head] = P_head [128 x ell] . V_head [ell x d_h]
//   O * 1 / (row sum of the head) -> bf16
//   per half hf of the hidden columns:   [gate | up] = O . [W_g | W_u][:, hf]  ->  U = SiLU(gate) * up (bf16)
//   S' = U . W_o
//   S' -> (LayerNorm) -> bf16 -> global memory
// Every contraction but the value mix is issued 256 columns wide: at 128 columns an MMA re-reads its A operand from
// shared memory twice as often per flop, and shared-memory bandwidth (operands in, TMA writes, the row warps) is what
// the tensor pipe waits for here.
// TMEM (512 columns) as two regions.  A: scores of the first 256 stacked rows, then P of all of them (a thread's bf16 pairs
// over its own scores: the first group's in the first half of its columns, the second's in the other), then [gate | up] of the
// first half, then U of both halves.  B: scores of the other 256 stacked rows, then O, then [gate | up] of the second half, then S'.
// P and U are A operands there: no shared memory, no proxy fence.  A takes the next tile's first scores right behind this tile's
// last contraction.  Both halves' [gate | up] are issued back to back, so that the second is formed while the row warps work on the
// first (one after the other in A, with S' begun in between: 266 us a launch of 128 users of 1024..4096 tokens, 64 links x 8 heads,
// this way 242; 64 users of 100..1024, 32 links x 4 heads 42 -> 38 us).
// Shared memory: X tile 64 KB (dead once the scores are formed, then O as bf16) and a ring of four 32 KB operand slabs
// ([256 rows x 64 of the contraction index]) through which K2, V[T]^T, [W_g | W_u] and W_o stream from L2 in the order the MMA
// issuer consumes them.  (16 KB slabs of 32 of the contraction index, 64-byte swizzle - half again as many in flight - were
// measured and lose: what limits the stream is not its depth but the 64-byte pieces.)
// Warp 0 TMA producer, warp 1 MMA issuer, warps 2-17 token rows: for the softmax one thread per token and 64 stacked rows of
// each region (one head of 64 links, or two of 32, whose maxima and sums are the two halves' own: no exchange between
// threads); elsewhere four threads share a token, a quarter of the columns each.
// Measured (1024 users of 1024..4096 tokens, 64 links x 8 heads): 27500 cycles a tile against 32000 with P and U in shared memory
// (over the token tile, so that the softmax had to wait for every score), 11300 of them tensor time; 2.65 -> 2.41 ms a launch at
// the 1 kW power cap, where the batch runs.  What is left: the chain of one tile (TMEM has no room for a second), of which the
// exponentials take 5400 and the rows' way out 7000.  The slabs (640 KB a tile from L2) are not what is waited for: with half the
// bytes copied the launch took as long.
#include "lime_common.cuh"
#include "tc_common.cuh"

namespace lime {

constexpr int HC_D = 256, HC_F = 256, HC_TILE = 128;
constexpr int HC_PARTS = 4, HC_ROW_WARPS = 4 * HC_PARTS, HC_THREADS = 64 + 32 * HC_ROW_WARPS;
constexpr int HC_RING = 4;
constexpr uint32_t HC_SUB = 128 * 128;                          // bytes of one [128 rows x 64 bf16] swizzled sub-tile
constexpr uint32_t HC_SLAB = 2 * HC_SUB;                        // one ring slot: [256 rows x 64 bf16]
constexpr uint32_t HC_OFF_XO = 0;                               // token tile, then O: 4 K-blocks
constexpr uint32_t HC_OFF_RING = HC_OFF_XO + 4 * HC_SUB;
constexpr uint32_t HC_PATCH = 8 * 128;                          // a row warp's own: 8 of its 32 rows on their way out
constexpr uint32_t HC_OFF_PATCH = HC_OFF_RING + HC_RING * HC_SLAB;
constexpr uint32_t HC_OFF_EXCH = HC_OFF_PATCH + HC_ROW_WARPS * HC_PATCH;   // [PARTS][128] float2
constexpr uint32_t HC_OFF_INV = HC_OFF_EXCH + HC_PARTS * 128 * 8;     // [8 heads][128 rows] 1 / softmax row sum
constexpr uint32_t HC_OFF_BAR = HC_OFF_INV + 8 * 128 * 4;
constexpr int HC_IDX_CAP = kEarlyUsers + 1;                     // users + 1 whose offsets are staged in shared memory
constexpr uint32_t HC_OFF_IDX = HC_OFF_BAR + 512;
constexpr uint32_t HC_SMEM = HC_OFF_IDX + 2 * HC_IDX_CAP * 4 + 8;
static_assert(HC_SMEM <= 232448, "shared memory budget of one CTA");

struct HistUpdate256Params {
  __nv_bfloat16* out;            // [total x d]
  const int32_t* off;            // [B+1]
  const int32_t* tile_start;     // [B+1] prefix of per-user tile counts (tile = 128 tokens)
  int B, H, HL, shared, out_ln;
  int silu;                      // 1: P = SiLU(scores) / ell (Algorithm 2) instead of the per-head softmax
  float ln_eps;
  BesideLinkSide beside;
  int* err;
};

__device__ __forceinline__ uint32_t hc_chunk(uint32_t r, uint32_t c) { return r * 128u + ((c ^ (r & 7u)) << 4); }
__device__ __forceinline__ uint32_t hc_pack(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float hc_tanh(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float hc_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ bool hc_group_sync(uint64_t* bar, uint32_t& uses, int lane, int* err, int where) {
  __syncwarp();
  if (lane == 0) tc::mbar_arrive(bar);
  const bool ok = tc::mbar_wait(bar, uses & 1u, err, where);
  ++uses;
  return ok;
}
struct HcTileUser {
  int b = -1, lo = 0, hi = 0;
  __device__ __forceinline__ int of(const int32_t* __restrict__ tile_start, int B, int t) {
    if (t < lo || t >= hi) {
      if (b < 0) b = upper_user(tile_start, B, t);
      else if (t >= hi) { do { ++b; } while (tile_start[b + 1] <= t); }
      else { do { --b; } while (tile_start[b] > t); }
      lo = tile_start[b];
      hi = tile_start[b + 1];
    }
    return b;
  }
};

template <int ELL>
__global__ void __launch_bounds__(HC_THREADS, 1)
k_hist_update_d256_tc(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmK2,
                      const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmWgu,
                      const __grid_constant__ CUtensorMap tmWo, const HistUpdate256Params p) {
  using namespace tc;
  extern __shared__ __align__(1024) uint8_t smem[];
  if ((smem_u32(smem) & 1023u) != 0) {
    pdl_wait();                                               // nobody leaves ahead of it (lime_common.cuh)
    if (threadIdx.x == 0) atomicCAS(p.err, 0, 96);
    return;
  }
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + HC_OFF_BAR);
  uint64_t* full = bars;              // [HC_RING] operand slab landed
  uint64_t* empty = bars + 4;         // [HC_RING] the MMAs that read the slab have run
  uint64_t* x_full = bars + 8;        // per tile
  uint64_t* x_free = bars + 9;        // per tile: the last contraction that reads the X / O buffer has run
  uint64_t* s_full = bars + 10;       // [2] per tile: scores in region A / B
  uint64_t* p_ready = bars + 12;      // per tile: P in TMEM, scores consumed (16 warps)
  uint64_t* o_full = bars + 13;       // per tile: O complete in TMEM
  uint64_t* o_ready = bars + 14;      // per tile: O as bf16 in smem (16 warps)
  uint64_t* gu_full = bars + 15;      // [2] per tile: [gate | up] of a half complete
  uint64_t* gu_read = bars + 17;      // per tile: [gate | up] of the second half in registers (16 warps)
  uint64_t* u_ready = bars + 18;      // [2] per tile: U of a half in TMEM (16 warps)
  uint64_t* sp_full = bars + 20;      // per tile: S' complete
  uint64_t* sp_read = bars + 21;      // per tile: S' read out of TMEM (16 warps)
  uint64_t* row_bar = bars + 22;      // [4] rendezvous of the four warps sharing a TMEM lane quarter
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 26);
  static_assert(HC_RING == 4, "barrier table above");

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr uint32_t V_ROW = ELL * 2;                        // bytes of a V[T]^T row (its swizzle span)
  constexpr uint32_t V_BYTES = HC_D * V_ROW;
  const int d_h = HC_D / p.H;
  const int n_sg = (p.HL + 255) / 256;                       // score contractions per tile (four heads each)
  const int sc_boxes = p.HL >= 256 ? 2 : 1;                  // 128-row boxes of K2 per score slab

  if (threadIdx.x == 0) {
    for (int i = 0; i < HC_RING; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(x_full, 1); mbar_init(x_free, 1);
    mbar_init(&s_full[0], 1); mbar_init(&s_full[1], 1); mbar_init(p_ready, HC_ROW_WARPS);
    mbar_init(o_full, 1); mbar_init(o_ready, HC_ROW_WARPS);
    mbar_init(&gu_full[0], 1); mbar_init(&gu_full[1], 1); mbar_init(gu_read, HC_ROW_WARPS); mbar_init(&u_ready[0], HC_ROW_WARPS); mbar_init(&u_ready[1], HC_ROW_WARPS);
    mbar_init(sp_full, 1); mbar_init(sp_read, HC_ROW_WARPS);
    for (int i = 0; i < 4; ++i) mbar_init(&row_bar[i], HC_PARTS);
    fence_barrier_init();
    prefetch_tmap(&tmX); prefetch_tmap(&tmK2); prefetch_tmap(&tmV); prefetch_tmap(&tmWgu); prefetch_tmap(&tmWo);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // set-up done: the next kernel's CTAs may become resident; nothing an earlier kernel wrote is read before this wait (beside the
  // link side: before everything up to the attention is complete, see lime_common.cuh)
  pdl_launch_dependents();
  if (!p.beside.early) pdl_wait();
  const int n_tiles_all = __ldcg(p.tile_start + p.B);
  const int t_begin = early_first_tile(blockIdx.x, gridDim.x, n_tiles_all, p.beside.late, p.beside.late_by);
  const int t_end = early_first_tile(blockIdx.x + 1, gridDim.x, n_tiles_all, p.beside.late, p.beside.late_by);
  const int n = t_end - t_begin;
  const int32_t* tile_start = p.tile_start;
  const int32_t* off = p.off;
  if (p.B + 1 <= HC_IDX_CAP) {
    int32_t* idx = reinterpret_cast<int32_t*>(smem + HC_OFF_IDX);
    for (int i = threadIdx.x; i <= p.B; i += HC_THREADS) { idx[i] = __ldcg(p.tile_start + i); idx[HC_IDX_CAP + i] = __ldcg(p.off + i); }
    tile_start = idx;
    off = idx + HC_IDX_CAP;
    __syncthreads();
  }

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0 && n > 0) {
      const uint64_t pol_stream = policy_evict_first(), pol_keep = policy_evict_last();
      bool ok = true;
      int g = 0, sl = 0;
      // one ring slab: one or two boxes of 128 rows at contraction offset x
      auto slab = [&](const CUtensorMap* m, int x, int y0, int y1, int boxes) -> bool {
        const int s = sl % HC_RING;
        if (!mbar_wait(&empty[s], ((uint32_t)(sl / HC_RING) & 1u) ^ 1u, p.err, 11)) return false;
        mbar_arrive_expect_tx(&full[s], (uint32_t)boxes * HC_SUB);
        tma_load_2d_hint(smem + HC_OFF_RING + s * HC_SLAB, m, x, y0, &full[s], pol_keep);
        if (boxes == 2) tma_load_2d_hint(smem + HC_OFF_RING + s * HC_SLAB + HC_SUB, m, x, y1, &full[s], pol_keep);
        ++sl;
        return true;
      };
      HcTileUser tu;
      for (; g < n && ok; ++g) {
        const int t = t_begin + g;
        const int b = tu.of(tile_start, p.B, t);
        const int urow = p.shared ? 0 : b;
        auto k2_slab = [&](int sg, int kb) -> bool {
          const int y = urow * p.HL + sg * 256;
          return slab(&tmK2, kb * 64, y, y + 128, sc_boxes);
        };
        // Operand slabs go out in the order of use.  The first K2 slab is requested BEFORE the wait for the X buffer: it
        // only needs a free ring slot, so it travels while the previous tile is still being finished.
        ok = k2_slab(0, 0);
        if (!ok) break;
        // the X / O buffer is free once the previous tile's last contraction over O has run
        if (g > 0 && !mbar_wait(x_free, (uint32_t)(g - 1) & 1u, p.err, 12)) { ok = false; break; }
        const int row0 = off[b] + (t - tu.lo) * HC_TILE;
        mbar_arrive_expect_tx(x_full, 4 * HC_SUB);
        for (int kb = 0; kb < 4; ++kb) tma_load_2d_hint(smem + HC_OFF_XO + kb * HC_SUB, &tmX, kb * 64, row0, x_full, pol_stream);
        for (int kb = 1; kb < 4 && ok; ++kb) ok = k2_slab(0, kb);
        for (int sg = 1; sg < n_sg && ok; ++sg)
          for (int kb = 0; kb < 4 && ok; ++kb) ok = k2_slab(sg, kb);
        if (!ok) break;
        // the user's link values, a slab of their own layout ([256 features x ell links])
        {
          const int s = sl % HC_RING;
          if (!mbar_wait(&empty[s], ((uint32_t)(sl / HC_RING) & 1u) ^ 1u, p.err, 13)) { ok = false; break; }
          mbar_arrive_expect_tx(&full[s], V_BYTES);
          tma_load_2d_hint(smem + HC_OFF_RING + s * HC_SLAB, &tmV, 0, urow * HC_D, &full[s], pol_keep);
          ++sl;
        }
        // then per half of the hidden columns the gate and up columns of W_g / W_u (contraction over d), and W_o
        for (int hf = 0; hf < 2; ++hf)
          for (int kb = 0; kb < 4 && ok; ++kb) ok = slab(&tmWgu, kb * 64, hf * 128, HC_F + hf * 128, 2);
        for (int kb = 0; kb < 4 && ok; ++kb) ok = slab(&tmWo, kb * 64, 0, 128, 2);
      }
      if (!ok || *(volatile int*)p.err != 0) {
        // giving up: let the copies already issued land (bounded) before this CTA's shared memory goes away
        const int gl = g < n ? g : n - 1;
        if (g > 0 || sl > 0) mbar_wait_quiet(x_full, (uint32_t)gl & 1u);
        for (int j = 0; j < sl && j < HC_RING; ++j) mbar_wait_quiet(&full[(sl - 1 - j) % HC_RING], (uint32_t)((sl - 1 - j) / HC_RING) & 1u);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // The whole warp runs this code and one elected lane issues (warp-uniform descriptors, see k_link_attn_tmem_tc.cu).
    if (n > 0) {
      constexpr uint32_t idesc_256 = make_idesc_bf16(128, 256);
      const uint32_t idesc_sc = p.HL >= 256 ? idesc_256 : make_idesc_bf16(128, 128);
      const uint32_t idesc_v = make_idesc_bf16(128, d_h);
      const uint32_t sbase = smem_u32(smem);
      const uint32_t A = __shfl_sync(0xffffffffu, tmem_base, 0), B = A + 256u;
      const uint64_t dxo = make_sdesc_k_sw128(sbase + HC_OFF_XO), dring = make_sdesc_k_sw128(sbase + HC_OFF_RING);
      auto wait = [&](uint64_t* bar, uint32_t parity, int where) -> bool {
        const bool got = __all_sync(0xffffffffu, mbar_wait(bar, parity, p.err, where));
        tc_fence_after();
        return got;
      };
      bool ok = true;
      uint32_t slot = 0, slot_ph = 0;
      auto next_slot = [&]() { if (++slot == HC_RING) { slot = 0; slot_ph ^= 1u; } };
      // one operand slab (64 of the contraction index): D[128 x N] (+)= X / O K-block . slab^T, then up to two commits
      auto slab_ss = [&](uint32_t d, int kb, uint32_t idesc, bool first, uint64_t* done, uint64_t* done2) -> bool {
        if (!wait(&full[slot], slot_ph, 22)) return false;
        if (elect_one()) {
          const uint64_t da = dxo + (uint64_t)((uint32_t)kb * HC_SUB >> 4), db = dring + (uint64_t)(slot * HC_SLAB >> 4);
#pragma unroll
          for (int k = 0; k < 4; ++k) mma_bf16_ss(d, da + ((k * 32) >> 4), db + ((k * 32) >> 4), idesc, (first && k == 0) ? 0u : 1u);
          mma_commit(&empty[slot]);
          if (done != nullptr) mma_commit(done);
          if (done2 != nullptr) mma_commit(done2);
        }
        __syncwarp();
        next_slot();
        return true;
      };
      // the same with U in TMEM: 64 hidden columns are two threads' 16 columns each, 32 apart
      auto slab_u = [&](int kb, bool first, uint64_t* done) -> bool {
        if (!wait(&full[slot], slot_ph, 22)) return false;
        if (elect_one()) {
          const uint64_t db = dring + (uint64_t)(slot * HC_SLAB >> 4);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            mma_bf16_ts(B, A + (uint32_t)((kb * 2 + (k >> 1)) * 32 + (k & 1) * 8), db + ((k * 32) >> 4), idesc_256, (first && k == 0) ? 0u : 1u);
          mma_commit(&empty[slot]);
          if (done != nullptr) mma_commit(done);
        }
        __syncwarp();
        next_slot();
        return true;
      };
      for (int g = 0; g < n && ok; ++g) {
        if (!wait(x_full, (uint32_t)g & 1u, 23)) break;
        // 1. scores.  A held U of the previous tile (handed to the pipe, which keeps the order); B its S'
        for (int kb = 0; kb < 4 && ok; ++kb) ok = slab_ss(A, kb, idesc_sc, kb == 0, kb == 3 ? &s_full[0] : nullptr, nullptr);
        if (!ok) break;
        if (g > 0 && !wait(sp_read, (uint32_t)(g - 1) & 1u, 26)) break;
        if (n_sg == 2)
          for (int kb = 0; kb < 4 && ok; ++kb) ok = slab_ss(B, kb, idesc_256, kb == 0, kb == 3 ? &s_full[1] : nullptr, nullptr);
        if (!ok) break;
        // 2. value mix, head by head: O[:, head] = P_head . V_head (contraction over the links of the head), over the scores of
        //    B, once they are all consumed
        if (!wait(&full[slot], slot_ph, 28) || !wait(p_ready, (uint32_t)g & 1u, 24)) break;
        if (elect_one()) {
          const uint64_t dv = make_sdesc_k_sw(sbase + HC_OFF_RING + slot * HC_SLAB, V_ROW);
          for (int h = 0; h < p.H; ++h) {
            const int row = h * ELL, c = row >> 7;          // stacked row, group of 128: P of 64 rows is 32 columns
            const uint32_t pa = A + (uint32_t)((c & 1) * 128 + ((row >> 6) & 1) * 64 + (c >> 1) * 32 + ((row & 63) >> 1));
#pragma unroll
            for (int kk = 0; kk < ELL / 16; ++kk)
              mma_bf16_ts(B + (uint32_t)(h * d_h), pa + kk * 8, dv + ((uint32_t)(h * d_h) * V_ROW >> 4) + ((kk * 32) >> 4), idesc_v, kk != 0);
          }
          mma_commit(&empty[slot]);
          mma_commit(o_full);
        }
        __syncwarp();
        next_slot();
        // 3. GatedMLP on O (bf16 in the X / O buffer), the hidden columns in two halves: the second's [gate | up] over O in B,
        //    under the row warps' work on the first
        if (!wait(o_ready, (uint32_t)g & 1u, 25)) break;
        for (int hf = 0; hf < 2; ++hf)
          for (int kb = 0; kb < 4 && ok; ++kb)
            ok = slab_ss(hf ? B : A, kb, idesc_256, kb == 0, kb == 3 ? &gu_full[hf] : nullptr, kb == 3 && hf == 1 ? x_free : nullptr);
        // S' over the second half's [gate | up], once that is in registers: U(0) . W_o[0..127, :] under the work on it
        for (int kb = 0; kb < 4 && ok; ++kb) {
          if ((kb & 1) == 0 && !wait(&u_ready[kb >> 1], (uint32_t)g & 1u, 27)) ok = false;
          if (kb == 0 && ok) ok = wait(gu_read, (uint32_t)g & 1u, 29);
          if (ok) ok = slab_u(kb, kb == 0, kb == 3 ? sp_full : nullptr);
        }
      }
    }
  } else if (n > 0) {
    // ------------------------------------------------------------------ token-row warps (2..17)
    const int rw = warp - 2;                                 // 0..15
    const int q4 = warp & 3;                                 // TMEM lane quarter of this warp
    const int part = rw >> 2;                                // which quarter of the columns of every step
    const uint32_t r = (uint32_t)(q4 * 32 + lane);           // token row of the tile == TMEM lane
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q4 * 32) << 16);
    constexpr uint32_t RA = 0, RB = 256;                     // the two regions
    float2* exch = reinterpret_cast<float2*>(smem + HC_OFF_EXCH);         // [PARTS][128]
    float* inv_sum = reinterpret_cast<float*>(smem + HC_OFF_INV);         // [8][128]
    uint8_t* patch = smem + HC_OFF_PATCH + rw * HC_PATCH;
    uint32_t row_uses = 0;
    bool ok = true;
    HcTileUser tu;
    for (int g = 0; g < n && ok; ++g) {
      const int t = t_begin + g;
      const int b = tu.of(tile_start, p.B, t);
      const int row0 = off[b] + (t - tu.lo) * HC_TILE;
      // ---- softmax over the links of this thread's heads: 64 stacked rows of either region, P over its own scores in A
      for (int sg = 0; sg < n_sg && ok; ++sg) {
        if (!mbar_wait(&s_full[sg], (uint32_t)g & 1u, p.err, 32)) { ok = false; break; }
        tc_fence_after();
        const int first = sg * 256 + part * 64;              // first stacked row
        if (first >= p.HL) break;
        float v[64];
        tmem_ld_32x32(lane_addr + (sg ? RB : RA) + part * 64, *reinterpret_cast<float(*)[32]>(&v[0]));
        tmem_ld_32x32(lane_addr + (sg ? RB : RA) + part * 64 + 32, *reinterpret_cast<float(*)[32]>(&v[32]));
        tmem_wait_ld();
#pragma unroll
        for (int h = 0; h < 64 / ELL; ++h) {                 // with ELL = 32 the two halves are heads of their own
          float2* w = reinterpret_cast<float2*>(&v[h * ELL]);
          float inv = 1.0f;
          if (p.silu) {
            // SiLU(s) / ell: every history query attends to the ell links of the head (Algorithm 1)
#pragma unroll
            for (int j = 0; j < ELL / 2; ++j) {
              const float2 hx = __fmul2_rn(w[j], make_float2(0.5f, 0.5f));
              w[j] = __fmul2_rn(__ffma2_rn(hx, make_float2(hc_tanh(hx.x), hc_tanh(hx.y)), hx), make_float2(1.0f / ELL, 1.0f / ELL));
            }
          } else {
            float m0 = w[0].x, m1 = w[0].y, m2 = w[1].x, m3 = w[1].y;
#pragma unroll
            for (int j = 2; j < ELL / 2; j += 2) {
              m0 = fmaxf(m0, w[j].x); m1 = fmaxf(m1, w[j].y); m2 = fmaxf(m2, w[j + 1].x); m3 = fmaxf(m3, w[j + 1].y);
            }
            const float mx = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
            float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll
            for (int j = 0; j < ELL / 2; j += 2) {
              const float2 a0 = __fadd2_rn(w[j], make_float2(-mx, -mx)), a1 = __fadd2_rn(w[j + 1], make_float2(-mx, -mx));
              w[j] = make_float2(hc_ex2(a0.x), hc_ex2(a0.y));
              w[j + 1] = make_float2(hc_ex2(a1.x), hc_ex2(a1.y));
              s0 = __fadd2_rn(s0, w[j]);
              s1 = __fadd2_rn(s1, w[j + 1]);
            }
            s0 = __fadd2_rn(s0, s1);
            inv = __fdividef(1.0f, s0.x + s0.y);
          }
          // the exponentials go to the value mix unnormalised; O is divided by the row sum of its head afterwards
          inv_sum[(first / ELL + h) * 128 + (int)r] = inv;
        }
#pragma unroll
        for (int c = 0; c < 64; c += 32) {
          float pk[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) pk[j] = __uint_as_float(hc_pack(v[c + 2 * j], v[c + 2 * j + 1]));
          tmem_st_32x16(lane_addr + RA + (uint32_t)(part * 64 + sg * 32 + (c >> 1)), pk);
        }
      }
      if (!ok) break;
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_ready);
      // ---- O: this thread's 64 columns / row sum of their heads -> bf16 -> K-block `part` of the X / P / O buffer
      if (!mbar_wait(o_full, (uint32_t)g & 1u, p.err, 33)) { ok = false; break; }
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < 64; c += 32) {
        float a[32];
        tmem_ld_32x32(lane_addr + RB + part * 64 + c, a);
        const float sc = inv_sum[((part * 64 + c) / d_h) * 128 + (int)r];
        tmem_wait_ld();
#pragma unroll
        for (int c8 = 0; c8 < 4; ++c8) {
          uint4 o;
          o.x = hc_pack(a[c8 * 8 + 0] * sc, a[c8 * 8 + 1] * sc); o.y = hc_pack(a[c8 * 8 + 2] * sc, a[c8 * 8 + 3] * sc);
          o.z = hc_pack(a[c8 * 8 + 4] * sc, a[c8 * 8 + 5] * sc); o.w = hc_pack(a[c8 * 8 + 6] * sc, a[c8 * 8 + 7] * sc);
          *reinterpret_cast<uint4*>(smem + HC_OFF_XO + part * HC_SUB + hc_chunk(r, (uint32_t)(c >> 3) + c8)) = o;
        }
      }
      tc_fence_before();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(o_ready);
      // ---- per half of the hidden columns: U = SiLU(gate) * up for this thread's 32 columns, over its own gates and ups of the
      //      first half
      for (int hf = 0; hf < 2 && ok; ++hf) {
        if (!mbar_wait(&gu_full[hf], (uint32_t)g & 1u, p.err, 34)) { ok = false; break; }
        tc_fence_after();
        float gt[32], up[32], pk[16];
        tmem_ld_32x32(lane_addr + (hf ? RB : RA) + part * 32, gt);
        tmem_ld_32x32(lane_addr + (hf ? RB : RA) + 128 + part * 32, up);
        tmem_wait_ld();
        if (hf == 1) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(gu_read);
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float2 hx = __fmul2_rn(make_float2(gt[2 * j], gt[2 * j + 1]), make_float2(0.5f, 0.5f));
          const float2 y = __fmul2_rn(__ffma2_rn(hx, make_float2(hc_tanh(hx.x), hc_tanh(hx.y)), hx), make_float2(up[2 * j], up[2 * j + 1]));
          pk[j] = __uint_as_float(hc_pack(y.x, y.y));
        }
        tmem_st_32x16(lane_addr + RA + (uint32_t)hf * 128 + part * 32, pk);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&u_ready[hf]);
      }
      if (!ok) break;
      // ---- S': this thread's 64 columns of its row -> (LayerNorm) -> bf16 -> global, straight from registers
      if (!mbar_wait(sp_full, (uint32_t)g & 1u, p.err, 37)) { ok = false; break; }
      tc_fence_after();
      float v[64];
      tmem_ld_32x32(lane_addr + RB + part * 64, *reinterpret_cast<float(*)[32]>(&v[0]));
      tmem_ld_32x32(lane_addr + RB + part * 64 + 32, *reinterpret_cast<float(*)[32]>(&v[32]));
      tmem_wait_ld();
      // S' is in registers: the columns may take the next tile's scores while this tile is normalised and stored
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(sp_read);
      if (p.out_ln) {
        // each quarter sends the mean of its 64 columns and their squared deviations from it; the four combine exactly.
        // (The slots are rewritten a tile later, when every warp has moved on.)
        float2* w = reinterpret_cast<float2*>(v);
        float2 s0 = w[0], s1 = w[1];
#pragma unroll
        for (int j = 2; j < 32; j += 2) { s0 = __fadd2_rn(s0, w[j]); s1 = __fadd2_rn(s1, w[j + 1]); }
        s0 = __fadd2_rn(s0, s1);
        const float m_q = (s0.x + s0.y) * (1.0f / 64);
        float2 q0 = make_float2(0.f, 0.f), q1 = q0;
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
          const float2 d0 = __fadd2_rn(w[j], make_float2(-m_q, -m_q)), d1 = __fadd2_rn(w[j + 1], make_float2(-m_q, -m_q));
          q0 = __ffma2_rn(d0, d0, q0);
          q1 = __ffma2_rn(d1, d1, q1);
        }
        q0 = __fadd2_rn(q0, q1);
        exch[part * 128 + r] = make_float2(m_q, q0.x + q0.y);
        if (!hc_group_sync(&row_bar[q4], row_uses, lane, p.err, 38)) { ok = false; break; }
        float2 e[HC_PARTS];
#pragma unroll
        for (int i = 0; i < HC_PARTS; ++i) e[i] = exch[i * 128 + r];
        const float mu = 0.25f * (e[0].x + e[1].x + e[2].x + e[3].x);
        float tot = 0.f;
#pragma unroll
        for (int i = 0; i < HC_PARTS; ++i) { const float dm = e[i].x - mu; tot += e[i].y + 64.0f * dm * dm; }
        const float rstd = rsqrtf(tot * (1.0f / HC_D) + p.ln_eps);
#pragma unroll
        for (int j = 0; j < 32; ++j) w[j] = __fmul2_rn(__fadd2_rn(w[j], make_float2(-mu, -mu)), make_float2(rstd, rstd));
      }
      // Out through the warp's own patch, eight rows of its 64 columns at a time (128 bytes a row, 16-byte chunk c at position
      // c ^ row: no bank conflicts), so that a store writes whole 128-byte lines.  (32-byte stores straight from the thread's
      // row, one line per lane, were measured: as fast here, 2 us slower in the d = 128 kernel.)
      const uint32_t x7 = (uint32_t)(lane & 7);
      const int rsub = lane >> 3, row_end = off[b + 1];
      __nv_bfloat16* dst = p.out + part * 64 + (lane & 7) * 8;
      uint4 o[8];
#pragma unroll
      for (int c = 0; c < 8; ++c)
        o[c] = make_uint4(hc_pack(v[c * 8], v[c * 8 + 1]), hc_pack(v[c * 8 + 2], v[c * 8 + 3]), hc_pack(v[c * 8 + 4], v[c * 8 + 5]),
                          hc_pack(v[c * 8 + 6], v[c * 8 + 7]));
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        if (rsub == m) {
#pragma unroll
          for (int c = 0; c < 8; ++c) *reinterpret_cast<uint4*>(patch + hc_chunk(x7, (uint32_t)c)) = o[c];
        }
        __syncwarp();
        const uint4 o0 = *reinterpret_cast<const uint4*>(patch + hc_chunk((uint32_t)rsub, x7));
        const uint4 o1 = *reinterpret_cast<const uint4*>(patch + hc_chunk((uint32_t)rsub + 4, x7));
        __syncwarp();
        const int row = row0 + q4 * 32 + m * 8 + rsub;
        if (row < row_end) *reinterpret_cast<uint4*>(dst + (int64_t)row * HC_D) = o0;
        if (row + 4 < row_end) *reinterpret_cast<uint4*>(dst + (int64_t)(row + 4) * HC_D) = o1;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
  if (p.beside.early) pdl_wait();                            // whoever waits for this kernel waits for the link side too
}

bool hist_update_d256_tc_supported(int dtype, int d, int f, int H, int ell, int phi, int gated_mlp) {
  return dtype == LIME_BF16 && d == HC_D && f == HC_F && ((ell == 64 && H == 2) || ((ell == 64 || ell == 32) && (H == 4 || H == 8))) &&
         (phi == LIME_PHI_SOFTMAX || phi == LIME_PHI_SILU) && gated_mlp != 0;
}

template <int ELL>
static lime_status launch_hist_update_d256_t(const HistUpdate256Args& a, cudaStream_t st) {
  if (a.total == 0) return LIME_OK;
  const int HL = a.H * ELL;
  CUtensorMap tmX, tmK2, tmV, tmWgu, tmWo;
  const uint64_t users = a.shared ? 1 : (uint64_t)a.B;
  if (!make_tmap_bf16_sw128(&tmX, a.hist_in, (uint64_t)a.total, HC_D, HC_D, HC_TILE) ||
      !make_tmap_bf16_sw128(&tmK2, a.K2, users * HL, HC_D, HC_D, 128) ||
      !make_tmap_bf16_kmajor(&tmV, a.V2t, users * HC_D, ELL, ELL, 256, ELL) ||
      !make_tmap_bf16_sw128(&tmWgu, a.WguT, 2 * HC_F, HC_D, HC_D, 128) ||
      !make_tmap_bf16_sw128(&tmWo, a.WoT, HC_D, HC_F, HC_F, 128))
    return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
  HistUpdate256Params p;
  p.out = (__nv_bfloat16*)a.hist_out; p.off = a.off; p.tile_start = a.tile_start; p.B = a.B; p.H = a.H; p.HL = HL;
  p.shared = a.shared; p.silu = a.silu; p.out_ln = a.out_ln; p.ln_eps = a.ln_eps; p.beside = a.beside; p.err = a.err;
  int grid = a.n_tile_upper < kSMs ? a.n_tile_upper : kSMs;
  if (grid < 1) return LIME_OK;
  static bool smem_set[kMaxDeviceOrdinals] = {};
  lime_status es = ensure_dynamic_smem((const void*)k_hist_update_d256_tc<ELL>, (int)HC_SMEM, smem_set);
  if (es != LIME_OK) return es;
  ProfScope _p("k_hist_update_d256_tc", st);
  launch_pdl(k_hist_update_d256_tc<ELL>, dim3(grid), dim3(HC_THREADS), HC_SMEM, st, tmX, tmK2, tmV, tmWgu, tmWo, p);
  LIME_LAUNCH_CHECK("k_hist_update_d256_tc");
  return LIME_OK;
}

lime_status launch_hist_update_d256_tc(const HistUpdate256Args& a, cudaStream_t st) {
  return a.ell == 32 ? launch_hist_update_d256_t<32>(a, st) : launch_hist_update_d256_t<64>(a, st);
}

}  // namespace lime
