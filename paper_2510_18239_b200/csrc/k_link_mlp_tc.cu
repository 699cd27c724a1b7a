// GatedMLP on the link rows of one XOR layer, fused with everything that consumes its result (bf16 operands, fp32
// accumulation in TMEM):
//
//   T^j = GatedMLP(O[T]) = ( SiLU(O[T] W_g) * (O[T] W_u) ) W_o                                   (Eq. 5 on link rows, Eq. 8)
//
// The attention kernel leaves Ohat [rows x H*d]: per (user, link) row the H un-projected head outputs side by side.
// d = d_ff = 128 (k_link_mlp_tc): W_V is folded into the gate / up weights (k_link_prep.cu)
//   1. [gate | up] [128 x 2*128] = Ohat_tile [128 x H*d] . [Mvg | Mvu]  streamed over K = H*d through a TMA stage ring
//   2. U = SiLU(gate) * up -> bf16 -> shared memory (A operand of the next contraction)
//   3. T^j = U [128 x 128] . W_o [128 x 128]
// d = d_ff = 256 (k_link_mlp_d256_tc): unfolded, as below.
// The epilogue, one thread pair per row, writes what the rest of the layer stack needs:
//   - T^j as fp32 (only when the caller asks for the layer's link rows)
//   - L^P (+)= T^j, the running sum of Eq. 8
//   - LN(T^j) as bf16, the A operand of the next layer's link-side GEMM (LayerNorm before the projections, App. C), or
//   - (d = 128, the next layer is the last) that layer's folded queries Q2 = LN(T^j) . W, the only operands it needs: four or
//     more tiles of 128 columns, formed here under the history update that runs beside this kernel, instead of a launch of
//     the link-side GEMM between the update and the next attention (256 users x 32 links: 6.5 us)
//   - on the last layer, the link states bf16(L^P) of Eq. 4 in its place when no candidate-side value projection follows
// One CTA per 128 rows.  Warp 0 TMA producer, warp 1 MMA issuer, warps 2-9 epilogue (two threads per row, half of the
// columns each; a warp may only touch the TMEM lane quarter warp_id % 4).
#include "lime_common.cuh"
#include "tc_common.cuh"

namespace lime {

constexpr int LM_THREADS = 64 + 256;
constexpr uint32_t LM_SUB = 128 * 128;                       // [128 rows x 64 bf16]
constexpr uint32_t LM_STAGE = 3 * LM_SUB;                    // A tile + 256 rows of B

// the output tile is staged over the operand buffers once the last contraction has finished
template <int D> struct LmOut {
  static constexpr int TS_LD = D + 4;                                  // floats per staged fp32 row (16-byte aligned, spread banks)
  static constexpr int TH_LD = D + 8;                                  // bf16 per staged LN row
  static constexpr uint32_t OFF_TH = 128 * TS_LD * 4;
  static constexpr uint32_t END = OFF_TH + 128 * TH_LD * 2;
};
struct LmLayout {                                                      // d = 128
  static constexpr int STAGES = 3;
  static constexpr uint32_t OFF_WO = STAGES * LM_STAGE;                // W_o^T: 2 K-blocks
  static constexpr uint32_t WO_BYTES = 2 * LM_SUB;
  static constexpr uint32_t OFF_U = OFF_WO + WO_BYTES;                 // U [128 x 128]: 2 K-blocks
  static constexpr uint32_t OPS_END = OFF_U + 2 * LM_SUB;
  // the queries of the next layer: LN(T) [128 x 128] behind the staged fp32 tile, a patch of 1 KB per epilogue warp, the weights of a
  // tile [128 x 128] over W_o and over U in turn
  static constexpr uint32_t OFF_LN = (LmOut<128>::OFF_TH + 1023) / 1024 * 1024, OFF_PATCH = OFF_LN + 2 * LM_SUB;
  static_assert(OFF_PATCH + 8 * 1024 <= OFF_WO && WO_BYTES == 2 * LM_SUB, "beside the operands of the last contraction");
  static constexpr uint32_t OFF_EXCH = OPS_END > LmOut<128>::END ? OPS_END : LmOut<128>::END;   // [2 slots][2 halves][128] floats
  static constexpr uint32_t OFF_BAR = OFF_EXCH + 4 * 128 * 4;
  static constexpr uint32_t SMEM = OFF_BAR + 256;
  static_assert(SMEM <= 232448, "shared memory budget of one CTA");
};
struct Lm256 {                                                         // d = 256
  static constexpr uint32_t OFF_O = 0;                                 // O [128 x 256] as value and remainder: 2 x 4 K-blocks
  static constexpr uint32_t HEADS_BYTES = 8 * LM_SUB;                  // before that: stages of [Ohat 128 x 64 | W_V^T d_h x 64]
  static constexpr uint32_t OFF_RING = HEADS_BYTES;                    // 2 slabs [256 rows x 64 of the contraction index]
  static constexpr int RING = 2, MAX_HEAD_STAGES = 6;
  static constexpr uint32_t SLAB = 2 * LM_SUB;
  static constexpr uint32_t OFF_U = OFF_RING + RING * SLAB;            // U of half of the hidden columns: 2 K-blocks
  static constexpr uint32_t OFF_EXCH = OFF_U + 2 * LM_SUB;
  static constexpr uint32_t OFF_BAR = OFF_EXCH + 4 * 128 * 4;
  static constexpr uint32_t SMEM = OFF_BAR + 320;
  static_assert(LmOut<256>::END <= OFF_EXCH && SMEM <= 232448, "shared memory budget of one CTA");
};

struct LinkMlpParams {
  int64_t M;                    // rows (users x links)
  int kblocks;                  // H*d / 64
  int H;
  float* T_out;                 // nullable: fp32 [M x d]
  float* LP;                    // nullable: fp32 [M x d] running sum
  int lp_accumulate;            // 0: LP = T, 1: LP += T
  __nv_bfloat16* That_next;     // nullable: bf16 [M x d] = LN(T) (or T when ln == 0)
  __nv_bfloat16* Q2;            // nullable (d = 128): [users x H*ell x d], the next layer's queries
  int ell;
  __nv_bfloat16* link_states;   // nullable: bf16 [M x d] = LP after this layer, which is then not stored
  int ln;
  float ln_eps;
  int* err;
};

__device__ __forceinline__ uint32_t lm_pack(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float lm_tanh(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t lm_chunk(uint32_t r, uint32_t c) { return r * 128u + ((c ^ (r & 7u)) << 4); }

// U = SiLU(gate) * up for 64 hidden columns of a row: gates at `gates`, ups 128 TMEM columns further, U into K-block `ub`.
__device__ __forceinline__ void lm_glu(uint8_t* ub, uint32_t gates, uint32_t r) {
#pragma unroll
  for (int c = 0; c < 64; c += 32) {
    float gt[32], up[32];
    tc::tmem_ld_32x32(gates + c, gt);
    tc::tmem_ld_32x32(gates + 128 + c, up);
    tc::tmem_wait_ld();
#pragma unroll
    for (int c8 = 0; c8 < 4; ++c8) {
      float y[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float hx = 0.5f * gt[c8 * 8 + j];
        y[j] = fmaf(hx, lm_tanh(hx), hx) * up[c8 * 8 + j];
      }
      *reinterpret_cast<uint4*>(ub + lm_chunk(r, (uint32_t)(c >> 3) + c8)) =
          make_uint4(lm_pack(y[0], y[1]), lm_pack(y[2], y[3]), lm_pack(y[4], y[5]), lm_pack(y[6], y[7]));
    }
  }
}

// The epilogue of T = U . W_o, by the eight epilogue warps once the last contraction is done: this thread's D/2 columns of its row (TMEM
// columns col_out on), 64 at a time.
// With p.Q2 the rows LN(T) go to the operand at `ln_at` instead of global memory.  Returns whether every wait ended well.
template <int D>
__device__ __forceinline__ bool lm_epilogue(const LinkMlpParams& p, uint8_t* smem, uint32_t lane_addr, uint32_t col_out, int64_t m0, int ew, int q, int half,
                                            uint32_t r, int lane, float* exch, uint64_t* all_bar, uint64_t* pair_bar, uint8_t* ln_at) {
  using namespace tc;
  using Lay = LmOut<D>;
  bool ok = true;
  constexpr int CH = D / 128;                                  // 64-column pieces per thread
  tc_fence_after();
  auto load64 = [&](int ch, float (&v)[64]) {
    float v0[32], v1[32];
    tmem_ld_32x32(lane_addr + col_out + half * (D / 2) + ch * 64, v0);
    tmem_ld_32x32(lane_addr + col_out + half * (D / 2) + ch * 64 + 32, v1);
    tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < 32; ++j) { v[j] = v0[j]; v[32 + j] = v1[j]; }
  };
  // T, the running sum of Eq. 8 and (last layer) the link states leave row by row: a thread owns half a row, so
  // direct accesses would touch 32 lines per instruction.  The tile is staged as fp32 over the operand buffers
  // (free since the last contraction finished) and each warp then moves whole rows.
  constexpr int TS_LD = Lay::TS_LD;
  float* Ts = reinterpret_cast<float*>(smem);
  float s = 0.f;
#pragma unroll
  for (int ch = 0; ch < CH; ++ch) {
    float v[64];
    load64(ch, v);
#pragma unroll
    for (int j = 0; j < 64; j += 4)
      *reinterpret_cast<float4*>(Ts + r * TS_LD + half * (D / 2) + ch * 64 + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
#pragma unroll
    for (int j = 0; j < 64; ++j) s += v[j];
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(all_bar);
  ok = mbar_wait(all_bar, 0, p.err, 79);
  if (ok) {
    // a warp takes rows ew, ew + 8, ...; the reads of the running sum for a batch of rows are issued together
    constexpr int BATCH = 8;
    const int n_valid = (int)(p.M - m0 < 128 ? p.M - m0 : 128);
    const bool acc = p.LP != nullptr && p.lp_accumulate != 0;
#pragma unroll 1
    for (int cb = 0; cb < D; cb += 128) {                    // 128 columns (one float4 per lane) at a time
      for (int i0 = ew; i0 < 128; i0 += 8 * BATCH) {
        float4 prev[BATCH];
#pragma unroll
        for (int k = 0; k < BATCH; ++k) {
          const int i = i0 + 8 * k;
          prev[k] = (acc && i < n_valid) ? *reinterpret_cast<const float4*>(p.LP + (m0 + i) * D + cb + lane * 4)
                                         : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < BATCH; ++k) {
          const int i = i0 + 8 * k;
          if (i >= n_valid) continue;
          float4 t = *reinterpret_cast<const float4*>(Ts + i * TS_LD + cb + lane * 4);
          const int64_t o = (m0 + i) * D + cb + lane * 4;
          if (p.T_out) *reinterpret_cast<float4*>(p.T_out + o) = t;
          if (p.LP) {
            t.x += prev[k].x; t.y += prev[k].y; t.z += prev[k].z; t.w += prev[k].w;
            if (p.link_states) *reinterpret_cast<uint2*>(p.link_states + o) = make_uint2(lm_pack(t.x, t.y), lm_pack(t.z, t.w));
            else *reinterpret_cast<float4*>(p.LP + o) = t;
          }
        }
      }
    }
  }
  if (p.That_next || p.Q2) {
    // LN(T) for the next layer's link-side GEMM: the two halves of a row exchange their partial sums
    float mu = 0.f, rstd = 1.f;
    if (p.ln) {
      uint32_t uses = 0;
      auto pair_sync = [&](int where) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&pair_bar[q]);
        const bool w = mbar_wait(&pair_bar[q], uses & 1u, p.err, where);
        ++uses;
        return w;
      };
      exch[half * 128 + r] = s;
      ok = ok && pair_sync(77);
      mu = (s + exch[(half ^ 1) * 128 + r]) * (1.0f / D);
      float var = 0.f;
#pragma unroll
      for (int ch = 0; ch < CH; ++ch) {
        float v[64];
        load64(ch, v);
#pragma unroll
        for (int j = 0; j < 64; ++j) { const float c = v[j] - mu; var = fmaf(c, c, var); }
      }
      exch[256 + half * 128 + r] = var;
      ok = ok && pair_sync(78);
      rstd = rsqrtf((var + exch[256 + (half ^ 1) * 128 + r]) * (1.0f / D) + p.ln_eps);
    }
    // the same way out for the bf16 rows: staged behind the fp32 tile, then whole rows per warp
    constexpr int TH_LD = Lay::TH_LD;
    __nv_bfloat16* Th = reinterpret_cast<__nv_bfloat16*>(smem + Lay::OFF_TH);
#pragma unroll
    for (int ch = 0; ch < CH; ++ch) {
      float v[64];
      load64(ch, v);
#pragma unroll
      for (int j = 0; j < 64; j += 8) {
        uint4 o;
        o.x = lm_pack((v[j] - mu) * rstd, (v[j + 1] - mu) * rstd); o.y = lm_pack((v[j + 2] - mu) * rstd, (v[j + 3] - mu) * rstd);
        o.z = lm_pack((v[j + 4] - mu) * rstd, (v[j + 5] - mu) * rstd); o.w = lm_pack((v[j + 6] - mu) * rstd, (v[j + 7] - mu) * rstd);
        if (p.Q2) *reinterpret_cast<uint4*>(ln_at + half * LM_SUB + lm_chunk(r, (uint32_t)(j >> 3))) = o;        // (D = 128)
        else *reinterpret_cast<uint4*>(Th + r * TH_LD + half * (D / 2) + ch * 64 + j) = o;
      }
    }
    if (p.Q2) return ok;
    __syncwarp();
    if (lane == 0) mbar_arrive(all_bar);
    ok = ok && mbar_wait(all_bar, 1, p.err, 80);
    if (ok) {
#pragma unroll 4
      for (int i = ew; i < 128; i += 8) {
        const int64_t grow = m0 + i;
        if (grow >= p.M) break;
#pragma unroll
        for (int cb = 0; cb < D; cb += 128)
          *reinterpret_cast<uint2*>(p.That_next + grow * D + cb + lane * 4) = *reinterpret_cast<const uint2*>(Th + i * TH_LD + cb + lane * 4);
      }
    }
  }
  return ok;
}

__global__ void __launch_bounds__(LM_THREADS, 1)
k_link_mlp_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              const __grid_constant__ CUtensorMap tmWo, const __grid_constant__ CUtensorMap tmQ, const LinkMlpParams p) {
  using namespace tc;
  using Lay = LmLayout;
  constexpr int D = 128, STAGES = Lay::STAGES;
  extern __shared__ __align__(1024) uint8_t smem[];
  if ((smem_u32(smem) & 1023u) != 0) {
    pdl_wait();                                               // nobody leaves ahead of it (lime_common.cuh)
    if (threadIdx.x == 0) atomicCAS(p.err, 0, 93);
    return;
  }
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Lay::OFF_BAR);
  uint64_t* full = bars;                 // [STAGES]
  uint64_t* empty = bars + 3;            // [STAGES]
  uint64_t* wo_full = bars + 6;          // W_o^T landed
  uint64_t* gu_full = bars + 7;          // [gate | up] complete
  uint64_t* u_ready = bars + 8;          // U in shared memory (8 warps)
  uint64_t* out_full = bars + 9;         // T complete
  uint64_t* pair_bar = bars + 10;        // [4], 2 warps each
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 14);
  uint64_t* ln_ready = bars + 16;        // LN(T) in shared memory, T read (8 warps)
  uint64_t* q_full = bars + 17;          // [2] weights of a tile of queries
  uint64_t* q_empty = bars + 19;         // [2]
  uint64_t* acc_full = bars + 21;        // [2] a tile of queries complete, in the columns of gate or up
  uint64_t* acc_empty = bars + 23;       // [2] read (8 warps)
  uint64_t* all_bar = bars + 15;         // rendezvous of the 8 epilogue warps (tiles staged in shared memory)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * 128;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(wo_full, 1); mbar_init(gu_full, 1); mbar_init(u_ready, 8); mbar_init(out_full, 1); mbar_init(ln_ready, 8);
    for (int i = 0; i < 2; ++i) { mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 1); mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 8); }
    for (int i = 0; i < 4; ++i) mbar_init(&pair_bar[i], 2);
    mbar_init(all_bar, 8);
    fence_barrier_init();
    prefetch_tmap(&tmA); prefetch_tmap(&tmB); prefetch_tmap(&tmWo);
    if (p.Q2) prefetch_tmap(&tmQ);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  constexpr uint32_t COL_GU = 0, COL_OUT = 256;
  // set-up done; nothing an earlier kernel wrote is read before this wait.  The signal follows it: a history update that runs beside
  // this kernel starts behind all that this one waits for (lime_common.cuh)
  pdl_wait();
  pdl_launch_dependents();

  if (warp == 0) {
    if (lane == 0) {
      const uint64_t pol = policy_evict_last();
      mbar_arrive_expect_tx(wo_full, Lay::WO_BYTES);
      for (int kb = 0; kb < 2; ++kb) tma_load_2d_hint(smem + Lay::OFF_WO + (uint32_t)kb * LM_SUB, &tmWo, kb * 64, 0, wo_full, pol);
      bool ok = true;
      int it = 0;
      for (int kb = 0; kb < p.kblocks; ++kb, ++it) {
        const int s = it % STAGES;
        if (!mbar_wait(&empty[s], ((uint32_t)(it / STAGES) & 1u) ^ 1u, p.err, 71)) { ok = false; break; }
        uint8_t* st = smem + (size_t)s * LM_STAGE;
        mbar_arrive_expect_tx(&full[s], LM_STAGE);
        tma_load_2d_hint(st, &tmA, kb * 64, m0, &full[s], pol);
        tma_load_2d_hint(st + LM_SUB, &tmB, kb * 64, 0, &full[s], pol);           // gate rows
        tma_load_2d_hint(st + 2 * LM_SUB, &tmB, kb * 64, D, &full[s], pol);       // up rows
      }
      // the next layer's query weights, a tile of 128 columns at a time, over W_o and U, once T has been formed from these
      int nq = 0;
      if (p.Q2 && ok) ok = mbar_wait(out_full, 0, p.err, 84);
      for (; p.Q2 && ok && nq < p.H; ++nq) {
        const int b = nq & 1;
        if (!mbar_wait(&q_empty[b], ((uint32_t)(nq >> 1) & 1u) ^ 1u, p.err, 85)) { ok = false; break; }
        mbar_arrive_expect_tx(&q_full[b], 2 * LM_SUB);
        for (int kb = 0; kb < 2; ++kb)
          tma_load_2d_hint(smem + (b ? Lay::OFF_U : Lay::OFF_WO) + (uint32_t)kb * LM_SUB, &tmQ, kb * 64, nq * 128, &q_full[b], pol);
      }
      if (!ok || *(volatile int*)p.err != 0) {
        for (int j = 0; j < it && j < STAGES; ++j)
          mbar_wait_quiet(&full[(it - 1 - j) % STAGES], (uint32_t)((it - 1 - j) / STAGES) & 1u);
        for (int j = 0; j < nq && j < 2; ++j) mbar_wait_quiet(&q_full[(nq - 1 - j) & 1], (uint32_t)((nq - 1 - j) >> 1) & 1u);
        mbar_wait_quiet(wo_full, 0);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc_256 = make_idesc_bf16(128, 256);
      constexpr uint32_t idesc_128 = make_idesc_bf16(128, 128);
      const uint32_t sbase = smem_u32(smem);
      bool ok = true;
      for (int it = 0; it < p.kblocks; ++it) {                   // 1. [gate | up]
        const int s = it % STAGES;
        if (!mbar_wait(&full[s], (uint32_t)(it / STAGES) & 1u, p.err, 72)) { ok = false; break; }
        tc_fence_after();
#pragma unroll
        for (int k = 0; k < 4; ++k)
          mma_bf16_ss(tmem_base + COL_GU, make_sdesc_k_sw128(sbase + s * LM_STAGE + k * 32),
                      make_sdesc_k_sw128(sbase + s * LM_STAGE + LM_SUB + k * 32), idesc_256, (it | k) != 0);
        mma_commit(&empty[s]);
      }
      if (ok) {
        mma_commit(gu_full);
        ok = mbar_wait(wo_full, 0, p.err, 74) && mbar_wait(u_ready, 0, p.err, 75);
      }
      if (ok) {
        tc_fence_after();                                        // 3. T = U . W_o
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t o = (uint32_t)(kk >> 2) * LM_SUB + (uint32_t)(kk & 3) * 32;
          mma_bf16_ss(tmem_base + COL_OUT, make_sdesc_k_sw128(sbase + Lay::OFF_U + o), make_sdesc_k_sw128(sbase + Lay::OFF_WO + o), idesc_128, kk != 0);
        }
        mma_commit(out_full);
      }
      if (p.Q2 && ok) ok = mbar_wait(ln_ready, 0, p.err, 86);
      for (int n = 0; p.Q2 && ok && n < p.H; ++n) {              // 4. the next layer's queries, over gate and up in turn
        const int b = n & 1;
        const uint32_t ph = (uint32_t)(n >> 1) & 1u;
        ok = mbar_wait(&acc_empty[b], ph ^ 1u, p.err, 87) && mbar_wait(&q_full[b], ph, p.err, 88);
        if (!ok) break;
        tc_fence_after();
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t o = (uint32_t)(kk >> 2) * LM_SUB + (uint32_t)(kk & 3) * 32;
          mma_bf16_ss(tmem_base + COL_GU + (uint32_t)b * 128, make_sdesc_k_sw128(sbase + Lay::OFF_LN + o),
                      make_sdesc_k_sw128(sbase + (b ? Lay::OFF_U : Lay::OFF_WO) + o), idesc_128, kk != 0);
        }
        mma_commit(&q_empty[b]);
        mma_commit(&acc_full[b]);
      }
    }
  } else {
    const int ew = warp - 2;                                   // 0..7
    const int q = warp & 3;
    const int half = ew >> 2;
    const uint32_t r = (uint32_t)(q * 32 + lane);
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    float* exch = reinterpret_cast<float*>(smem + Lay::OFF_EXCH);
    if (mbar_wait(gu_full, 0, p.err, 73)) {
      tc_fence_after();
      lm_glu(smem + Lay::OFF_U + half * LM_SUB, lane_addr + COL_GU + half * 64, r);          // 2.
      tc_fence_before();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(u_ready);
      bool ok = mbar_wait(out_full, 0, p.err, 76);
      if (ok) ok = lm_epilogue<D>(p, smem, lane_addr, COL_OUT, m0, ew, q, half, r, lane, exch, all_bar, pair_bar, smem + Lay::OFF_LN);
      if (p.Q2 && ok) {
        tc_fence_before();
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(ln_ready);
        // rows of a tile leave as whole 128-byte lines through the warp's patch, as in k_gemm_tc.cu
        uint8_t* patch = smem + Lay::OFF_PATCH + ew * 1024;
        const int row = m0 + (int)r, HL = p.H * p.ell;
        const int base_row = row < p.M ? row / p.ell * HL + row % p.ell : -1;
        const int x7 = lane & 7, rsub = lane >> 3;
        __nv_bfloat16* dst = p.Q2 + half * 64 + x7 * 8;
        for (int n = 0; n < p.H; ++n) {
          const int b = n & 1;
          if (!mbar_wait(&acc_full[b], (uint32_t)(n >> 1) & 1u, p.err, 89)) break;
          tc_fence_after();
          float v[64];
          tmem_ld_32x32(lane_addr + COL_GU + b * 128 + half * 64, *reinterpret_cast<float(*)[32]>(&v[0]));
          tmem_ld_32x32(lane_addr + COL_GU + b * 128 + half * 64 + 32, *reinterpret_cast<float(*)[32]>(&v[32]));
          tmem_wait_ld();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[b]);
          uint4 o[8];
#pragma unroll
          for (int c = 0; c < 8; ++c)
            o[c] = make_uint4(lm_pack(v[c * 8], v[c * 8 + 1]), lm_pack(v[c * 8 + 2], v[c * 8 + 3]), lm_pack(v[c * 8 + 4], v[c * 8 + 5]),
                              lm_pack(v[c * 8 + 6], v[c * 8 + 7]));
          const int out_row = base_row < 0 ? -1 : base_row + n * p.ell;
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            if (rsub == m) {
#pragma unroll
              for (int c = 0; c < 8; ++c) *reinterpret_cast<uint4*>(patch + x7 * 128 + ((c ^ x7) << 4)) = o[c];
            }
            __syncwarp();
            const uint4 o0 = *reinterpret_cast<const uint4*>(patch + rsub * 128 + ((x7 ^ rsub) << 4));
            const uint4 o1 = *reinterpret_cast<const uint4*>(patch + (rsub + 4) * 128 + ((x7 ^ (rsub + 4)) << 4));
            const int r0 = __shfl_sync(0xffffffffu, out_row, m * 8 + rsub), r1 = __shfl_sync(0xffffffffu, out_row, m * 8 + rsub + 4);
            if (r0 >= 0) *reinterpret_cast<uint4*>(dst + (int64_t)r0 * D) = o0;
            if (r1 >= 0) *reinterpret_cast<uint4*>(dst + (int64_t)r1 * D) = o1;
            __syncwarp();
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// d = d_ff = 256.  Folding W_V into W_g and W_u, as at d = 128, makes the contraction of [gate | up] H * d = 2048 wide at 8 heads: 2 MB of
// weights per 128 rows through L2 and Ohat twice (its accumulator takes two passes), 250 us a layer of 1024 users x 64 links.  Here
//   1. O[:, head] = Ohat_head [128 x 256] . W_V[:, head]    per head, streamed; O -> a bf16 value and its remainder (no rounding to speak of)
//   2. per half of the hidden columns: [gate | up] = O . [W_g | W_u]  ->  U = SiLU(gate) * up -> bf16
//   3. T (+)= U . W_o[that half, :]
// 1 MB per 128 rows instead of 3, half of it the rows' own, and a quarter of the operations: 128 users x 64 links x 8 heads 56 -> 33 us a
// launch, and the link states of four layers nearer fp64 (1.11 -> 0.99 % and 1.69 -> 1.51 % on two seeds: the folded weights were rounded
// once more).  What bounds it: HBM for Ohat, L^P and LN(T), 425 KB per 128 rows each way, and a tail of waves.  TMEM: O, then T, in the first 256 columns,
// [gate | up] of a half in the others.  The stages of 1 lie where O's two parts come to lie.
__global__ void __launch_bounds__(LM_THREADS, 1)
k_link_mlp_d256_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmGU,
                   const __grid_constant__ CUtensorMap tmWo, const LinkMlpParams p) {
  using namespace tc;
  using Lay = Lm256;
  constexpr int D = 256;
  extern __shared__ __align__(1024) uint8_t smem[];
  if ((smem_u32(smem) & 1023u) != 0) {
    pdl_wait();                                               // nobody leaves ahead of it (lime_common.cuh)
    if (threadIdx.x == 0) atomicCAS(p.err, 0, 93);
    return;
  }
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Lay::OFF_BAR);
  uint64_t* h_full = bars;               // [6] stages of step 1
  uint64_t* h_empty = bars + 6;          // [6]
  uint64_t* full = bars + 12;            // [2] weight slabs
  uint64_t* empty = bars + 14;           // [2]
  uint64_t* o_full = bars + 16;          // O complete
  uint64_t* o_ready = bars + 17;         // O in shared memory (8 warps)
  uint64_t* gu_full = bars + 18;         // [2] per half: [gate | up] complete
  uint64_t* u_ready = bars + 20;         // [2] per half: U in shared memory, [gate | up] read (8 warps)
  uint64_t* out_full = bars + 22;        // T complete
  uint64_t* pair_bar = bars + 23;        // [4], 2 warps each
  uint64_t* all_bar = bars + 27;         // rendezvous of the 8 epilogue warps (tiles staged in shared memory)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 28);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * 128, d_h = D / p.H;
  const uint32_t v_bytes = (uint32_t)d_h * 128, stage = LM_SUB + v_bytes;      // multiples of 1024: d_h is one of 8
  const int n_stages = min((int)(Lay::HEADS_BYTES / stage), Lay::MAX_HEAD_STAGES);

  if (threadIdx.x == 0) {
    for (int s = 0; s < Lay::MAX_HEAD_STAGES; ++s) { mbar_init(&h_full[s], 1); mbar_init(&h_empty[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); mbar_init(&gu_full[s], 1); mbar_init(&u_ready[s], 8); }
    mbar_init(o_full, 1); mbar_init(o_ready, 8); mbar_init(out_full, 1);
    for (int i = 0; i < 4; ++i) mbar_init(&pair_bar[i], 2);
    mbar_init(all_bar, 8);
    fence_barrier_init();
    prefetch_tmap(&tmA); prefetch_tmap(&tmV); prefetch_tmap(&tmGU); prefetch_tmap(&tmWo);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  constexpr uint32_t COL_O = 0, COL_GU = 256;                    // T over O
  // set-up done; nothing an earlier kernel wrote is read before this wait.  The signal follows it: a history update that runs beside
  // this kernel starts behind all that this one waits for (lime_common.cuh)
  pdl_wait();
  pdl_launch_dependents();

  if (warp == 0) {
    if (lane == 0) {
      const uint64_t pol = policy_evict_last(), pol_stream = policy_evict_first();
      // weight slabs in the order of use: per half four of [W_g | W_u]^T, two of W_o^T
      int sl = 0;
      auto slab = [&]() -> bool {
        const int s = sl % Lay::RING, half = sl / 6, i = sl % 6;
        if (!mbar_wait(&empty[s], ((uint32_t)(sl / Lay::RING) & 1u) ^ 1u, p.err, 71)) return false;
        uint8_t* dst = smem + Lay::OFF_RING + s * Lay::SLAB;
        mbar_arrive_expect_tx(&full[s], Lay::SLAB);
        if (i < 4) {
          tma_load_2d_hint(dst, &tmGU, i * 64, half * 128, &full[s], pol);                   // gate rows of this half
          tma_load_2d_hint(dst + LM_SUB, &tmGU, i * 64, D + half * 128, &full[s], pol);      // up rows
        } else {
          tma_load_2d_hint(dst, &tmWo, half * 128 + (i - 4) * 64, 0, &full[s], pol);
          tma_load_2d_hint(dst + LM_SUB, &tmWo, half * 128 + (i - 4) * 64, 128, &full[s], pol);
        }
        ++sl;
        return true;
      };
      bool ok = true;
      int it = 0;
      for (; it < p.kblocks && ok; ++it) {
        const int s = it % n_stages;
        if (!mbar_wait(&h_empty[s], ((uint32_t)(it / n_stages) & 1u) ^ 1u, p.err, 81)) { ok = false; break; }
        mbar_arrive_expect_tx(&h_full[s], stage);
        tma_load_2d_hint(smem + s * stage, &tmA, it * 64, m0, &h_full[s], pol_stream);
        tma_load_2d_hint(smem + s * stage + LM_SUB, &tmV, (it & 3) * 64, (it >> 2) * d_h, &h_full[s], pol);
        if (it + 1 == n_stages || it + 1 == p.kblocks)           // the first two are there when O is
          while (sl < Lay::RING && ok) ok = slab();
      }
      while (sl < 12 && ok) ok = slab();
      if (!ok || *(volatile int*)p.err != 0) {
        for (int j = 0; j < it && j < n_stages; ++j) mbar_wait_quiet(&h_full[(it - 1 - j) % n_stages], (uint32_t)((it - 1 - j) / n_stages) & 1u);
        for (int j = 0; j < sl && j < Lay::RING; ++j) mbar_wait_quiet(&full[(sl - 1 - j) % Lay::RING], (uint32_t)((sl - 1 - j) / Lay::RING) & 1u);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc_256 = make_idesc_bf16(128, 256);
      const uint32_t idesc_v = make_idesc_bf16(128, d_h);
      const uint32_t sbase = smem_u32(smem);
      bool ok = true;
      for (int it = 0; it < p.kblocks && ok; ++it) {             // 1. O, 256 of Ohat's columns a head
        const int s = it % n_stages;
        if (!mbar_wait(&h_full[s], (uint32_t)(it / n_stages) & 1u, p.err, 72)) { ok = false; break; }
        tc_fence_after();
#pragma unroll
        for (int k = 0; k < 4; ++k)
          mma_bf16_ss(tmem_base + COL_O + (uint32_t)((it >> 2) * d_h), make_sdesc_k_sw128(sbase + s * stage + k * 32),
                      make_sdesc_k_sw128(sbase + s * stage + LM_SUB + k * 32), idesc_v, ((it & 3) | k) != 0);
        mma_commit(&h_empty[s]);
      }
      if (ok) {
        mma_commit(o_full);
        ok = mbar_wait(o_ready, 0, p.err, 82);
      }
      int sl = 0;
      for (int half = 0; half < 2 && ok; ++half) {
        for (int i = 0; i < 6 && ok; ++i, ++sl) {
          const int s = sl % Lay::RING;
          // U of this half, and [gate | up] read
          if (i == 4) { mma_commit(&gu_full[half]); ok = mbar_wait(&u_ready[half], 0, p.err, 75); }
          if (ok) ok = mbar_wait(&full[s], (uint32_t)(sl / Lay::RING) & 1u, p.err, 74);
          if (!ok) break;
          tc_fence_after();
          const uint32_t b = sbase + Lay::OFF_RING + s * Lay::SLAB;
          if (i < 4) {                                           // 2. O's value, then its remainder
#pragma unroll
            for (int k = 0; k < 8; ++k)
              mma_bf16_ss(tmem_base + COL_GU, make_sdesc_k_sw128(sbase + Lay::OFF_O + ((k >> 2) * 4 + i) * LM_SUB + (k & 3) * 32),
                          make_sdesc_k_sw128(b + (k & 3) * 32), idesc_256, (i | k) != 0);
          } else {                                               // 3.
#pragma unroll
            for (int k = 0; k < 4; ++k)
              mma_bf16_ss(tmem_base + COL_O, make_sdesc_k_sw128(sbase + Lay::OFF_U + (i - 4) * LM_SUB + k * 32), make_sdesc_k_sw128(b + k * 32),
                          idesc_256, (half | (i - 4) | k) != 0);
          }
          mma_commit(&empty[s]);
        }
      }
      if (ok) mma_commit(out_full);
    }
  } else {
    const int ew = warp - 2;                                     // 0..7
    const int q = warp & 3;
    const int half = ew >> 2;
    const uint32_t r = (uint32_t)(q * 32 + lane);
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    float* exch = reinterpret_cast<float*>(smem + Lay::OFF_EXCH);
    bool ok = mbar_wait(o_full, 0, p.err, 83);
    if (ok) {
      // O as value and remainder, this thread's 128 columns, over the stages of step 1 (every contraction that read them is done)
      tc_fence_after();
#pragma unroll 1
      for (int c = 0; c < 128; c += 32) {
        float a[32];
        tmem_ld_32x32(lane_addr + COL_O + half * 128 + c, a);
        tmem_wait_ld();
        uint8_t* hi = smem + Lay::OFF_O + (half * 2 + (c >> 6)) * LM_SUB;
#pragma unroll
        for (int c8 = 0; c8 < 4; ++c8) {
          uint32_t h[4], l[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float x = a[c8 * 8 + 2 * j], y = a[c8 * 8 + 2 * j + 1];
            h[j] = lm_pack(x, y);
            l[j] = lm_pack(x - __uint_as_float(h[j] << 16), y - __uint_as_float(h[j] & 0xffff0000u));
          }
          const uint32_t at = lm_chunk(r, (uint32_t)((c & 63) >> 3) + c8);
          *reinterpret_cast<uint4*>(hi + at) = make_uint4(h[0], h[1], h[2], h[3]);
          *reinterpret_cast<uint4*>(hi + 4 * LM_SUB + at) = make_uint4(l[0], l[1], l[2], l[3]);
        }
      }
      tc_fence_before();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(o_ready);
    }
    for (int hf = 0; hf < 2 && ok; ++hf) {
      // (the last half's U has been read: gu_full is committed behind the contraction over it)
      if (!mbar_wait(&gu_full[hf], 0, p.err, 73)) { ok = false; break; }
      tc_fence_after();
      lm_glu(smem + Lay::OFF_U + half * LM_SUB, lane_addr + COL_GU + half * 64, r);
      tc_fence_before();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&u_ready[hf]);
    }
    if (ok && mbar_wait(out_full, 0, p.err, 76))
      lm_epilogue<D>(p, smem, lane_addr, COL_O, m0, ew, q, half, r, lane, exch, all_bar, pair_bar, nullptr);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// a.K = H * d; d = d_ff = a.d
lime_status launch_link_mlp_tc(const LinkMlpArgs& a, cudaStream_t st) {
  if (a.M == 0) return LIME_OK;
  if (a.d != 128 && a.d != 256) return LIME_UNSUPPORTED_SHAPE;
  const uint64_t K = (uint64_t)a.K, d = (uint64_t)a.d;
  const bool wide = a.d == 256;
  if (wide && a.K != 2 * 256 && a.K != 4 * 256 && a.K != 8 * 256) return LIME_UNSUPPORTED_SHAPE;
  CUtensorMap tmA, tmB, tmV, tmWo, tmQ;
  if (a.Q2 && (wide || a.WprepT == nullptr || a.ell < 1 || a.M * (a.K / 128) > 0x7fffffff)) return LIME_INVALID_ARG;
  if (!make_tmap_bf16_sw128(&tmA, a.Ohat, (uint64_t)a.M, K, K, 128) ||
      !make_tmap_bf16_sw128(&tmB, wide ? a.WguT : a.WpostT, 2 * d, wide ? d : K, wide ? d : K, 128) ||
      (wide && !make_tmap_bf16_sw128(&tmV, a.WvT, d, d, d, (uint32_t)(a.d * a.d / a.K))) || !make_tmap_bf16_sw128(&tmWo, a.WoT, d, d, d, 128) ||
      !make_tmap_bf16_sw128(&tmQ, a.Q2 ? a.WprepT : a.WoT, a.Q2 ? K : d, d, d, 128))
    return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
  LinkMlpParams p;
  p.M = a.M; p.kblocks = a.K / 64; p.H = a.K / a.d; p.T_out = a.T_out; p.LP = a.LP; p.lp_accumulate = a.lp_accumulate;
  p.Q2 = (__nv_bfloat16*)a.Q2; p.ell = a.ell; p.That_next = (__nv_bfloat16*)a.That_next; p.link_states = (__nv_bfloat16*)a.link_states; p.ln = a.ln; p.ln_eps = a.ln_eps;
  p.err = a.err;
  const dim3 grid((unsigned)((a.M + 127) / 128));
  static bool smem_set[2][kMaxDeviceOrdinals] = {};
  const lime_status es = wide ? ensure_dynamic_smem((const void*)k_link_mlp_d256_tc, (int)Lm256::SMEM, smem_set[1])
                              : ensure_dynamic_smem((const void*)k_link_mlp_tc, (int)LmLayout::SMEM, smem_set[0]);
  if (es != LIME_OK) return es;
  if (wide) {
    ProfScope _p("k_link_mlp_d256_tc", st);
    launch_pdl(k_link_mlp_d256_tc, grid, dim3(LM_THREADS), Lm256::SMEM, st, tmA, tmV, tmB, tmWo, p);
  } else {
    ProfScope _p("k_link_mlp_tc", st);
    launch_pdl(k_link_mlp_tc, grid, dim3(LM_THREADS), LmLayout::SMEM, st, tmA, tmB, tmWo, tmQ, p);
  }
  LIME_LAUNCH_CHECK("k_link_mlp_tc");
  return LIME_OK;
}

}  // namespace lime
