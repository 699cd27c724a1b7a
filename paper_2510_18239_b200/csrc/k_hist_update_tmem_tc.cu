// History update of one XOR layer on tcgen05, two token tiles in flight per SM (bf16 storage, d = d_ff = 128, H * ell = 128 or
// 256):
//
//   S'[t,:] = GatedMLP( O[S]_t ),   O[S]_t = concat_h phi( Q[S]_{t,h} K[T]_{l,h}^T * scale ) V[T]_{l,h}          (Eq. 7, Eq. 5)
//
// With W_K and scale * log2(e) folded into the link keys (K2) and W_V with the GatedMLP's first weights into [G2 | U2]
// (k_link_prep.cu).  Rows that still need their LayerNorm (LN, the first layer of a raw lookup) get it afterwards, exact for
// the bf16 operands, from the statistics the attention kernel leaves.  More stacked rows: k_hist_update2_tc.cu.
//   scores [128 x HL]      = X . K2^T;   per-head softmax over the links (or SiLU(s) / ell) -> P (bf16)
//   [gate | up] [128 x 2f] = P . [G2 | U2];   U = SiLU(gate) * up (bf16);   S' = U . W_o -> (LayerNorm) -> bf16 -> global
// With `out_ln` the rows are written LayerNorm-ed: the next layer normalises every row it reads and nothing else reads them
// (Eq. 8).
//
// What bounds it: the chain of four contractions and three passes of the row warps between them, which takes several times
// the tensor time of a tile.  So two tiles are in the chain at once, half a period apart, each with its own issuing warp,
// its own eight row warps and its own half of TMEM, and the chain is kept short:
//  * P and U are A operands in TMEM, written over the thread's own scores: no shared memory, no proxy fence, and the
//    contractions read half as much of it.
//  * A tile has 256 TMEM columns, L and R.  Scores of the first 128 stacked rows in L, of the second in R, all their P in L;
//    [gate | up] of one half of the hidden columns at a time in R (the second half is formed while the row warps work on the
//    first, taken into registers); U over P; S' in R; and the next tile's scores are issued right behind S'.
//  * Shared memory: W_o resident, the user's K2, one token tile (dead once its scores are formed; it also keeps the two
//    tiles' scores in order), and a ring of 16 KB slabs of [G2 | U2] streamed from L2 in tile order.
// Warp 0 loads tokens and K2, warp 3 the slabs, warps 1 and 2 issue, each for every other tile.
// Measured: 32 users x 32768 tokens, 64 links (HL = 256) 352 -> 293 us a launch, the tensor pipe busy 40% of the time; 256
// users x 512 tokens, 32 links (HL = 128) 33 -> 31 us.  What is left is the row warps' chain.  Dropped: all sixteen row warps on
// every step of both tiles, four threads per token (372 us: a step takes as long, its TMEM loads and barriers are the same).
#include "lime_common.cuh"
#include "tc_common.cuh"

namespace lime {

constexpr int HT_D = 128, HT_F = 128, HT_TILE = 128;
constexpr int HT_PARTS = 2;                                   // threads per token row, 64 columns each
constexpr int HT_GROUP_WARPS = 4 * HT_PARTS, HT_THREADS = 128 + 2 * 32 * HT_GROUP_WARPS;
constexpr int HT_RING = 4;
constexpr uint32_t HT_SUB = 128 * 128;                        // bytes of one [128 rows x 64 bf16] swizzled sub-tile
constexpr uint32_t HT_OFF_WO = 0;                             // [d x f]: 2 K-blocks
constexpr uint32_t HT_OFF_K2 = HT_OFF_WO + 2 * HT_SUB;        // 256 stacked rows: one user's (HL = 256) or two users' (HL = 128)
constexpr uint32_t HT_OFF_X = HT_OFF_K2 + 4 * HT_SUB;         // token tile: 2 K-blocks
constexpr uint32_t HT_OFF_RING = HT_OFF_X + 2 * HT_SUB;       // slabs [64 gate rows, 64 up rows] x 64 of the contraction index
constexpr uint32_t HT_PATCH = 32 * 32;                        // a row warp's own: 8 of its 32 rows on their way out
constexpr uint32_t HT_OFF_PATCH = HT_OFF_RING + HT_RING * HT_SUB;
constexpr uint32_t HT_OFF_EXCH = HT_OFF_PATCH + 2 * HT_GROUP_WARPS * HT_PATCH;      // [2 groups][PARTS][128] float2 {mean, M2}
constexpr uint32_t HT_OFF_CK = HT_OFF_EXCH + 2 * HT_PARTS * 128 * 8;  // [2 groups][256] (LN) row sums of their user's K2
constexpr uint32_t HT_OFF_BAR = HT_OFF_CK + 2 * 256 * 4;
constexpr int HT_IDX_CAP = kEarlyUsers + 1;                             // users + 1 whose offsets are staged in shared memory (the
constexpr uint32_t HT_OFF_IDX = HT_OFF_BAR + 512;             // search for a tile's user is a chain of dependent reads)
constexpr uint32_t HT_SMEM = HT_OFF_IDX + 2 * HT_IDX_CAP * 4 + 8;
constexpr int HT_REGS_LAUNCH = 96, HT_REGS_CONTROL = 64, HT_REGS_ROWS = 104;     // registers a thread: at launch, after the split
static_assert(HT_SMEM <= 232448, "shared memory budget of one CTA");
static_assert(128 * HT_REGS_CONTROL + (HT_THREADS - 128) * HT_REGS_ROWS <= HT_THREADS * HT_REGS_LAUNCH, "register split");

struct HistUpdateTmemParams {
  __nv_bfloat16* out;            // [total x d]
  const float* cK;               // [users x HL] (LN) row sums of K2
  const float2* stats_in;        // (LN) {rstd, mean} of every row read, left by the attention kernel of the layer
  const int32_t* off;            // [B+1]
  const int32_t* tile_start;     // [B+1] prefix of per-user tile counts (tile = 128 tokens)
  int B, shared, out_ln;
  int silu;                      // 1: P = SiLU(scores) / ell (Algorithm 2) instead of the per-head softmax
  float ln_eps;
  BesideLinkSide beside;
  int* err;
};

__device__ __forceinline__ float ht_pack(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return __uint_as_float(*reinterpret_cast<uint32_t*>(&v));
}
__device__ __forceinline__ float ht_tanh(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ht_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// x * sigmoid(x) = x/2 * (1 + tanh(x/2)) of two numbers
__device__ __forceinline__ float2 ht_silu2(float2 x) {
  const float2 h = __fmul2_rn(x, make_float2(0.5f, 0.5f));
  return __ffma2_rn(h, make_float2(ht_tanh(h.x), ht_tanh(h.y)), h);
}
__device__ __forceinline__ bool ht_wait_all(uint64_t* bar, uint32_t parity, int* err, int where) {
  return __all_sync(0xffffffffu, tc::mbar_wait(bar, parity, err, where));
}

// User of tile t, cached: consecutive tiles are the same user most of the time, and when they are not the user is a
// neighbour of the cached one.  `seg` counts the changes of user since the first tile asked for.
struct HtTileUser {
  int b = -1, lo = 0, hi = 0, seg = 0;
  __device__ __forceinline__ int of(const int32_t* __restrict__ tile_start, int B, int t) {
    if (t >= hi) {
      if (b < 0) b = upper_user(tile_start, B, t);
      else { do { ++b; } while (tile_start[b + 1] <= t); ++seg; }
      lo = tile_start[b];
      hi = tile_start[b + 1];
    }
    return b;
  }
};

template <int NG, int ELL, bool LN>
__global__ void __launch_bounds__(HT_THREADS, 1)
k_hist_update_tmem_tc(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmK2,
                      const __grid_constant__ CUtensorMap tmG, const __grid_constant__ CUtensorMap tmU,
                      const __grid_constant__ CUtensorMap tmWo, const HistUpdateTmemParams p) {
  using namespace tc;
  static_assert(NG == 1 || NG == 2, "groups of 128 stacked rows");
  static_assert(64 % ELL == 0, "a thread owns whole heads");
  constexpr int KBUFS = 2 / NG;                               // users whose K2 is held
  constexpr int SLABS = 4 * NG;                               // slabs of a tile: halves x groups x 64 of 128 stacked rows
  extern __shared__ __align__(1024) uint8_t smem[];
  if ((smem_u32(smem) & 1023u) != 0) {                        // the swizzled tiles need a 1024-byte aligned base
    pdl_wait();                                               // nobody leaves ahead of it (lime_common.cuh)
    if (threadIdx.x == 0) atomicCAS(p.err, 0, 98);
    return;
  }
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + HT_OFF_BAR);
  uint64_t* full = bars;              // [HT_RING] slab landed
  uint64_t* empty = bars + 5;         // [HT_RING] the MMAs that read the slab have run
  uint64_t* x_empty = bars + 10;      // per tile: scores formed
  uint64_t* wo_full = bars + 11;
  uint64_t* k2_full = bars + 12;      // [2] per user
  uint64_t* k2_empty = bars + 14;     // [2] per user: its last scores formed
  // [2], by tile parity (a barrier with several waiters that skip phases would be mistaken for an earlier one)
  uint64_t* x_full = bars + 16;       // tokens landed
  uint64_t* s_full = bars + 18;       // scores in TMEM
  uint64_t* p_ready = bars + 20;      // P in TMEM (8 warps)
  uint64_t* gu_full = bars + 22;      // [gate | up] of a half in TMEM
  uint64_t* gu_read = bars + 24;      // first half taken into registers (8 warps)
  uint64_t* u_ready = bars + 26;      // U in TMEM, second half read (8 warps)
  uint64_t* sp_full = bars + 28;      // S' in TMEM
  uint64_t* sp_free = bars + 30;      // S' taken into registers (8 warps)
  uint64_t* slabs_used = bars + 32;   // every slab of the tile has landed and been handed to the pipe (the issuing warp)
  uint64_t* pair_bar = bars + 34;     // [2 groups][4 quarters] rendezvous of the two warps sharing token rows
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 42);
  static_assert(HT_RING <= 5, "barrier table above");

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < HT_RING; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(x_empty, 1); mbar_init(wo_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&k2_full[i], 1); mbar_init(&k2_empty[i], 1); mbar_init(&s_full[i], 1); mbar_init(&p_ready[i], HT_GROUP_WARPS);
      mbar_init(&gu_full[i], 1); mbar_init(&gu_read[i], HT_GROUP_WARPS); mbar_init(&u_ready[i], HT_GROUP_WARPS);
      mbar_init(&sp_full[i], 1); mbar_init(&sp_free[i], HT_GROUP_WARPS); mbar_init(&x_full[i], 1); mbar_init(&slabs_used[i], 1);
    }
    for (int i = 0; i < 8; ++i) mbar_init(&pair_bar[i], HT_PARTS);
    fence_barrier_init();
    prefetch_tmap(&tmX); prefetch_tmap(&tmK2); prefetch_tmap(&tmG); prefetch_tmap(&tmU); prefetch_tmap(&tmWo);
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
  const int n = t_end - t_begin;                              // tiles of this CTA, g = 0..n-1
  const int32_t* tile_start = p.tile_start;
  const int32_t* off = p.off;
  if (p.B + 1 <= HT_IDX_CAP) {
    int32_t* idx = reinterpret_cast<int32_t*>(smem + HT_OFF_IDX);
    for (int i = threadIdx.x; i <= p.B; i += HT_THREADS) { idx[i] = __ldcg(p.tile_start + i); idx[HT_IDX_CAP + i] = __ldcg(p.off + i); }
    tile_start = idx;
    off = idx + HT_IDX_CAP;
    __syncthreads();
  }

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(HT_REGS_CONTROL));
    if (warp == 0) {
      // ---------------------------------------------------------------- TMA producer: W_o, tokens, K2
      if (lane == 0 && n > 0) {
        const uint64_t pol_stream = policy_evict_first(), pol_keep = policy_evict_last();
        mbar_arrive_expect_tx(wo_full, 2 * HT_SUB);
        for (int kb = 0; kb < 2; ++kb) tma_load_2d_hint(smem + HT_OFF_WO + kb * HT_SUB, &tmWo, kb * 64, 0, wo_full, pol_keep);
        int g = 0, segs = 0;                                  // users' K2 requested
        bool ok = true;
        HtTileUser tu;
        for (; g < n && ok; ++g) {
          const int t = t_begin + g;
          const int b = tu.of(tile_start, p.B, t);
          if (p.shared ? segs == 0 : tu.seg == segs) {
            const int kb2 = segs % KBUFS;
            if (!mbar_wait(&k2_empty[kb2], ((uint32_t)(segs / KBUFS) & 1u) ^ 1u, p.err, 11)) { ok = false; break; }
            mbar_arrive_expect_tx(&k2_full[kb2], NG * 2 * HT_SUB);
            for (int i = 0; i < 2 * NG; ++i)
              tma_load_2d_hint(smem + HT_OFF_K2 + (kb2 * 2 * NG + i) * HT_SUB, &tmK2, (i & 1) * 64,
                               (p.shared ? 0 : b) * (NG * 128) + (i >> 1) * 128, &k2_full[kb2], pol_keep);
            ++segs;
          }
          if (g > 0 && !mbar_wait(x_empty, (uint32_t)(g - 1) & 1u, p.err, 12)) { ok = false; break; }
          const int row0 = off[b] + (t - tu.lo) * HT_TILE;
          mbar_arrive_expect_tx(&x_full[g & 1], 2 * HT_SUB);
          for (int kb = 0; kb < 2; ++kb) tma_load_2d_hint(smem + HT_OFF_X + kb * HT_SUB, &tmX, kb * 64, row0, &x_full[g & 1], pol_stream);
        }
        if (!ok || *(volatile int*)p.err != 0) {
          // giving up: let the copies already issued land (bounded) before this CTA's shared memory goes away
          if (g > 0) mbar_wait_quiet(&x_full[(g - 1) & 1], (uint32_t)((g - 1) >> 1) & 1u);
          for (int j = 0; j < segs && j < KBUFS; ++j)
            mbar_wait_quiet(&k2_full[(segs - 1 - j) % KBUFS], (uint32_t)((segs - 1 - j) / KBUFS) & 1u);
          mbar_wait_quiet(wo_full, 0);
        }
      }
    } else if (warp == 3) {
      // ---------------------------------------------------------------- TMA producer: slabs of [G2 | U2] in tile order
      if (lane == 0 && n > 0) {
        const uint64_t pol_keep = policy_evict_last();
        int sl = 0, slot = 0;
        uint32_t phase = 1u;                                  // the first round waits for the phase before the first: passed
        bool ok = true;
        HtTileUser tu;
        for (int g = 0; g < n && ok; ++g) {
          const int urow = p.shared ? 0 : tu.of(tile_start, p.B, t_begin + g);
          for (int i = 0; i < SLABS; ++i) {
            // half of the hidden columns, then group of stacked rows and 64 of them
            const int hf = i / (2 * NG), k = (i % (2 * NG)) * 64;
            if (!mbar_wait(&empty[slot], phase, p.err, 13)) { ok = false; break; }
            mbar_arrive_expect_tx(&full[slot], HT_SUB);
            uint8_t* dst = smem + HT_OFF_RING + slot * HT_SUB;
            tma_load_2d_hint(dst, &tmG, k, urow * HT_F + hf * 64, &full[slot], pol_keep);
            tma_load_2d_hint(dst + HT_SUB / 2, &tmU, k, urow * HT_F + hf * 64, &full[slot], pol_keep);
            ++sl;
            if (++slot == HT_RING) { slot = 0; phase ^= 1u; }
          }
        }
        if (!ok || *(volatile int*)p.err != 0)
          for (int j = 0; j < sl && j < HT_RING; ++j) mbar_wait_quiet(&full[(sl - 1 - j) % HT_RING], (uint32_t)((sl - 1 - j) / HT_RING) & 1u);
      }
    } else if (n > 0) {
      // ---------------------------------------------------------------- MMA issuers: warp 1 even tiles, warp 2 odd ones
      // The whole warp runs this code and one elected lane issues (warp-uniform descriptors, see k_link_attn_tmem_tc.cu).
      constexpr uint32_t idesc_128 = make_idesc_bf16(128, 128);
      const int grp = warp - 1;
      const uint32_t sbase = smem_u32(smem);
      const uint32_t L = __shfl_sync(0xffffffffu, tmem_base, 0) + (uint32_t)grp * 256u, R = L + 128u;
      const uint64_t dx = make_sdesc_k_sw128(sbase + HT_OFF_X), dk = make_sdesc_k_sw128(sbase + HT_OFF_K2);
      const uint64_t dw = make_sdesc_k_sw128(sbase + HT_OFF_WO), dr = make_sdesc_k_sw128(sbase + HT_OFF_RING);
      uint32_t i_ph = 0;                                      // parity of this group's tile count
      bool ok = ht_wait_all(wo_full, 0, p.err, 21);
      HtTileUser tu;
      for (int g = 0; g < n && ok; ++g) {
        const int t = t_begin + g;
        tu.of(tile_start, p.B, t);
        if ((g & 1) != grp) continue;
        const int seg = p.shared ? 0 : tu.seg;
        const bool last_of_user = !p.shared && g + 1 < n && t + 1 >= tu.hi;
        // 1. scores: L (its U has been handed to the pipe, which keeps the order), R once S' of the group's last tile is read
        //    (tokens first: they are requested after the user's K2, whose barrier is then in the phase asked for)
        if (!ht_wait_all(&x_full[grp], i_ph, p.err, 23)) break;
        if (!ht_wait_all(&k2_full[seg % KBUFS], (uint32_t)(seg / KBUFS) & 1u, p.err, 22)) break;
        if (NG == 2 && !ht_wait_all(&sp_free[grp], i_ph ^ 1u, p.err, 26)) break;
        const uint64_t dku = dk + (uint64_t)((uint32_t)(seg % KBUFS) * 2 * NG * HT_SUB >> 4);
        tc_fence_after();
        if (elect_one()) {
#pragma unroll
          for (int c = 0; c < NG; ++c)
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              mma_bf16_ss(c ? R : L, dx + (((kk >> 2) * HT_SUB + (kk & 3) * 32) >> 4),
                          dku + (((c * 2 + (kk >> 2)) * HT_SUB + (kk & 3) * 32) >> 4), idesc_128, kk != 0);
          mma_commit(&s_full[grp]);
          mma_commit(x_empty);
          if (last_of_user) mma_commit(&k2_empty[seg % KBUFS]);
        }
        __syncwarp();
        if (!ht_wait_all(&p_ready[grp], i_ph, p.err, 24)) break;
        if (NG == 1 && !ht_wait_all(&sp_free[grp], i_ph ^ 1u, p.err, 26)) break;
        // 2. [gate | up] of each half of the hidden columns: P in TMEM, the thread's own 64 score columns hold its P of
        //    every group, 32 columns each
        if (g > 0 && !ht_wait_all(&slabs_used[grp ^ 1], (uint32_t)((g - 1) >> 1) & 1u, p.err, 29)) break;
        uint32_t sl = (uint32_t)g * SLABS;
        for (int hf = 0; hf < 2 && ok; ++hf) {
          if (hf == 1 && !ht_wait_all(&gu_read[grp], i_ph, p.err, 27)) { ok = false; break; }
#pragma unroll
          for (int i = 0; i < 2 * NG; ++i, ++sl) {
            const uint32_t slot = sl % HT_RING;
            if (ok && !ht_wait_all(&full[slot], (sl / HT_RING) & 1u, p.err, 28)) ok = false;
            tc_fence_after();
            if (ok && elect_one()) {
              const uint64_t ds = dr + (uint64_t)(slot * HT_SUB >> 4);
#pragma unroll
              for (int k = 0; k < 4; ++k)
                mma_bf16_ts(R, L + (i & 1) * 64 + (i >> 1) * 32 + k * 8, ds + ((k * 32) >> 4), idesc_128, (i | k) != 0);
              mma_commit(&empty[slot]);
              if (i == 2 * NG - 1) mma_commit(&gu_full[grp]);
            }
            __syncwarp();
          }
        }
        if (!ok) break;
        if (lane == 0) mbar_arrive(&slabs_used[grp]);
        // 3. S' = U . W_o: the thread's U of half hf in columns 16 hf .. of its 64
        if (!ht_wait_all(&u_ready[grp], i_ph, p.err, 25)) break;
        tc_fence_after();
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {                    // hidden columns 16 kk ..: half kk / 4, thread (kk / 2) % 2
            mma_bf16_ts(R, L + ((kk >> 1) & 1) * 64 + (kk >> 2) * 16 + (kk & 1) * 8, dw + (((kk >> 2) * HT_SUB + (kk & 3) * 32) >> 4),
                        idesc_128, kk != 0);
          }
          mma_commit(&sp_full[grp]);
        }
        __syncwarp();
        i_ph ^= 1u;
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(HT_REGS_ROWS));
    // ------------------------------------------------------------------ token-row warps (4..19), eight per tile parity
    const int q4 = warp & 3;                                   // TMEM lane quarter of this warp
    const int grp = (warp - 4) / HT_GROUP_WARPS, part = ((warp - 4) >> 2) % HT_PARTS;
    const uint32_t r = (uint32_t)(q4 * 32 + lane);             // token row of the tile == TMEM lane
    const uint32_t base = tmem_base + (uint32_t)grp * 256u + ((uint32_t)(q4 * 32) << 16);
    const uint32_t L = base + (uint32_t)part * 64u, R = base + 128u;      // this thread's columns of L; R as a whole
    float2* exch = reinterpret_cast<float2*>(smem + HT_OFF_EXCH) + grp * HT_PARTS * 128;
    uint8_t* patch = smem + HT_OFF_PATCH + (warp - 4) * HT_PATCH;
    float* ck_s = reinterpret_cast<float*>(smem + HT_OFF_CK) + grp * 256;
    int ck_user = -1;
    uint32_t i_ph = 0, gu_ph = 0;
    bool ok = true;
    HtTileUser tu;
    for (int g = 0; g < n && ok; ++g) {
      const int t = t_begin + g;
      const int b = tu.of(tile_start, p.B, t);
      if ((g & 1) != grp) continue;
      const int row0 = off[b] + (t - tu.lo) * HT_TILE, row_end = off[b + 1];
      // ---- softmax over the links of this thread's heads, P over its own scores
      float rstd_r = 1.f, mu_r = 0.f;
      if (LN && row0 + (int)r < row_end) {
        const float2 st = __ldcg(p.stats_in + row0 + r);
        rstd_r = st.x; mu_r = st.y;
      }
      if (!mbar_wait(&s_full[grp], i_ph, p.err, 32)) { ok = false; break; }
      tc_fence_after();
      if (LN && b != ck_user && (ck_user < 0 || !p.shared)) {
        // these scores exist, so every warp of the group is past the softmax of its last tile (its U was needed first): nobody
        // still reads the last user's sums.  Every warp of a part writes the same values.
        const float* src = p.cK + (int64_t)(p.shared ? 0 : b) * (NG * 128) + part * 64;
#pragma unroll
        for (int c = 0; c < NG; ++c) {
          ck_s[c * 128 + part * 64 + lane] = __ldcg(src + c * 128 + lane);
          ck_s[c * 128 + part * 64 + 32 + lane] = __ldcg(src + c * 128 + 32 + lane);
        }
        __syncwarp();
      }
      ck_user = b;
#pragma unroll
      for (int c = 0; c < NG; ++c) {
        float v[64];
        const uint32_t src = c ? R + (uint32_t)part * 64u : L;
        tmem_ld_32x32(src, *reinterpret_cast<float(*)[32]>(&v[0]));
        tmem_ld_32x32(src + 32, *reinterpret_cast<float(*)[32]>(&v[32]));
        tmem_wait_ld();
        if (LN) {
          // s = rstd (raw - mu rowsum(K2)): the LayerNorm of the row, exact for the bf16 operands
          const float4* ck = reinterpret_cast<const float4*>(ck_s + c * 128 + part * 64);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float4 k = ck[j];
            float2* w = reinterpret_cast<float2*>(&v[4 * j]);
            w[0] = __fmul2_rn(__ffma2_rn(make_float2(-mu_r, -mu_r), make_float2(k.x, k.y), w[0]), make_float2(rstd_r, rstd_r));
            w[1] = __fmul2_rn(__ffma2_rn(make_float2(-mu_r, -mu_r), make_float2(k.z, k.w), w[1]), make_float2(rstd_r, rstd_r));
          }
        }
#pragma unroll
        for (int h = 0; h < 64 / ELL; ++h) {
          float2* w = reinterpret_cast<float2*>(&v[h * ELL]);
          float inv;
          if (p.silu) {
            // SiLU(s) / ell: every history query attends to the ell links of the head (Algorithm 1)
#pragma unroll
            for (int j = 0; j < ELL / 2; ++j) w[j] = ht_silu2(w[j]);
            inv = 1.0f / ELL;
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
              const float2 a = __fadd2_rn(w[j], make_float2(-mx, -mx)), c2 = __fadd2_rn(w[j + 1], make_float2(-mx, -mx));
              w[j] = make_float2(ht_ex2(a.x), ht_ex2(a.y));
              w[j + 1] = make_float2(ht_ex2(c2.x), ht_ex2(c2.y));
              s0 = __fadd2_rn(s0, w[j]);
              s1 = __fadd2_rn(s1, w[j + 1]);
            }
            s0 = __fadd2_rn(s0, s1);
            inv = __fdividef(1.f, s0.x + s0.y);
          }
#pragma unroll
          for (int j = 0; j < ELL / 2; ++j) w[j] = __fmul2_rn(w[j], make_float2(inv, inv));
        }
#pragma unroll
        for (int hv = 0; hv < 2; ++hv) {
          float pk[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) pk[j] = ht_pack(v[hv * 32 + 2 * j], v[hv * 32 + 2 * j + 1]);
          tmem_st_32x16(L + (uint32_t)(c * 32 + hv * 16), pk);
        }
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_ready[grp]);
      // ---- U = SiLU(gate) * up, this thread's 32 hidden columns of each half; over P once the second half has read it
      float u[2][16];
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        if (!mbar_wait(&gu_full[grp], gu_ph, p.err, 33)) { ok = false; break; }
        gu_ph ^= 1u;
        tc_fence_after();
        float gt[32], up[32];
        tmem_ld_32x32(R + (uint32_t)part * 32u, gt);
        tmem_ld_32x32(R + 64u + (uint32_t)part * 32u, up);
        tmem_wait_ld();
        if (hf == 0) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&gu_read[grp]);
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float2 y = __fmul2_rn(ht_silu2(make_float2(gt[2 * j], gt[2 * j + 1])), make_float2(up[2 * j], up[2 * j + 1]));
          u[hf][j] = ht_pack(y.x, y.y);
        }
      }
      if (!ok) break;
      tmem_st_32x16(L, u[0]);
      tmem_st_32x16(L + 16u, u[1]);
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&u_ready[grp]);
      // ---- this thread's 64 columns of its S' row -> (LayerNorm) -> bf16 -> global
      if (!mbar_wait(&sp_full[grp], i_ph, p.err, 34)) { ok = false; break; }
      tc_fence_after();
      float v[64];
      tmem_ld_32x32(R + (uint32_t)part * 64u, *reinterpret_cast<float(*)[32]>(&v[0]));
      tmem_ld_32x32(R + (uint32_t)part * 64u + 32u, *reinterpret_cast<float(*)[32]>(&v[32]));
      tmem_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sp_free[grp]);
      if (p.out_ln) {
        // one exchange per row: each part sends the mean of its columns and their squared deviations from it; the two
        // pairs combine exactly.  (The slots are rewritten a tile later, when every warp of the group has moved on.)
        float2* w = reinterpret_cast<float2*>(v);
        float2 s0 = w[0], s1 = w[1];
#pragma unroll
        for (int j = 2; j < 32; j += 2) { s0 = __fadd2_rn(s0, w[j]); s1 = __fadd2_rn(s1, w[j + 1]); }
        s0 = __fadd2_rn(s0, s1);
        const float m_part = (s0.x + s0.y) * (1.0f / 64);
        float2 q0 = make_float2(0.f, 0.f), q1 = q0;
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
          const float2 d0 = __fadd2_rn(w[j], make_float2(-m_part, -m_part)), d1 = __fadd2_rn(w[j + 1], make_float2(-m_part, -m_part));
          q0 = __ffma2_rn(d0, d0, q0);
          q1 = __ffma2_rn(d1, d1, q1);
        }
        q0 = __fadd2_rn(q0, q1);
        const float m2 = q0.x + q0.y;
        exch[part * 128 + r] = make_float2(m_part, m2);
        __syncwarp();
        if (lane == 0) mbar_arrive(&pair_bar[grp * 4 + q4]);
        if (!mbar_wait(&pair_bar[grp * 4 + q4], i_ph, p.err, 37)) { ok = false; break; }
        const float2 other = exch[(part ^ 1) * 128 + r];
        const float mu = 0.5f * (m_part + other.x);
        const float dm = m_part - mu;
        const float rstd = rsqrtf((m2 + other.y + 128.0f * dm * dm) * (1.0f / HT_D) + p.ln_eps);
#pragma unroll
        for (int j = 0; j < 32; ++j) w[j] = __fmul2_rn(__fadd2_rn(w[j], make_float2(-mu, -mu)), make_float2(rstd, rstd));
      }
      // Out through the warp's own patch, eight rows of its 64 columns at a time (128 bytes a row, 16-byte chunk c at position
      // c ^ row: no bank conflicts), so that a store writes whole 128-byte lines: with 32- or 64-byte pieces of rows the
      // stores of a tile took 2000 cycles of the row warps' chain.
      const uint32_t wr = (uint32_t)(lane & 7) * 128u, x7 = (uint32_t)(lane & 7);
      const int rsub = lane >> 3;
      const uint8_t* rd = patch + rsub * 128;
      __nv_bfloat16* dst = p.out + part * 64 + (lane & 7) * 8;
      float4 o[8];
#pragma unroll
      for (int c = 0; c < 8; ++c)
        o[c] = make_float4(ht_pack(v[c * 8], v[c * 8 + 1]), ht_pack(v[c * 8 + 2], v[c * 8 + 3]), ht_pack(v[c * 8 + 4], v[c * 8 + 5]),
                           ht_pack(v[c * 8 + 6], v[c * 8 + 7]));
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        if (rsub == m) {
#pragma unroll
          for (int c = 0; c < 8; ++c) *reinterpret_cast<float4*>(patch + wr + (((uint32_t)c ^ x7) << 4)) = o[c];
        }
        __syncwarp();
        const float4 o0 = *reinterpret_cast<const float4*>(rd + ((x7 ^ (uint32_t)rsub) << 4));
        const float4 o1 = *reinterpret_cast<const float4*>(rd + 512 + ((x7 ^ (uint32_t)(rsub + 4)) << 4));
        __syncwarp();
        const int row = row0 + q4 * 32 + m * 8 + rsub;
        if (row < row_end) *reinterpret_cast<float4*>(dst + (int64_t)row * HT_D) = o0;
        if (row + 4 < row_end) *reinterpret_cast<float4*>(dst + (int64_t)(row + 4) * HT_D) = o1;
      }
      i_ph ^= 1u;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
  if (p.beside.early) pdl_wait();                             // whoever waits for this kernel waits for the link side too
}

template <int NG, int ELL, bool LN>
static lime_status launch_ht(const HistUpdateArgs& a, cudaStream_t st) {
  CUtensorMap tmX, tmK2, tmG, tmU, tmWo;
  const uint64_t users = a.shared ? 1 : (uint64_t)a.B, HL = NG * 128;
  if (!make_tmap_bf16_sw128(&tmX, a.hist_in, (uint64_t)a.total, HT_D, HT_D, HT_TILE) ||
      !make_tmap_bf16_sw128(&tmK2, a.K2, users * HL, HT_D, HT_D, 128) ||
      !make_tmap_bf16_sw128(&tmG, a.G2t, users * HT_F, HL, HL, 64) || !make_tmap_bf16_sw128(&tmU, a.U2t, users * HT_F, HL, HL, 64) ||
      !make_tmap_bf16_sw128(&tmWo, a.WoT, HT_D, HT_F, HT_F, 128))
    return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
  HistUpdateTmemParams p;
  p.out = (__nv_bfloat16*)a.hist_out; p.off = a.off; p.tile_start = a.tile_start; p.B = a.B; p.silu = a.silu;
  p.cK = a.cK; p.stats_in = a.stats_in; p.shared = a.shared; p.out_ln = a.out_ln; p.ln_eps = a.ln_eps; p.beside = a.beside; p.err = a.err;
  const int grid = a.n_tile_upper < kSMs ? a.n_tile_upper : kSMs;
  if (grid < 1) return LIME_OK;
  static bool smem_set[kMaxDeviceOrdinals] = {};
  const lime_status es = ensure_dynamic_smem((const void*)k_hist_update_tmem_tc<NG, ELL, LN>, (int)HT_SMEM, smem_set);
  if (es != LIME_OK) return es;
  ProfScope _p("k_hist_update_tmem_tc", st);
  launch_pdl(k_hist_update_tmem_tc<NG, ELL, LN>, dim3(grid), dim3(HT_THREADS), HT_SMEM, st, tmX, tmK2, tmG, tmU, tmWo, p);
  LIME_LAUNCH_CHECK("k_hist_update_tmem_tc");
  return LIME_OK;
}

bool hist_update_tmem_supported(int dtype, int d, int f, int H, int ell, int phi, int gated_mlp) {
  const int HL = H * ell;
  return dtype == LIME_BF16 && d == HT_D && f == HT_F && ((HL == 128 && (ell == 16 || ell == 32)) || (HL == 256 && (ell == 32 || ell == 64))) &&
         (phi == LIME_PHI_SOFTMAX || phi == LIME_PHI_SILU) && gated_mlp != 0;
}

template <int NG, int ELL>
static lime_status launch_ht_ln(const HistUpdateArgs& a, cudaStream_t st) {
  return a.ln ? launch_ht<NG, ELL, true>(a, st) : launch_ht<NG, ELL, false>(a, st);
}

lime_status launch_hist_update_tmem(const HistUpdateArgs& a, int H, cudaStream_t st) {
  if (a.total == 0) return LIME_OK;
  if (a.ln && (a.stats_in == nullptr || a.cK == nullptr)) return LIME_INVALID_ARG;
  if (H * a.ell == 128) return a.ell == 16 ? launch_ht_ln<1, 16>(a, st) : launch_ht_ln<1, 32>(a, st);
  return a.ell == 32 ? launch_ht_ln<2, 32>(a, st) : launch_ht_ln<2, 64>(a, st);
}

}  // namespace lime
