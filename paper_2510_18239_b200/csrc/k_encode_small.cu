// The whole user-side encode of a narrow model in one launch (bf16 storage, d = d_ff = 32): all XOR layers of a user in one
// block, the history resident in shared memory from the first layer to the last (Eq. 7, Eq. 5, Eq. 8).
//
// At d = 32 a history row is 64 bytes and a layer about 24 k operations per token: a batch of short histories is a few
// hundred million operations and under a megabyte, so what bounds it is latency - launches, dependent reads and the passes
// of materialised Q / K / V / U rows - and not a pipe.  As in the wider tensor-core kernels the history-side projections are
// folded into the link side, but a tile is 16 tokens of one warp and the contractions chain through registers
// (mma.m16n8k16: the accumulator of one is the A operand of the next): at these widths a 128-row tcgen05 tile would be
// mostly padding and its hand-overs longer than the work.  Per layer, with HL = H * ell:
//   PREP   Q2 = (LN(T) W_Q,h) W_K,h^T * scale, K2 likewise, G2 = (LN(T) W_V,h) W_g[h rows], U2 likewise     warp = operand x half the heads
//   links  S = Q2 . X^T, online softmax (or SiLU), acc += P . X    warp = 16 stacked rows x a share of the tokens; shares merged
//   MLP    O = Ohat W_V, T = (SiLU(O W_g) * (O W_u)) W_o, L^P += T  four warps, L^P stays in registers
//   rows   P = softmax_h(X . K2^T), U = SiLU(P G2) * (P U2), X <- LN(U W_o)   the other warps at once, then all; 16 rows at a time
// The link rows are few and everything depends on them, so their activations enter each product as a bf16 value and its
// bf16 remainder (two products, fp32-level accuracy; the weights are exact as they are stored).  Rounded once instead, they
// alone would double the error of the link states (1.1 against 0.5 % of their norm).  Two more splits hold the error at that of the
// generic kernels, which keep link rows, probabilities and the first layer's LayerNorm in fp32 and round the history's K, V, Q, O, U:
// with SiLU, whose probabilities are not normalised, Q2, K2 and the probabilities; with rows that arrive raw, the normalised rows of
// the first layer.  Error of the link states against fp64, four heads of 16 links, three layers, 64 users of 10..256 tokens, rms over
// them (generic kernels; rounded once): softmax 0.91 % (1.14), SiLU 1.4 (1.9; 2.1), raw rows softmax 0.55 (0.66; 0.91), raw rows SiLU
// 0.91 (1.4; 2.1).
// A layer's six weights (12 KB) come in by cp.async a layer ahead.  Histories beyond the shared-memory capacity stay in
// global memory (`scratch`), 16 rows of it at a time in a patch per warp; the longest of a batch take a cluster of blocks each.
// Rows of 64 bytes sit at pitch 64 with 16-byte chunk c at c ^ ((row >> 1) & 3): 16-byte reads of whole rows and ldmatrix
// reads of one chunk of eight rows are both free of bank conflicts.  Where both operands are read as whole rows the
// contraction over the 32 features is permuted so that thread t of a quad holds features 8 t .. 8 t + 7 (one 16-byte read
// gives the fragments of both k-steps).
#include "lime_common.cuh"
#include "tc_common.cuh"

namespace lime {

constexpr int ES_D = 32, ES_WARPS = 8, ES_THREADS = ES_WARPS * 32;
constexpr int ES_CAP = 1024;     // history rows a block keeps in shared memory
// Histories over 2048 tokens are shared out over a cluster of eight blocks, in a launch of their own, at most fifteen of them (the
// clusters that run at once; the line doubles until that holds).  One user of n tokens among 99 of 100, three layers, one block /
// a cluster / the generic kernels, which split by token: n = 2000 183 / 84 / 776 us, 8000 701 / 127 / 925, 32000 2776 / 401 / 1592,
// 150000 12971 / 1619 / 3860.  With 32 users of 2000 a block each is the better (184 against 214 us): what a layer's exchange
// costs a cluster (about 14 us) wants a long history.
constexpr int ES_LONG = 2048, ES_CLUSTER = 8, ES_CLUSTERS = 15;

template <int H_, int ELL_>
struct EsCfg {
  static constexpr int H = H_, ELL = ELL_, HL = H * ELL;
  static constexpr int LMT = (ELL + 15) / 16;                  // 16-row tiles of link rows
  static constexpr int MT = HL / 16;                           // 16-row tiles of stacked rows
  static constexpr int TG = ES_WARPS / MT;                     // shares of the tokens in the links <- history direction
  static constexpr int DH = ES_D / H;
  static constexpr int PART_LD = 36;                           // floats per partial accumulator row
  static constexpr int OFF_W = 0;                              // two layers' weights: W_Q, W_K, W_V, W_g, W_u, W_o
  static constexpr int OFF_OPS = OFF_W + 2 * 6 * 2048;         // Q2, K2, G2, U2 [HL x 32]
  static constexpr int OFF_PART = OFF_OPS + 4 * HL * 64;       // partial accumulators, maxima, sums
  static constexpr int OFF_PM = OFF_PART + TG * HL * PART_LD * 4;
  static constexpr int OFF_PS = OFF_PM + TG * HL * 4;
  static constexpr int LROWS = LMT * 16;                       // link rows, padded; all of the following as value | remainder
  static constexpr int OFF_OHAT = OFF_PS + TG * HL * 4;        // [link rows x H d]
  static constexpr int OFF_THAT = OFF_OHAT + 2 * LROWS * H * 64;
  static constexpr int OFF_O = OFF_THAT + 2 * LROWS * 64;
  static constexpr int OFF_U = OFF_O + 2 * LROWS * 64;
  static constexpr int OFF_LO = OFF_U + 2 * LROWS * 64;        // SiLU: remainders of Q2, K2
  static constexpr int OFF_NEXT = OFF_LO + 2 * HL * 64;        // tile counter
  static constexpr int OFF_PATCH = OFF_NEXT + 16;              // [warps][16 x 64 bytes], the same for the remainders of raw rows
  static constexpr int OFF_X = OFF_PATCH + 2 * ES_WARPS * 1024;
  static_assert(HL % 16 == 0 && MT <= ES_WARPS && ES_WARPS % MT == 0, "split of the stacked rows over the warps");
};

struct EncodeSmallParams {
  const __nv_bfloat16* hist; const int32_t* off;
  const float* links; int links_per_user;                      // [ell x d] fp32, or [B x ell x d]
  const __nv_bfloat16* w[LIME_MAX_LAYERS][6];                   // W_Q, W_K, W_V (NULL: identity), W_g, W_u, W_o, as stored
  __nv_bfloat16* scratch;                                       // [total x d]
  __nv_bfloat16* link_states; float* lp;                        // exactly one is wanted
  int B, clustered, skip_long;                                  // clustered: cluster k takes the k-th long user, else block b user b
  int n_layers, cap, ln;                                        // cap: history rows shared memory holds
  float eps, scale;                                             // scale of the scores (times log2 e with the softmax)
};

__device__ __forceinline__ uint32_t es_sw(int row, int chunk) { return (uint32_t)row * 64u + ((uint32_t)(chunk ^ ((row >> 1) & 3)) << 4); }
// x * sigmoid(x) with a fast quotient (relative error 1e-6)
__device__ __forceinline__ float es_silu(float x) { return __fdividef(x, 1.0f + __expf(-x)); }
__device__ __forceinline__ uint32_t es_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t es_pack(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float es_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float es_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }
__device__ __forceinline__ float es_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void es_mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void es_mma8(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(b0));
}
// a pair of fp32 values as packed bf16 values and packed bf16 remainders
__device__ __forceinline__ void es_split(float x, float y, uint32_t& hi, uint32_t& lo) {
  hi = es_pack(x, y);
  lo = es_pack(x - es_lo(hi), y - es_hi(hi));
}
// the remainders alone
__device__ __forceinline__ uint32_t es_rest(float x, float y, uint32_t hi) { return es_pack(x - es_lo(hi), y - es_hi(hi)); }
// both k-steps of a 32-feature contraction in the permuted order: rows g and g + 8 of A, one row of B
__device__ __forceinline__ void es_mma32(float (&c)[4], const uint4& a, const uint4& a8, const uint4& b) {
  es_mma(c, a.x, a8.x, a.y, a8.y, b.x, b.y);
  es_mma(c, a.z, a8.z, a.w, a8.w, b.z, b.w);
}
__device__ __forceinline__ void es_ldsm(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void es_ldsm_t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void es_cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(es_addr(dst)), "l"(src) : "memory");
}
// A fragments of 16 rows x 16 columns (chunks c, c + 1) of a swizzled [rows x 32] operand
__device__ __forceinline__ void es_lda(uint32_t (&a)[4], const uint8_t* base, int row0, int chunk, int lane) {
  es_ldsm(a, es_addr(base + es_sw(row0 + (lane & 15), chunk + (lane >> 4))));
}
// B fragments of both k-steps (32 rows of W, columns of one chunk) of a [32 x 32] weight as stored
__device__ __forceinline__ void es_ldb(uint32_t (&w)[4], const uint8_t* W, int chunk, int lane) {
  es_ldsm_t(w, es_addr(W + es_sw(lane, chunk)));
}
__device__ __forceinline__ float es_quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}
__device__ __forceinline__ float es_quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ uint4 es_lds(const uint8_t* p) { return *reinterpret_cast<const uint4*>(p); }

// LayerNorm of the 32 columns a quad holds of one row: c[n][i], c[n][i + 1] for n = 0..3
__device__ __forceinline__ void es_ln(float (&c)[4][4], int i, float eps) {
  float s = 0.f;
#pragma unroll
  for (int n = 0; n < 4; ++n) s += c[n][i] + c[n][i + 1];
  const float mu = es_quad_sum(s) * (1.0f / ES_D);
  float v = 0.f;
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    c[n][i] -= mu; c[n][i + 1] -= mu;
    v = fmaf(c[n][i], c[n][i], v); v = fmaf(c[n][i + 1], c[n][i + 1], v);
  }
  const float rstd = rsqrtf(es_quad_sum(v) * (1.0f / ES_D) + eps);
#pragma unroll
  for (int n = 0; n < 4; ++n) { c[n][i] *= rstd; c[n][i + 1] *= rstd; }
}

// all blocks of the cluster, or the one block of a user that has no cluster
__device__ __forceinline__ void es_sync(bool clustered) {
  if (clustered) cluster_sync_all();
  else __syncthreads();
}

// RAW: the rows arrive without their LayerNorm, and the first layer takes the normalised ones as value and remainder
template <class G, bool SILU, bool RAW>
__global__ void __launch_bounds__(ES_THREADS)
k_encode_small(const EncodeSmallParams p) {
  constexpr int H = G::H, ELL = G::ELL, HL = G::HL, LMT = G::LMT, MT = G::MT, TG = G::TG;
  extern __shared__ __align__(128) uint8_t sm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  uint8_t* const X = sm + G::OFF_X;
  uint8_t* const patch = sm + G::OFF_PATCH + warp * 1024;
  int* const next_tile = reinterpret_cast<int*>(sm + G::OFF_NEXT);
  pdl_launch_dependents();
  pdl_wait();
  // a long user belongs to a cluster of blocks, each with a share of the history; the link rows are done by every block of it, from
  // the shares' accumulators
  const bool clustered = p.clustered != 0;
  const int rank = clustered ? (int)blockIdx.x % ES_CLUSTER : 0, CL = clustered ? ES_CLUSTER : 1;
  const int b = clustered ? nth_long_user(p.off, p.B, ES_LONG, ES_CLUSTERS, (int)blockIdx.x / ES_CLUSTER, next_tile) : (int)blockIdx.x;
  if (b < 0) return;
  const int user0 = p.off[b], user_n = p.off[b + 1] - user0;
  if (p.skip_long && user_n > ES_LONG && user_n > long_user_line(p.off, p.B, ES_LONG, ES_CLUSTERS, next_tile)) return;
  const int share = ((user_n + CL - 1) / CL + 15) & ~15, first = min(user_n, rank * share);
  const int tok0 = user0 + first, n = min(user_n, first + share) - first;
  const bool resident = n <= p.cap;
  const int n_tiles = (n + 15) >> 4;

  auto load_weights = [&](int j) {
    uint8_t* dst = sm + G::OFF_W + (j & 1) * (6 * 2048);
    for (int i = tid; i < 6 * 128; i += ES_THREADS) {
      const int m = i >> 7, row = (i >> 2) & 31, c = i & 3;
      uint8_t* at = dst + m * 2048 + es_sw(row, c);
      const uint8_t* src = reinterpret_cast<const uint8_t*>(p.w[j][m]);
      if (src != nullptr) es_cp16(at, src + (i & 127) * 16);
      else {                                                    // identity
        uint32_t u[4] = {0, 0, 0, 0};
        if ((row >> 3) == c) u[(row & 7) >> 1] = (row & 1) ? 0x3f800000u : 0x00003f80u;
        *reinterpret_cast<uint4*>(at) = make_uint4(u[0], u[1], u[2], u[3]);
      }
    }
  };
  load_weights(0);

  // LayerNorm of a row that a quad holds eight features each of: packed values, and their remainders
  auto ln_row = [&](const uint4& v, uint4& hi, uint4& lo) {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
    float s = 0.f, q = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) s += es_lo(u[k]) + es_hi(u[k]);
    const float mu = es_quad_sum(s) * (1.0f / ES_D);
#pragma unroll
    for (int k = 0; k < 4; ++k) { const float x = es_lo(u[k]) - mu, y = es_hi(u[k]) - mu; q = fmaf(x, x, q); q = fmaf(y, y, q); }
    const float rstd = rsqrtf(es_quad_sum(q) * (1.0f / ES_D) + p.eps);
    uint32_t h[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) es_split((es_lo(u[k]) - mu) * rstd, (es_hi(u[k]) - mu) * rstd, h[k], l[k]);
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
  };
  // history rows -> shared memory, or to scratch where they are too many (raw ones stay where they are until the first update)
  uint8_t* const XL = X + ((p.cap + 15) & ~15) * 64;            // remainders of raw rows
  if (!RAW || resident) {
    __nv_bfloat16* const big = p.scratch + (int64_t)tok0 * ES_D;
    for (int i = tid; i < n_tiles * 64; i += ES_THREADS) {
      const int row = i >> 2, c = i & 3;
      uint4 v = make_uint4(0, 0, 0, 0), rest = v;
      if (row < n) v = __ldg(reinterpret_cast<const uint4*>(p.hist + (int64_t)(tok0 + row) * ES_D) + c);
      if constexpr (RAW) {
        ln_row(v, v, rest);
        if (row >= n) v = rest = make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(XL + es_sw(row, c)) = rest;
      }
      if (resident) *reinterpret_cast<uint4*>(X + es_sw(row, c)) = v;
      else if (row < n) *(reinterpret_cast<uint4*>(big + (int64_t)row * ES_D) + c) = v;
    }
  }
  // LN(T^0) -> That; the padding rows of an 8-row link tile stay zero
  for (int i = tid; i < 2 * G::LROWS * (H + 1) * 4; i += ES_THREADS) *reinterpret_cast<uint4*>(sm + G::OFF_OHAT + i * 16) = make_uint4(0, 0, 0, 0);
  __syncthreads();
  {
    const float* T0 = p.links + (p.links_per_user ? (int64_t)b * ELL * ES_D : 0);
    for (int l = warp; l < ELL; l += ES_WARPS) {
      float x = T0[l * ES_D + lane];
      if (p.ln) {
        x -= warp_sum(x) * (1.0f / ES_D);
        x *= rsqrtf(warp_sum(x * x) * (1.0f / ES_D) + p.eps);
      }
      const __nv_bfloat16 hi = __float2bfloat16_rn(x);
      uint8_t* dst = sm + G::OFF_THAT + es_sw(l, lane >> 3) + (lane & 7) * 2;
      *reinterpret_cast<__nv_bfloat16*>(dst) = hi;
      *reinterpret_cast<__nv_bfloat16*>(dst + G::LROWS * 64) = __float2bfloat16_rn(x - __bfloat162float(hi));
    }
  }
  // 16 rows of the history as a swizzled tile in shared memory; of raw rows (`first`) the remainders lie at rest(tile)
  auto tile = [&](int r0, bool first) -> uint8_t* {
    if (resident) return X + r0 * 64;
    const __nv_bfloat16* src = (first ? p.hist : p.scratch) + (int64_t)(tok0 + r0) * ES_D;
    __syncwarp();
    if (first) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {                             // four lanes a row
        const int row = k * 8 + g;
        uint4 v = make_uint4(0, 0, 0, 0), rest;
        if (r0 + row < n) v = __ldg(reinterpret_cast<const uint4*>(src + row * ES_D) + t);
        ln_row(v, v, rest);
        if (r0 + row >= n) v = rest = make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(patch + es_sw(row, t)) = v;
        *reinterpret_cast<uint4*>(patch + ES_WARPS * 1024 + es_sw(row, t)) = rest;
      }
    } else {
      const int row = lane >> 1;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int c = (lane & 1) * 2 + k;
        const uint4 v = r0 + row < n ? *(reinterpret_cast<const uint4*>(src + row * ES_D) + c) : make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(patch + es_sw(row, c)) = v;
      }
    }
    __syncwarp();
    return patch;
  };
  auto rest = [&](uint8_t* xt) { return resident ? XL + (xt - X) : xt + ES_WARPS * 1024; };

  float lp[4][4];                                              // running sum of T (warps 0 .. LMT - 1)
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) lp[i][e] = 0.f;

  for (int j = 0; j < p.n_layers; ++j) {
    const bool last = j + 1 == p.n_layers, raw = RAW && j == 0;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const uint8_t* W = sm + G::OFF_W + (j & 1) * (6 * 2048);
    if (!last) load_weights(j + 1);
    // ---- PREP: folded operands of this layer.  Warp = operand (Q2, K2, G2, U2) x half of the heads = 16 of the 32 columns
    // of the first product, whose accumulators are the A fragments of the second
    if (!last || (warp & 3) == 0) {
      const int op = warp & 3, half = warp >> 2;
      const uint8_t* W1 = W + (op < 2 ? op : 2) * 2048;
      const uint8_t* W2 = W + (op == 0 ? 1 : op == 1 ? 0 : op + 1) * 2048;
      const float sc = op < 2 ? p.scale : 1.0f;
#pragma unroll
      for (int m = 0; m < LMT; ++m) {
        float c[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) c[i][e] = 0.f;
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          uint32_t bw[4], a[4], al[4];
          es_ldsm_t(bw, es_addr(W1 + es_sw(ks * 16 + (lane & 15), half * 2 + (lane >> 4))));
          es_lda(a, sm + G::OFF_THAT, m * 16, ks * 2, lane);
          es_lda(al, sm + G::OFF_THAT + G::LROWS * 64, m * 16, ks * 2, lane);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            es_mma(c[i], a[0], a[1], a[2], a[3], bw[2 * i], bw[2 * i + 1]);
            es_mma(c[i], al[0], al[1], al[2], al[3], bw[2 * i], bw[2 * i + 1]);
          }
        }
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int i = 0; i < 2; ++i) { es_split(c[i][0], c[i][1], hi[2 * i], lo[2 * i]); es_split(c[i][2], c[i][3], hi[2 * i + 1], lo[2 * i + 1]); }
#pragma unroll
        for (int hh = 0; hh < H / 2; ++hh) {
          const int h = half * (H / 2) + hh;
          float d[4][4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) d[i][e] = 0.f;
          uint32_t w[4];
          if constexpr (G::DH == 8) {
            if (op < 2) es_ldsm(w, es_addr(W2 + es_sw(lane, h)));                                      // rows n, columns of head h
            else es_ldsm_t(w, es_addr(W2 + es_sw(h * 8 + (lane & 7), lane >> 3)));                    // rows of head h, columns n
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              es_mma8(d[i], hi[2 * hh], hi[2 * hh + 1], w[i]);
              es_mma8(d[i], lo[2 * hh], lo[2 * hh + 1], w[i]);
            }
          } else {
#pragma unroll
            for (int i = 0; i < 4; i += 2) {
              if (op < 2) es_ldsm(w, es_addr(W2 + es_sw((i + (lane >> 4)) * 8 + (lane & 7), h * 2 + ((lane >> 3) & 1))));
              else es_ldsm_t(w, es_addr(W2 + es_sw(h * 16 + (lane & 15), i + (lane >> 4))));
#pragma unroll
              for (int q = 0; q < 2; ++q) {
                es_mma(d[i + q], hi[0], hi[1], hi[2], hi[3], w[2 * q], w[2 * q + 1]);
                es_mma(d[i + q], lo[0], lo[1], lo[2], lo[3], w[2 * q], w[2 * q + 1]);
              }
            }
          }
          const int r = h * ELL + m * 16 + g;
          auto store = [&](uint8_t* dst) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              *reinterpret_cast<uint32_t*>(dst + es_sw(r, i) + t * 4) = es_pack(d[i][0], d[i][1]);
              if (ELL > 8) *reinterpret_cast<uint32_t*>(dst + es_sw(r + 8, i) + t * 4) = es_pack(d[i][2], d[i][3]);
            }
          };
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) d[i][e] *= sc;
          store(sm + G::OFF_OPS + op * (HL * 64));
          if (SILU && op < 2) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int e = 0; e < 4; ++e) d[i][e] -= __bfloat162float(__float2bfloat16_rn(d[i][e]));
            store(sm + G::OFF_LO + op * (HL * 64));
          }
        }
      }
    }
    if (tid == 0) *next_tile = 0;
    __syncthreads();
    // ---- links <- history: warp = 16 stacked rows x the tiles tg, tg + TG, ..
    {
      const int m = warp % MT, tg = warp / MT;
      const uint4 qa = es_lds(sm + G::OFF_OPS + es_sw(m * 16 + g, t)), qa8 = es_lds(sm + G::OFF_OPS + es_sw(m * 16 + g + 8, t));
      uint4 ql = make_uint4(0, 0, 0, 0), ql8 = ql;
      if (SILU) { ql = es_lds(sm + G::OFF_LO + es_sw(m * 16 + g, t)); ql8 = es_lds(sm + G::OFF_LO + es_sw(m * 16 + g + 8, t)); }
      float o[4][4], mx0 = -INFINITY, mx1 = -INFINITY, l0 = 0.f, l1 = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[i][e] = 0.f;
      for (int tt = tg; tt < n_tiles; tt += TG) {
        uint8_t* const xt = tile(tt * 16, raw);
        float s[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
#pragma unroll
          for (int e = 0; e < 4; ++e) s[i][e] = 0.f;
          es_mma32(s[i], qa, qa8, es_lds(xt + es_sw(i * 8 + g, t)));
          if (SILU) es_mma32(s[i], ql, ql8, es_lds(xt + es_sw(i * 8 + g, t)));
          if (raw) es_mma32(s[i], qa, qa8, es_lds(rest(xt) + es_sw(i * 8 + g, t)));
        }
        const int left = n - tt * 16;                          // valid tokens of the tile
        if (SILU) {
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[i][e] = es_silu(s[i][e]);       // padding rows are zero and SiLU(0) = 0
        } else {
          if (left < 16) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (i * 8 + 2 * t + (e & 1) >= left) s[i][e] = -INFINITY;
          }
          const float n0 = fmaxf(mx0, es_quad_max(fmaxf(fmaxf(s[0][0], s[0][1]), fmaxf(s[1][0], s[1][1]))));
          const float n1 = fmaxf(mx1, es_quad_max(fmaxf(fmaxf(s[0][2], s[0][3]), fmaxf(s[1][2], s[1][3]))));
          const float f0 = es_ex2(mx0 - n0), f1 = es_ex2(mx1 - n1);
          mx0 = n0; mx1 = n1;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            s[i][0] = es_ex2(s[i][0] - n0); s[i][1] = es_ex2(s[i][1] - n0);
            s[i][2] = es_ex2(s[i][2] - n1); s[i][3] = es_ex2(s[i][3] - n1);
          }
          l0 = fmaf(l0, f0, s[0][0] + s[0][1] + s[1][0] + s[1][1]);
          l1 = fmaf(l1, f1, s[0][2] + s[0][3] + s[1][2] + s[1][3]);
#pragma unroll
          for (int i = 0; i < 4; ++i) { o[i][0] *= f0; o[i][1] *= f0; o[i][2] *= f1; o[i][3] *= f1; }
        }
        const uint32_t a0 = es_pack(s[0][0], s[0][1]), a1 = es_pack(s[0][2], s[0][3]), a2 = es_pack(s[1][0], s[1][1]), a3 = es_pack(s[1][2], s[1][3]);
#pragma unroll
        for (int c0 = 0; c0 < 4; c0 += 2) {
          uint32_t r[4];
          es_ldsm_t(r, es_addr(xt + es_sw((lane & 15), c0 + (lane >> 4))));
          es_mma(o[c0], a0, a1, a2, a3, r[0], r[1]);
          es_mma(o[c0 + 1], a0, a1, a2, a3, r[2], r[3]);
          if (SILU) {
            const uint32_t l0 = es_rest(s[0][0], s[0][1], a0), l1 = es_rest(s[0][2], s[0][3], a1), l2 = es_rest(s[1][0], s[1][1], a2), l3 = es_rest(s[1][2], s[1][3], a3);
            es_mma(o[c0], l0, l1, l2, l3, r[0], r[1]);
            es_mma(o[c0 + 1], l0, l1, l2, l3, r[2], r[3]);
          }
          if (raw) {
            es_ldsm_t(r, es_addr(rest(xt) + es_sw((lane & 15), c0 + (lane >> 4))));
            es_mma(o[c0], a0, a1, a2, a3, r[0], r[1]);
            es_mma(o[c0 + 1], a0, a1, a2, a3, r[2], r[3]);
          }
        }
      }
      float* part = reinterpret_cast<float*>(sm + G::OFF_PART) + (tg * HL + m * 16 + g) * G::PART_LD + 2 * t;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        *reinterpret_cast<float2*>(part + i * 8) = make_float2(o[i][0], o[i][1]);
        *reinterpret_cast<float2*>(part + 8 * G::PART_LD + i * 8) = make_float2(o[i][2], o[i][3]);
      }
      l0 = es_quad_sum(l0); l1 = es_quad_sum(l1);
      if (t == 0) {
        float* pm = reinterpret_cast<float*>(sm + G::OFF_PM) + tg * HL + m * 16 + g;
        float* ps = reinterpret_cast<float*>(sm + G::OFF_PS) + tg * HL + m * 16 + g;
        pm[0] = mx0; pm[8] = mx1; ps[0] = l0; ps[8] = l1;
      }
    }
    es_sync(clustered);
    // ---- merge the shares, normalise: Ohat[l, h * 32 + i]
    for (int i = tid; i < HL * 4; i += ES_THREADS) {
      const int r = i >> 2, c = i & 3, h = r / ELL, l = r % ELL;
      float M = -INFINITY, S = 0.f, acc[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) acc[k] = 0.f;
      auto highest = [&](const uint8_t* at) {
        const float* pm = reinterpret_cast<const float*>(at + G::OFF_PM) + r;
#pragma unroll
        for (int s = 0; s < TG; ++s) M = fmaxf(M, pm[s * HL]);
      };
      auto add = [&](const uint8_t* at) {
        const float* pm = reinterpret_cast<const float*>(at + G::OFF_PM) + r;
        const float* ps = reinterpret_cast<const float*>(at + G::OFF_PS) + r;
#pragma unroll
        for (int s = 0; s < TG; ++s) {
          const float w = SILU ? 1.f : (M == -INFINITY ? 0.f : es_ex2(pm[s * HL] - M));
          S = fmaf(w, ps[s * HL], S);
          const float4* src = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(at + G::OFF_PART) + (s * HL + r) * G::PART_LD + c * 8);
          const float4 x = src[0], y = src[1];
          acc[0] = fmaf(w, x.x, acc[0]); acc[1] = fmaf(w, x.y, acc[1]); acc[2] = fmaf(w, x.z, acc[2]); acc[3] = fmaf(w, x.w, acc[3]);
          acc[4] = fmaf(w, y.x, acc[4]); acc[5] = fmaf(w, y.y, acc[5]); acc[6] = fmaf(w, y.z, acc[6]); acc[7] = fmaf(w, y.w, acc[7]);
        }
      };
      if (!clustered) {
        highest(sm);
        add(sm);
      } else {
#pragma unroll
        for (int q = 0; q < ES_CLUSTER; ++q) highest(cluster_peer(static_cast<const uint8_t*>(sm), q));
#pragma unroll 4
        for (int q = 0; q < ES_CLUSTER; ++q) add(cluster_peer(static_cast<const uint8_t*>(sm), q));
      }
      const float inv = user_n > 0 ? 1.0f / (SILU ? (float)user_n : S) : 0.f;
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) es_split(acc[2 * k] * inv, acc[2 * k + 1] * inv, hi[k], lo[k]);
      uint8_t* dst = sm + G::OFF_OHAT + l * (H * 64) + (((h * 4 + c) ^ (l & 7)) << 4);
      *reinterpret_cast<uint4*>(dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *reinterpret_cast<uint4*>(dst + G::LROWS * H * 64) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
    es_sync(clustered);                                         // (of a cluster: the peers have read this block's accumulators)
    // ---- GatedMLP on the link rows: warps 0..3 take eight columns each of O and of the hidden layer, warps 0 .. LMT - 1 the
    // rows of T
    if (warp < 4) {
      auto store_split = [&](int off, int m, const float (&c)[4]) {
        uint32_t hi, lo;
        uint8_t* dst = sm + off + es_sw(m * 16 + g, warp) + t * 4;
        es_split(c[0], c[1], hi, lo);
        *reinterpret_cast<uint32_t*>(dst) = hi; *reinterpret_cast<uint32_t*>(dst + G::LROWS * 64) = lo;
        es_split(c[2], c[3], hi, lo);
        *reinterpret_cast<uint32_t*>(dst + 8 * 64) = hi; *reinterpret_cast<uint32_t*>(dst + (G::LROWS + 8) * 64) = lo;
      };
      // c += rows m of the split operand at `off` . the two k-steps w
      auto product = [&](float (&c)[4], int off, int m, const uint32_t (&w)[4]) {
#pragma unroll
        for (int ks = 0; ks < 2; ++ks)
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            uint32_t a[4];
            es_lda(a, sm + off + s * G::LROWS * 64, m * 16, ks * 2, lane);
            es_mma(c, a[0], a[1], a[2], a[3], w[2 * ks], w[2 * ks + 1]);
          }
      };
      uint32_t wa[4], wb[4];
      es_ldb(wa, W + 2 * 2048, warp, lane);
      const int h = warp * 8 / G::DH;
#pragma unroll
      for (int m = 0; m < LMT; ++m) {
        float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int ks = 0; ks < 2; ++ks)
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            uint32_t a[4];
            const int row = m * 16 + (lane & 15);
            es_ldsm(a, es_addr(sm + G::OFF_OHAT + s * G::LROWS * H * 64 + row * (H * 64) + (((h * 4 + ks * 2 + (lane >> 4)) ^ (row & 7)) << 4)));
            es_mma(c, a[0], a[1], a[2], a[3], wa[2 * ks], wa[2 * ks + 1]);
          }
        store_split(G::OFF_O, m, c);
      }
      es_ldb(wa, W + 3 * 2048, warp, lane);
      es_ldb(wb, W + 4 * 2048, warp, lane);
      asm volatile("bar.sync 1, 128;" ::: "memory");
#pragma unroll
      for (int m = 0; m < LMT; ++m) {
        float gt[4] = {0.f, 0.f, 0.f, 0.f}, up[4] = {0.f, 0.f, 0.f, 0.f};
        product(gt, G::OFF_O, m, wa);
        product(up, G::OFF_O, m, wb);
#pragma unroll
        for (int e = 0; e < 4; ++e) gt[e] = es_silu(gt[e]) * up[e];
        store_split(G::OFF_U, m, gt);
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (warp < LMT) {
        float c[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          es_ldb(wa, W + 5 * 2048, i, lane);
#pragma unroll
          for (int e = 0; e < 4; ++e) c[i][e] = 0.f;
          product(c[i], G::OFF_U, warp, wa);
#pragma unroll
          for (int e = 0; e < 4; ++e) lp[i][e] += c[i][e];
        }
        if (!last) {
          if (p.ln) { es_ln(c, 0, p.eps); es_ln(c, 2, p.eps); }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int l = warp * 16 + g;
            uint32_t hi, lo;
            uint8_t* dst = sm + G::OFF_THAT + es_sw(l, i) + t * 4;
            es_split(c[i][0], c[i][1], hi, lo);
            if (l < ELL) { *reinterpret_cast<uint32_t*>(dst) = hi; *reinterpret_cast<uint32_t*>(dst + G::LROWS * 64) = lo; }
            es_split(c[i][2], c[i][3], hi, lo);
            if (l + 8 < ELL) { *reinterpret_cast<uint32_t*>(dst + 8 * 64) = hi; *reinterpret_cast<uint32_t*>(dst + (G::LROWS + 8) * 64) = lo; }
          }
        }
      }
    }
    if (last) break;
    // ---- history <- links, 16 rows at a time, rows replaced in place
    const uint8_t* K2 = sm + G::OFF_OPS + HL * 64;
    const uint8_t* G2 = K2 + HL * 64;
    for (;;) {
      int tt = 0;
      if (lane == 0) tt = atomicAdd(next_tile, 1);
      tt = __shfl_sync(0xffffffffu, tt, 0);
      if (tt >= n_tiles) break;
      uint8_t* const xt = tile(tt * 16, raw);
      const uint4 a = es_lds(xt + es_sw(g, t)), a8 = es_lds(xt + es_sw(g + 8, t));
      uint4 ar = make_uint4(0, 0, 0, 0), ar8 = ar;
      if (raw) { ar = es_lds(rest(xt) + es_sw(g, t)); ar8 = es_lds(rest(xt) + es_sw(g + 8, t)); }
      float gt[4][4], up[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) gt[i][e] = up[i][e] = 0.f;
      // heads in groups that fill a k-step of 16 stacked rows
      constexpr int NTG = ELL < 16 ? 2 : ELL / 8;               // n-tiles per group
      constexpr int HPG = ELL < 16 ? 16 / ELL : 1;              // heads per group
#pragma unroll
      for (int q = 0; q < HL / 8; q += NTG) {
        float s[NTG][4];
#pragma unroll
        for (int i = 0; i < NTG; ++i) {
#pragma unroll
          for (int e = 0; e < 4; ++e) s[i][e] = 0.f;
          es_mma32(s[i], a, a8, es_lds(K2 + es_sw((q + i) * 8 + g, t)));
          if (SILU) es_mma32(s[i], a, a8, es_lds(sm + G::OFF_LO + HL * 64 + es_sw((q + i) * 8 + g, t)));
          if (raw) es_mma32(s[i], ar, ar8, es_lds(K2 + es_sw((q + i) * 8 + g, t)));
        }
        if (SILU) {
#pragma unroll
          for (int i = 0; i < NTG; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[i][e] = es_silu(s[i][e]) * (1.0f / ELL);
        } else {
#pragma unroll
          for (int hh = 0; hh < HPG; ++hh) {
            constexpr int NH = NTG / HPG;                       // n-tiles of one head
#pragma unroll
            for (int e = 0; e < 4; e += 2) {                    // rows g and g + 8
              float mx = -INFINITY, sum = 0.f;
#pragma unroll
              for (int i = hh * NH; i < (hh + 1) * NH; ++i) mx = fmaxf(mx, fmaxf(s[i][e], s[i][e + 1]));
              mx = es_quad_max(mx);
#pragma unroll
              for (int i = hh * NH; i < (hh + 1) * NH; ++i) {
                s[i][e] = es_ex2(s[i][e] - mx); s[i][e + 1] = es_ex2(s[i][e + 1] - mx);
                sum += s[i][e] + s[i][e + 1];
              }
              const float inv = __fdividef(1.0f, es_quad_sum(sum));
#pragma unroll
              for (int i = hh * NH; i < (hh + 1) * NH; ++i) { s[i][e] *= inv; s[i][e + 1] *= inv; }
            }
          }
        }
#pragma unroll
        for (int ks = 0; ks < NTG / 2; ++ks) {
          const uint32_t a0 = es_pack(s[2 * ks][0], s[2 * ks][1]), a1 = es_pack(s[2 * ks][2], s[2 * ks][3]);
          const uint32_t a2 = es_pack(s[2 * ks + 1][0], s[2 * ks + 1][1]), a3 = es_pack(s[2 * ks + 1][2], s[2 * ks + 1][3]);
          const int r = (q + 2 * ks) * 8 + (lane & 15);
          auto mix = [&](uint32_t b0, uint32_t b1, uint32_t b2, uint32_t b3) {
#pragma unroll
            for (int c0 = 0; c0 < 4; c0 += 2) {
              uint32_t w[4];
              es_ldsm_t(w, es_addr(G2 + es_sw(r, c0 + (lane >> 4))));
              es_mma(gt[c0], b0, b1, b2, b3, w[0], w[1]);
              es_mma(gt[c0 + 1], b0, b1, b2, b3, w[2], w[3]);
              es_ldsm_t(w, es_addr(G2 + HL * 64 + es_sw(r, c0 + (lane >> 4))));
              es_mma(up[c0], b0, b1, b2, b3, w[0], w[1]);
              es_mma(up[c0 + 1], b0, b1, b2, b3, w[2], w[3]);
            }
          };
          mix(a0, a1, a2, a3);
          if (SILU)
            mix(es_rest(s[2 * ks][0], s[2 * ks][1], a0), es_rest(s[2 * ks][2], s[2 * ks][3], a1), es_rest(s[2 * ks + 1][0], s[2 * ks + 1][1], a2),
                es_rest(s[2 * ks + 1][2], s[2 * ks + 1][3], a3));
        }
      }
      uint32_t u[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        u[i][0] = es_pack(es_silu(gt[i][0]) * up[i][0], es_silu(gt[i][1]) * up[i][1]);
        u[i][1] = es_pack(es_silu(gt[i][2]) * up[i][2], es_silu(gt[i][3]) * up[i][3]);
      }
      float c[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint32_t w[4];
        es_ldb(w, W + 5 * 2048, i, lane);
#pragma unroll
        for (int e = 0; e < 4; ++e) c[i][e] = 0.f;
        es_mma(c[i], u[0][0], u[0][1], u[1][0], u[1][1], w[0], w[1]);
        es_mma(c[i], u[2][0], u[2][1], u[3][0], u[3][1], w[2], w[3]);
      }
      if (p.ln) { es_ln(c, 0, p.eps); es_ln(c, 2, p.eps); }
      __syncwarp();                                             // every lane has read its rows of the tile
      const int r0 = tt * 16 + g;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t lo = es_pack(c[i][0], c[i][1]), hi = es_pack(c[i][2], c[i][3]);
        if (resident) {
          // rows past the end of the history stay zero
          if (r0 < n) *reinterpret_cast<uint32_t*>(X + es_sw(r0, i) + t * 4) = lo;
          if (r0 + 8 < n) *reinterpret_cast<uint32_t*>(X + es_sw(r0 + 8, i) + t * 4) = hi;
        } else {
          __nv_bfloat16* dst = p.scratch + (int64_t)(tok0 + r0) * ES_D + i * 8 + 2 * t;
          if (r0 < n) *reinterpret_cast<uint32_t*>(dst) = lo;
          if (r0 + 8 < n) *reinterpret_cast<uint32_t*>(dst + 8 * ES_D) = hi;
        }
      }
    }
  }
  // L^P, as the link states (or for the projection that follows)
  if (warp < LMT && rank == 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 4; e += 2) {
        const int l = warp * 16 + g + 4 * e;
        if (l >= ELL) continue;
        const int64_t at = ((int64_t)b * ELL + l) * ES_D + i * 8 + 2 * t;
        if (p.link_states) *reinterpret_cast<uint32_t*>(p.link_states + at) = es_pack(lp[i][e], lp[i][e + 1]);
        else *reinterpret_cast<float2*>(p.lp + at) = make_float2(lp[i][e], lp[i][e + 1]);
      }
  }
}

static bool es_shape(int H, int ell) { return (H == 2 || H == 4) && (ell == 8 || ell == 16 || ell == 32); }
bool encode_small_supported(int dtype, int d, int d_ff, int H, int ell, int gated_mlp) {
  return dtype == LIME_BF16 && d == ES_D && d_ff == ES_D && gated_mlp && es_shape(H, ell);
}

template <class G, bool SILU, bool RAW>
static lime_status launch_es_t(const EncodeSmallArgs& a, cudaStream_t st) {
  EncodeSmallParams p;
  p.hist = (const __nv_bfloat16*)a.hist; p.off = a.off; p.links = a.links; p.links_per_user = a.links_per_user;
  for (int j = 0; j < a.n_layers; ++j) {
    const void* w[6] = {a.w->Wq[j], a.w->Wk[j], a.w->Wv[j], a.w->Wg[j], a.w->Wu[j], a.w->Wo[j]};
    for (int m = 0; m < 6; ++m) p.w[j][m] = (const __nv_bfloat16*)w[m];
  }
  p.scratch = (__nv_bfloat16*)a.scratch; p.link_states = (__nv_bfloat16*)a.link_states; p.lp = a.lp;
  p.n_layers = a.n_layers; p.ln = a.ln; p.eps = a.eps; p.scale = SILU ? 1.0f : a.scale * 1.4426950408889634f;
  p.B = a.B; p.skip_long = 0;
  constexpr int row_bytes = RAW ? 128 : 64, most = (232448 - G::OFF_X) / row_bytes / 16 * 16, cap = most < ES_CAP ? most : ES_CAP;
  p.cap = (int)(a.total < cap ? a.total : cap);
  const int smem = G::OFF_X + ((p.cap + 15) & ~15) * row_bytes;
  static bool smem_set[kMaxDeviceOrdinals] = {};
  lime_status s = ensure_dynamic_smem((const void*)k_encode_small<G, SILU, RAW>, G::OFF_X + cap * row_bytes, smem_set);
  if (s != LIME_OK) return s;
  // as many clusters as the total allows long users, which find theirs or leave; no launch where it allows none
  int64_t longs = a.total / (ES_LONG + 1);
  if (longs > a.B) longs = a.B;
  if (longs > ES_CLUSTERS) longs = ES_CLUSTERS;
  if (longs > 0) {
    p.clustered = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)longs * ES_CLUSTER);
    cfg.blockDim = dim3(ES_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = ES_CLUSTER; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    ProfScope _p("k_encode_small", st);
    cudaLaunchKernelEx(&cfg, k_encode_small<G, SILU, RAW>, p);
    LIME_LAUNCH_CHECK("k_encode_small");
  }
  p.clustered = 0;
  p.skip_long = longs > 0;
  ProfScope _p("k_encode_small", st);
  launch_pdl(k_encode_small<G, SILU, RAW>, dim3((unsigned)a.B), dim3(ES_THREADS), (size_t)smem, st, p);
  LIME_LAUNCH_CHECK("k_encode_small");
  return LIME_OK;
}

template <class G>
static lime_status launch_es(const EncodeSmallArgs& a, cudaStream_t st) {
  if (a.silu) return a.hist_ln ? launch_es_t<G, true, true>(a, st) : launch_es_t<G, true, false>(a, st);
  return a.hist_ln ? launch_es_t<G, false, true>(a, st) : launch_es_t<G, false, false>(a, st);
}

lime_status launch_encode_small(const EncodeSmallArgs& a, cudaStream_t st) {
  switch (a.H * 100 + a.ell) {
    case 208: return launch_es<EsCfg<2, 8>>(a, st);
    case 216: return launch_es<EsCfg<2, 16>>(a, st);
    case 232: return launch_es<EsCfg<2, 32>>(a, st);
    case 408: return launch_es<EsCfg<4, 8>>(a, st);
    case 416: return launch_es<EsCfg<4, 16>>(a, st);
    case 432: return launch_es<EsCfg<4, 32>>(a, st);
  }
  return LIME_UNSUPPORTED_SHAPE;
}

}  // namespace lime
