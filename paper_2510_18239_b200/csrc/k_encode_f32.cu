// The whole user-side encode in one launch for fp32 storage at d = d_ff = 64 (CUDA cores, fp32 throughout): all XOR layers of a
// user in one cluster of blocks, every block keeping its share of the history in shared memory (Eq. 7, Eq. 5, Eq. 8).
//
// With the history-side projections folded into the few link rows a token takes about 9 k multiply-adds per layer (28 k with
// Q / K / V / O rows formed), so what bounds it is the FMA rate where histories are long and the latency of the chain of
// small steps where they are short.  FMAs: a shared-memory load fills 4 bytes a lane per clock however many lanes share the
// address, against four FMAs of a warp, so a product only runs near the FMA rate with register tiles (8 tokens x 8 or 4
// columns here, two thirds of it); a lane or a quad per token, with everything in registers and every operand a broadcast,
// was measured first and is bound by those loads (21 and 38 us a layer however short the history).  Tiles are 128 tokens.
// Chain: the blocks of a user exchange one message per layer (maximum, sum and accumulator of their share, pushed into each
// other's shared memory with the arrival counted on a barrier there) and then do the link rows redundantly; a weight is read
// straight from L2 into registers by the thread that multiplies with it, a step ahead of its use, a quarter of the
// contraction per thread (reads of adjacent columns by adjacent lanes: split over the lanes of a quad instead, they were the
// largest part of a layer).
#include "lime_common.cuh"
#include "tc_common.cuh"

namespace lime {

constexpr int EF_D = 64, EF_THREADS = 256, EF_TILE = 128;
// A user whose share would be over 2048 tokens takes a cluster of sixteen blocks, in a launch of their own, at most seven of them (the
// clusters that run at once; the line doubles until that holds).  One user of n tokens among 99 of 100, two layers, without it /
// with it / the generic kernels, which split by token: n = 2000 351 / 353 / 395 us, 4000 680 / 105 / 442, 32000 2985 / 466 / 886,
// 150000 3645 / 2050 / 2035; 200000 among 399 of 50: 9817 / 2820 / 2612.
constexpr int EF_LONG = 2048, EF_LONG_CLUSTER = 16, EF_LONG_CLUSTERS = 7;
// From 37 users on - two blocks a user run at once up to 72, one beyond - the blocks are dealt by length instead (ef_plan), in clusters of
// four, of which 33 run at once.  A share below 48 tokens does not pay for the exchange.  Two layers, same blocks for every user / dealt:
// 64 users of 50..1000 113.7 / 79.1 us, 64 of 525 88.0 / 68.0, 40 of 8..1000 80.8 / 61.0, 80 of 125..1000 131.2 / 115.3, 100 of 0..500
// 91.6 / 80.8, one of 1900 among 99 of 100 374 / 115; where there is nothing to deal the plan costs 1 to 4 us: 132 of 10..300 68.8 /
// 72.8, 60 of 1..100 37.6 / 39.2, hence up to 116 users and from a mean of two shares on.
constexpr int EF_PLAN_FROM = 37, EF_PLAN_CLUSTERS = 33, EF_PLAN_USERS = 116, EF_SHARE = 48;
constexpr int EF_LD = 68;                                        // floats per row of operands read along the contraction: spreads the banks

template <int H_, int ELL_>
struct EfCfg {
  static constexpr int H = H_, ELL = ELL_, HL = H * ELL, DH = EF_D / H;
  static constexpr int PLD = HL + 4;                             // floats per row of scores / probabilities
  static constexpr int MSG = HL * EF_D + 2 * HL;                 // floats of a block's message: accumulator, maxima, sums
  // float offsets
  static constexpr int Q2 = 0;                                   // [HL x EF_LD]
  static constexpr int K2 = Q2 + HL * EF_LD;                     // [HL x EF_LD]
  static constexpr int GU = K2 + HL * EF_LD;                     // [HL x (gate 64 | up 64)]
  static constexpr int WO = GU + HL * 2 * EF_D;                  // [64 x 64]
  static constexpr int S = WO + EF_D * EF_D;                     // [tile x PLD] scores, then probabilities
  static constexpr int U = S + EF_TILE * PLD;                    // [tile x EF_LD] hidden units
  static constexpr int S_END = U + EF_TILE * EF_LD;
  static constexpr int PART = U;                                 // over U: partial accumulators [4][HL x 64]
  static constexpr int RED = S;                                  // over S and U: [4 quarters][ELL x 64] x up to 4 products
  static constexpr int R_END = RED + 16 * ELL * EF_D > S_END ? RED + 16 * ELL * EF_D : S_END;
  static_assert(4 * HL * EF_D <= EF_TILE * EF_LD, "partial accumulators over U");
  static constexpr int OHAT = R_END;                             // [HL x 64]
  static constexpr int THAT = OHAT + HL * EF_D;                  // [ELL x 64] each
  static constexpr int ROW_A = THAT + ELL * EF_D;                // Q, then O
  static constexpr int ROW_B = ROW_A + ELL * EF_D;               // K, then U
  static constexpr int ROW_C = ROW_B + ELL * EF_D;               // V, then T
  static constexpr int LP = ROW_C + ELL * EF_D;
  static constexpr int MX = LP + ELL * EF_D;                     // [tokens' 256 / HL shares][HL]: maxima, then sums
  static constexpr int RUN = MX + EF_THREADS;                    // [HL] running maximum, [HL] running sum, [HL] factor
  static constexpr int BAR = RUN + 3 * HL;                       // one barrier
  static constexpr int EX = BAR + 4;                             // [2 layers' parity][cluster][MSG], then the history rows
};

struct EncodeF32Params {
  const float* hist; const int32_t* off;
  const float* links; int links_per_user;
  const float* w[LIME_MAX_LAYERS][6];                            // W_Q, W_K, W_V (NULL: identity), W_g, W_u, W_o
  float* scratch;                                                // [total x d]: histories beyond shared memory
  float* out;                                                    // L^P
  int B, longer_than, skip_long;                                 // a user has to be longer than that to be a long one
  int planned, total;                                            // 1: the blocks of a cluster are dealt to users by length (ef_plan)
  int n_layers, cluster, cap, ln, hist_ln, silu;                 // cap: history rows a block holds
  float eps, scale;                                              // scale times log2 e with the softmax
  int* err;
};

__device__ __forceinline__ float ef_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ef_silu(float x) { return __fdividef(x, 1.0f + __expf(-x)); }
__device__ __forceinline__ float4 ef_ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void ef_push(uint32_t addr, const float4& v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(addr), "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)), "r"(__float_as_uint(v.w)), "r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t ef_peer(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// 16 weights of column c: rows k0 .. k0 + 15 of W [64 x 64] (NULL: identity)
__device__ __forceinline__ void ef_wcol(float (&w)[16], const float* __restrict__ W, int k0, int c) {
#pragma unroll
  for (int k = 0; k < 16; ++k) w[k] = W != nullptr ? __ldg(W + (k0 + k) * EF_D + c) : (k0 + k == c ? 1.f : 0.f);
}
// the same of row i: columns k0 ..
__device__ __forceinline__ void ef_wrow(float (&w)[16], const float* __restrict__ W, int k0, int i) {
#pragma unroll
  for (int k = 0; k < 16; k += 4) {
    const float4 v = W != nullptr ? __ldg(reinterpret_cast<const float4*>(W + i * EF_D + k0 + k))
                                  : make_float4(k0 + k == i, k0 + k + 1 == i, k0 + k + 2 == i, k0 + k + 3 == i);
    w[k] = v.x; w[k + 1] = v.y; w[k + 2] = v.z; w[k + 3] = v.w;
  }
}
// red[q][r * 64 + c] = sum over this thread's 16 of the contraction of rows[r][k0 ..] . w[q], for NR rows and NW weights that
// share them (the rows' reads are what such a product costs)
template <int NR, int NW>
__device__ __forceinline__ void ef_quarter(float* const (&red)[NW], const float* rows, const float (*const (&w)[NW])[16], int k0, int c) {
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    float s[NW];
#pragma unroll
    for (int q = 0; q < NW; ++q) s[q] = 0.f;
#pragma unroll
    for (int k = 0; k < 16; k += 4) {
      const float4 a = ef_ld4(rows + r * EF_D + k0 + k);
#pragma unroll
      for (int q = 0; q < NW; ++q) {
        s[q] = fmaf(a.x, (*w[q])[k], s[q]); s[q] = fmaf(a.y, (*w[q])[k + 1], s[q]);
        s[q] = fmaf(a.z, (*w[q])[k + 2], s[q]); s[q] = fmaf(a.w, (*w[q])[k + 3], s[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < NW; ++q) red[q][r * EF_D + c] = s[q];
  }
}
// acc[i][n] += A[i] . B[n] over four of the contraction, both read along it
template <int M, int N>
__device__ __forceinline__ void ef_dot4(float (&acc)[M][N], const float4 (&a)[M], const float4 (&b)[N]) {
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int n = 0; n < N; ++n) {
      acc[i][n] = fmaf(a[i].x, b[n].x, acc[i][n]); acc[i][n] = fmaf(a[i].y, b[n].y, acc[i][n]);
      acc[i][n] = fmaf(a[i].z, b[n].z, acc[i][n]); acc[i][n] = fmaf(a[i].w, b[n].w, acc[i][n]);
    }
}
__device__ __forceinline__ void ef_fma4(float (&acc)[4], float a, const float4& b) {
  acc[0] = fmaf(a, b.x, acc[0]); acc[1] = fmaf(a, b.y, acc[1]); acc[2] = fmaf(a, b.z, acc[2]); acc[3] = fmaf(a, b.w, acc[3]);
}
// S[token][row] = X[token] . ops[row] for a tile of nr <= 16 M tokens: thread = M / 2 tokens (tg, tg + 32, ..) x HL / 8 rows
// (rg, rg + 8, ..)
template <class G, int M>
__device__ __forceinline__ void ef_scores(float* S, const float* x, int xld, const float* ops, int nr, int tid) {
  constexpr int NR = G::HL / 8, MT = M / 2;
  const int tg = tid >> 3, rg = tid & 7;
  if (tg >= nr) return;
  float acc[MT][NR];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[i][r] = 0.f;
  const float* xr[MT];
#pragma unroll
  for (int i = 0; i < MT; ++i) xr[i] = x + (int64_t)min(tg + 32 * i, nr - 1) * xld;
#pragma unroll 4
  for (int k = 0; k < EF_D; k += 4) {
    float4 a[MT], b[NR];
#pragma unroll
    for (int i = 0; i < MT; ++i) a[i] = ef_ld4(xr[i] + k);
#pragma unroll
    for (int r = 0; r < NR; ++r) b[r] = ef_ld4(ops + (rg + 8 * r) * EF_LD + k);
    ef_dot4(acc, a, b);
  }
#pragma unroll
  for (int i = 0; i < MT; ++i)
    if (tg + 32 * i < nr)
#pragma unroll
      for (int r = 0; r < NR; ++r) S[(tg + 32 * i) * G::PLD + rg + 8 * r] = acc[i][r];
}

// history <- links for a tile of nr <= 16 M tokens at x, rows replaced in place (contains barriers: every thread calls it)
template <class G, int M>
__device__ __forceinline__ void ef_update_tile(float* fs, float* x, int ld, int nr, int tid, int silu, int ln, float eps) {
  constexpr int H = G::H, ELL = G::ELL, HL = G::HL, D = EF_D;
  ef_scores<G, M>(fs + G::S, x, ld, fs + G::K2, nr, tid);
  __syncthreads();
  // probabilities: thread = (token, head)
  for (int i = tid; i < nr * H; i += EF_THREADS) {
    float* s = fs + G::S + (i / H) * G::PLD + (i % H) * ELL;
    float v[ELL];
#pragma unroll
    for (int l = 0; l < ELL; l += 4) *reinterpret_cast<float4*>(v + l) = ef_ld4(s + l);
    if (silu) {
#pragma unroll
      for (int l = 0; l < ELL; ++l) v[l] = ef_silu(v[l]) * (1.0f / ELL);
    } else {
      float m = v[0], sum = 0.f;
#pragma unroll
      for (int l = 1; l < ELL; ++l) m = fmaxf(m, v[l]);
#pragma unroll
      for (int l = 0; l < ELL; ++l) { v[l] = ef_ex2(v[l] - m); sum += v[l]; }
      const float inv = 1.0f / sum;
#pragma unroll
      for (int l = 0; l < ELL; ++l) v[l] *= inv;
    }
#pragma unroll
    for (int l = 0; l < ELL; l += 4) *reinterpret_cast<float4*>(s + l) = make_float4(v[l], v[l + 1], v[l + 2], v[l + 3]);
  }
  __syncthreads();
  // [gate | up] = P [G2 | U2], U = SiLU(gate) * up: thread = M tokens (tg, tg + 16, ..) x 4 hidden units
  const int tg = tid >> 4, fg = tid & 15;
  if (tg < nr) {
    float gt[M][4], up[M][4];
#pragma unroll
    for (int i = 0; i < M; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) gt[i][e] = up[i][e] = 0.f;
#pragma unroll 1
    for (int r = 0; r < HL; r += 4) {
      float4 a[M];
#pragma unroll
      for (int i = 0; i < M; ++i) a[i] = ef_ld4(fs + G::S + min(tg + 16 * i, nr - 1) * G::PLD + r);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 g4 = ef_ld4(fs + G::GU + (r + q) * 2 * D + fg * 4), u4 = ef_ld4(fs + G::GU + (r + q) * 2 * D + D + fg * 4);
#pragma unroll
        for (int i = 0; i < M; ++i) {
          const float w = q == 0 ? a[i].x : q == 1 ? a[i].y : q == 2 ? a[i].z : a[i].w;
          ef_fma4(gt[i], w, g4);
          ef_fma4(up[i], w, u4);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < M; ++i)
      if (tg + 16 * i < nr)
        *reinterpret_cast<float4*>(fs + G::U + (tg + 16 * i) * EF_LD + fg * 4) =
            make_float4(ef_silu(gt[i][0]) * up[i][0], ef_silu(gt[i][1]) * up[i][1], ef_silu(gt[i][2]) * up[i][2], ef_silu(gt[i][3]) * up[i][3]);
  }
  __syncthreads();
  // rows = LN(U W_o): the same tokens x 4 columns; the 16 lanes of a token normalise it
  if (tg < nr) {
    float o[M][4];
#pragma unroll
    for (int i = 0; i < M; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[i][e] = 0.f;
#pragma unroll 2
    for (int k = 0; k < D; k += 4) {
      float4 a[M];
#pragma unroll
      for (int i = 0; i < M; ++i) a[i] = ef_ld4(fs + G::U + min(tg + 16 * i, nr - 1) * EF_LD + k);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 w4 = ef_ld4(fs + G::WO + (k + q) * D + fg * 4);
#pragma unroll
        for (int i = 0; i < M; ++i) ef_fma4(o[i], q == 0 ? a[i].x : q == 1 ? a[i].y : q == 2 ? a[i].z : a[i].w, w4);
      }
    }
    const unsigned half = tg & 1 ? 0xffff0000u : 0x0000ffffu;   // the token's lanes: a warp holds two token groups
#pragma unroll
    for (int i = 0; i < M; ++i) {
      if (ln) {
        float s = (o[i][0] + o[i][1]) + (o[i][2] + o[i][3]);
#pragma unroll
        for (int q = 8; q > 0; q >>= 1) s += __shfl_xor_sync(half, s, q);
        s *= 1.0f / D;
        float v = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) { o[i][e] -= s; v = fmaf(o[i][e], o[i][e], v); }
#pragma unroll
        for (int q = 8; q > 0; q >>= 1) v += __shfl_xor_sync(half, v, q);
        const float rstd = rsqrtf(v * (1.0f / D) + eps);
#pragma unroll
        for (int e = 0; e < 4; ++e) o[i][e] *= rstd;
      }
      if (tg + 16 * i < nr) *reinterpret_cast<float4*>(x + (int64_t)(tg + 16 * i) * ld + fg * 4) = make_float4(o[i][0], o[i][1], o[i][2], o[i][3]);
    }
  }
}

// Which user this block serves, as which of how many blocks, and where they begin in the cluster: the clusters of four are dealt by
// length, so that no share is much longer than the others.  A share length L is taken, a user gets one to four blocks of at most L
// tokens (no fewer than EF_SHARE each), and L grows from the mean until the users fit the clusters: those of four blocks take one each,
// those of three share theirs with one of one block, those of two go in pairs.  Every block finds the same L.  The long users of the other
// launch, if there is one, are left out (the line as long_user_line finds it).  Warp 0 works; word: four words of shared memory.
struct EfSlot { int b, rank, blocks, base; };
__device__ __forceinline__ EfSlot ef_plan(const int32_t* __restrict__ off, int B, int total, int longer_than, bool skip_long, int* word) {
  const int clusters = gridDim.x / 4, c = blockIdx.x / 4, q = blockIdx.x % 4, lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {
    constexpr int N = (EF_PLAN_USERS + 31) / 32;
    int len[N], most[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int b = i * 32 + lane;
      len[i] = b < B ? off[b + 1] - off[b] : -1;
    }
    for (int line = longer_than; skip_long; line *= 2) {
      int over = 0;
#pragma unroll
      for (int i = 0; i < N; ++i) over += len[i] > line;
      if (__reduce_add_sync(0xffffffffu, over) <= EF_LONG_CLUSTERS || line > (1 << 29)) {
#pragma unroll
        for (int i = 0; i < N; ++i) len[i] = len[i] > line ? -1 : len[i];
        break;
      }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) most[i] = max(1, min(4, len[i] / EF_SHARE));
    int L = max(EF_SHARE, (total + 4 * clusters - 1) / (4 * clusters)), n1, n2, n3, n4;
    auto blocks = [&](int i) { return len[i] < 0 ? 0 : min(most[i], 1 + (len[i] > L) + (len[i] > 2 * L) + (len[i] > 3 * L)); };
    for (;;) {
      int cnt = 0;                                               // users of one, two, three and four blocks, a byte each
#pragma unroll
      for (int i = 0; i < N; ++i) { const int k = blocks(i); cnt += k ? 1 << (8 * (k - 1)) : 0; }
      cnt = __reduce_add_sync(0xffffffffu, cnt);
      n1 = cnt & 255; n2 = (cnt >> 8) & 255; n3 = (cnt >> 16) & 255; n4 = (cnt >> 24) & 255;
      const int single = max(0, n1 - n3 - 2 * (n2 & 1));
      if (n4 + n3 + (n2 + 1) / 2 + (single + 3) / 4 <= clusters || L > (1 << 28)) break;
      L += max(8, L / 16);
    }
    const int c3 = c - n4, c2 = c3 - n3, c1 = c2 - (n2 + 1) / 2;
    int k = 1, which, rank = 0, base = q;                        // the which-th user of k blocks
    if (c3 < 0) { k = 4; which = c; rank = q; base = 0; }
    else if (c2 < 0) {
      which = c3;
      if (q < 3) { k = 3; rank = q; base = 0; }
    } else if (c1 < 0) {
      which = 2 * c2 + (q >> 1);
      if (which < n2) { k = 2; rank = q & 1; base = q & 2; }
      else which = n3 + (q & 1);
    } else which = n3 + 2 * (n2 & 1) + 4 * c1 + q;
    if (lane == 0) { word[0] = -1; word[1] = rank; word[2] = k; word[3] = base; }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const unsigned m = __ballot_sync(0xffffffffu, blocks(i) == k);
      if (((m >> lane) & 1u) && __popc(m & ((1u << lane) - 1u)) == which) word[0] = i * 32 + lane;
      which -= __popc(m);
    }
  }
  __syncthreads();
  const EfSlot s{word[0], word[1], word[2], word[3]};
  __syncthreads();
  return s;
}

// LONG: cluster k takes the k-th long user, and the blocks read each other's message in place (pushed, sixteen slots would not fit
// beside the operands); without it cluster b takes user b and a long user is left out.
template <class G, bool LONG>
__global__ void __launch_bounds__(EF_THREADS, 1)
k_encode_f32(const EncodeF32Params p) {
  constexpr int ELL = G::ELL, HL = G::HL, DH = G::DH, D = EF_D;
  extern __shared__ __align__(128) float fs[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int CL = LONG ? EF_LONG_CLUSTER : p.cluster;
  const int c = tid & 63, kq = tid >> 6, k0 = kq * 16;           // link rows: output column, quarter of the contraction
  float* const ex = fs + G::EX;
  float* const X = ex + (LONG ? 1 : 2 * CL) * G::MSG;
  uint64_t* const bar = reinterpret_cast<uint64_t*>(fs + G::BAR);
  if (!LONG && tid == 0) {
    tc::mbar_init(bar, 1);
    tc::fence_barrier_init();
  }
  if (!LONG && CL > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  pdl_launch_dependents();
  pdl_wait();
  int* const word = reinterpret_cast<int*>(fs + G::MX);
  EfSlot me{(int)blockIdx.x / CL, (int)blockIdx.x % CL, CL, 0};
  if (LONG) me.b = nth_long_user(p.off, p.B, p.longer_than, EF_LONG_CLUSTERS, blockIdx.x / CL, word);
  if (LONG && me.b < 0) return;                                  // the whole cluster
  if (!LONG && p.planned)
    me = ef_plan(p.off, p.B, p.total, p.longer_than, p.skip_long != 0, word);
  const int b = me.b, rank = me.rank, nb = me.blocks;
  const int u0 = b < 0 ? 0 : p.off[b], un = b < 0 ? 0 : p.off[b + 1] - u0;
  if (!LONG && (b < 0 || (!p.planned && p.skip_long && un > p.longer_than &&
                          un > long_user_line(p.off, p.B, p.longer_than, EF_LONG_CLUSTERS, word)))) {
    if (CL > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    return;
  }
  const uint32_t msg_bytes = (uint32_t)(nb - 1) * G::MSG * 4;
  // (a peer's message that is here before the bytes are expected is counted all the same: the phase waits for this arrival)
  if (!LONG && tid == 0) tc::mbar_arrive_expect_tx(bar, msg_bytes);
  const int share = (un + nb - 1) / nb, tok0 = u0 + min(un, rank * share), n = min(un, (rank + 1) * share) - min(un, rank * share);
  const bool resident = share <= p.cap;
  float* const rows = resident ? X : p.scratch + (int64_t)tok0 * D;    // the block's history
  const int ld = resident ? EF_LD : D;

  // operand weights of the first layer are on their way while the history comes in
  float wa[16], wb[16], wc[16];
  ef_wcol(wa, p.w[0][0], k0, c); ef_wcol(wb, p.w[0][1], k0, c); ef_wcol(wc, p.w[0][2], k0, c);
  for (int i = tid; i < ((n + 15) & ~15) * 16; i += EF_THREADS) {   // 16 lanes per row
    const int row = i >> 4, q = i & 15;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < n) v = __ldg(reinterpret_cast<const float4*>(p.hist + (int64_t)(tok0 + row) * D) + q);
    if (p.hist_ln) {
      float s = v.x + v.y + v.z + v.w;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const float mu = s * (1.0f / D);
      v.x -= mu; v.y -= mu; v.z -= mu; v.w -= mu;
      s = v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const float rstd = rsqrtf(s * (1.0f / D) + p.eps);
      v.x *= rstd; v.y *= rstd; v.z *= rstd; v.w *= rstd;
    }
    if (row < n) *reinterpret_cast<float4*>(rows + (int64_t)row * ld + q * 4) = v;
  }
  // LN of link row r (64 values at src) -> That, by one warp
  auto ln_row = [&](const float* src, int r) {
    float2 x = *reinterpret_cast<const float2*>(src + lane * 2);
    if (p.ln) {
      const float mu = warp_sum(x.x + x.y) * (1.0f / D);
      x.x -= mu; x.y -= mu;
      const float rstd = rsqrtf(warp_sum(x.x * x.x + x.y * x.y) * (1.0f / D) + p.eps);
      x.x *= rstd; x.y *= rstd;
    }
    *reinterpret_cast<float2*>(fs + G::THAT + r * D + lane * 2) = x;
  };
  for (int r = warp; r < ELL; r += 8) ln_row(p.links + (p.links_per_user ? (int64_t)b * ELL * D : 0) + r * D, r);
  for (int i = tid; i < ELL * D; i += EF_THREADS) fs[G::LP + i] = 0.f;

  // sum of the four quarters of product `which` at row r, column col; head_sum: of head h's quarters only
  auto red4 = [&](int which, int r, int col) {
    const float* s = fs + G::RED + which * 4 * ELL * D + r * D + col;
    return (s[0] + s[ELL * D]) + (s[2 * ELL * D] + s[3 * ELL * D]);
  };
  auto head_sum = [&](int which, int h, int l, int col) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < DH / 16; ++q) s += fs[G::RED + (which * 4 + h * (DH / 16) + q) * ELL * D + l * D + col];
    return s;
  };
  auto red_at = [&](int which) { return fs + G::RED + (which * 4 + kq) * ELL * D; };

  for (int j = 0; j < p.n_layers; ++j) {
    const bool last = j + 1 == p.n_layers;
    __syncthreads();
    // ---- Q | K | V of the link rows, then Q2 (K2 and [G2 | U2] follow behind the attention)
    ef_quarter<ELL, 3>({red_at(0), red_at(1), red_at(2)}, fs + G::THAT, {&wa, &wb, &wc}, k0, c);
    if (!last)                                                    // W_o for the history update, under all that comes before it
      for (int i = tid; i < D * D / 4; i += EF_THREADS)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(fs + G::WO + i * 4)), "l"(p.w[j][5] + i * 4) : "memory");
    ef_wrow(wa, p.w[j][1], k0, c);
    __syncthreads();
    for (int i = tid; i < ELL * D; i += EF_THREADS) {
      fs[G::ROW_A + i] = red4(0, i / D, i % D);
      fs[G::ROW_B + i] = red4(1, i / D, i % D);
      fs[G::ROW_C + i] = red4(2, i / D, i % D);
    }
    if (tid < HL) { fs[G::RUN + tid] = p.silu ? 0.f : -INFINITY; fs[G::RUN + HL + tid] = 0.f; }
    __syncthreads();
    ef_quarter<ELL, 1>({red_at(0)}, fs + G::ROW_A, {&wa}, k0, c);
    __syncthreads();
    for (int i = tid; i < HL * D; i += EF_THREADS)
      fs[G::Q2 + (i / D) * EF_LD + i % D] = head_sum(0, i / (ELL * D), (i / D) % ELL, i % D) * p.scale;
    // ---- links <- history over this block's share, a tile at a time.  Values: thread = tokens grp, grp + 4, .. x rows rg *
    // HL / 4 .. x columns cg * 4 ..
    constexpr int RPT = HL / 4, SEG = EF_THREADS / HL;
    float acc[RPT][4];
#pragma unroll
    for (int r = 0; r < RPT; ++r)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[r][e] = 0.f;
    const int grp = tid >> 6, rg = (tid >> 4) & 3, cg = tid & 15;
    for (int r0 = 0; r0 < n; r0 += EF_TILE) {
      const int nr = min(EF_TILE, n - r0);
      __syncthreads();
      if (nr > 64) ef_scores<G, 8>(fs + G::S, rows + (int64_t)r0 * ld, ld, fs + G::Q2, nr, tid);
      else ef_scores<G, 4>(fs + G::S, rows + (int64_t)r0 * ld, ld, fs + G::Q2, nr, tid);
      __syncthreads();
      // probabilities of stacked row pr, tokens seg, seg + SEG, ..: against the running maximum of the row
      const int pr = tid % HL, seg = tid / HL;
      float* const sp = fs + G::S + pr;
      float sum = 0.f;
      if (!p.silu) {
        float m = -INFINITY;
        for (int i = seg; i < nr; i += SEG) m = fmaxf(m, sp[i * G::PLD]);
        fs[G::MX + seg * HL + pr] = m;
        __syncthreads();
        m = fs[G::RUN + pr];
        const float m_old = m;
#pragma unroll
        for (int s = 0; s < SEG; ++s) m = fmaxf(m, fs[G::MX + s * HL + pr]);
        for (int i = seg; i < nr; i += SEG) {
          const float e = ef_ex2(sp[i * G::PLD] - m);
          sp[i * G::PLD] = e;
          sum += e;
        }
        __syncthreads();                                          // every thread has the maxima
        if (seg == 0) { fs[G::RUN + pr] = m; fs[G::RUN + 2 * HL + pr] = ef_ex2(m_old - m); }
      } else {
        for (int i = seg; i < nr; i += SEG) sp[i * G::PLD] = ef_silu(sp[i * G::PLD]);
        if (seg == 0) fs[G::RUN + 2 * HL + pr] = 1.f;
      }
      fs[G::MX + seg * HL + pr] = sum;
      __syncthreads();
      if (tid < HL) {
        float s = fs[G::RUN + HL + tid] * fs[G::RUN + 2 * HL + tid];
#pragma unroll
        for (int q = 0; q < SEG; ++q) s += fs[G::MX + q * HL + tid];
        fs[G::RUN + HL + tid] = s;
      }
      if (r0 > 0)
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
          const float f = fs[G::RUN + 2 * HL + rg * RPT + r];
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[r][e] *= f;
        }
      const float* xv = rows + (int64_t)r0 * ld + cg * 4;
#pragma unroll 2
      for (int i = grp; i < nr; i += 4) {
        const float4 x = ef_ld4(xv + (int64_t)i * ld);
#pragma unroll
        for (int r = 0; r < RPT; r += 4) {
          const float4 w = ef_ld4(fs + G::S + i * G::PLD + rg * RPT + r);
          ef_fma4(acc[r], w.x, x); ef_fma4(acc[r + 1], w.y, x); ef_fma4(acc[r + 2], w.z, x); ef_fma4(acc[r + 3], w.w, x);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < RPT; ++r)
      *reinterpret_cast<float4*>(fs + G::PART + (grp * HL + rg * RPT + r) * D + cg * 4) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
    // the message: accumulator, maxima, sums of this share -> slot `rank` here and in every peer
    float* const slot = LONG ? ex : ex + ((j & 1) * CL + rank) * G::MSG;
    // weights of what follows
    float wk[16];
    if (!last) ef_wrow(wk, p.w[j][0], k0, c);
    ef_wcol(wa, p.w[j][2], k0, c); ef_wcol(wb, p.w[j][3], k0, c); ef_wcol(wc, p.w[j][4], k0, c);
    __syncthreads();
    for (int i = tid; i < HL * D / 4; i += EF_THREADS) {
      const float* s = fs + G::PART + i * 4;
      const float4 x = ef_ld4(s), y = ef_ld4(s + HL * D), z = ef_ld4(s + 2 * HL * D), w = ef_ld4(s + 3 * HL * D);
      *reinterpret_cast<float4*>(slot + i * 4) = make_float4((x.x + y.x) + (z.x + w.x), (x.y + y.y) + (z.y + w.y), (x.z + y.z) + (z.z + w.z), (x.w + y.w) + (z.w + w.w));
    }
    if (tid < 2 * HL) slot[HL * D + tid] = fs[G::RUN + tid];      // maxima, sums
    if (LONG) cluster_sync_all();
    else __syncthreads();
    if (!LONG && CL > 1 && j == 0) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");     // the peers run
    if (!LONG && nb > 1) {
      const uint32_t at = (uint32_t)__cvta_generic_to_shared(slot), ba = (uint32_t)__cvta_generic_to_shared(bar);
      for (int i = tid; i < G::MSG / 4; i += EF_THREADS) {
        const float4 v = ef_ld4(slot + i * 4);
        for (int r = 1; r < nb; ++r) ef_push(ef_peer(at + i * 16, me.base + (rank + r) % nb), v, ef_peer(ba, me.base + (rank + r) % nb));
      }
      tc::mbar_wait(bar, (uint32_t)j & 1u, p.err, 88);
    }
    // ---- merge the shares: Ohat [(h, l)][64]
    for (int i = tid; i < HL * D / 4; i += EF_THREADS) {
      const int r = i / (D / 4);
      float M = -INFINITY, S = 0.f;
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
      auto msg = [&](int q) -> const float* {
        if constexpr (LONG) return cluster_peer(static_cast<const float*>(ex), q);
        else return ex + ((j & 1) * CL + q) * G::MSG;
      };
      for (int q = 0; q < nb; ++q) M = fmaxf(M, msg(q)[HL * D + r]);
      for (int q = 0; q < nb; ++q) {
        const float m = msg(q)[HL * D + r], w = m == -INFINITY ? 0.f : ef_ex2(m - M);
        S = fmaf(w, msg(q)[HL * D + HL + r], S);
        const float4 x = ef_ld4(msg(q) + i * 4);
        o.x = fmaf(w, x.x, o.x); o.y = fmaf(w, x.y, o.y); o.z = fmaf(w, x.z, o.z); o.w = fmaf(w, x.w, o.w);
      }
      const float inv = un > 0 ? 1.0f / (p.silu ? (float)un : S) : 0.f;
      *reinterpret_cast<float4*>(fs + G::OHAT + i * 4) = make_float4(o.x * inv, o.y * inv, o.z * inv, o.w * inv);
    }
    if (LONG) cluster_sync_all();                                 // the peers have read this block's message
    else __syncthreads();
    if (!LONG && tid == 0 && !last) tc::mbar_arrive_expect_tx(bar, msg_bytes);     // every thread has seen this layer's messages
    // ---- what the history update multiplies with (K, V of this layer still in their rows): K2, [G2 | U2], W_o
    if (!last) {
      ef_quarter<ELL, 2>({red_at(2), red_at(3)}, fs + G::ROW_C, {&wb, &wc}, k0, c);
      ef_quarter<ELL, 1>({red_at(1)}, fs + G::ROW_B, {&wk}, k0, c);
      asm volatile("cp.async.wait_all;" ::: "memory");
    }
    // O = Ohat W_V: column c belongs to head c / d_h
    ef_quarter<ELL, 1>({red_at(0)}, fs + G::OHAT + (c / DH) * ELL * D, {&wa}, k0, c);
    ef_wcol(wa, p.w[j][5], k0, c);
    __syncthreads();
    if (!last)
      for (int i = tid; i < HL * D; i += EF_THREADS) {
        const int h = i / (ELL * D), l = (i / D) % ELL, col = i % D, r = i / D;
        fs[G::K2 + r * EF_LD + col] = head_sum(1, h, l, col) * p.scale;
        fs[G::GU + r * 2 * D + col] = head_sum(2, h, l, col);
        fs[G::GU + r * 2 * D + D + col] = head_sum(3, h, l, col);
      }
    for (int i = tid; i < ELL * D; i += EF_THREADS) fs[G::ROW_A + i] = red4(0, i / D, i % D);
    __syncthreads();
    // ---- T = (SiLU(O W_g) * (O W_u)) W_o, L^P += T, LN(T)
    ef_quarter<ELL, 2>({red_at(0), red_at(1)}, fs + G::ROW_A, {&wb, &wc}, k0, c);
    __syncthreads();
    for (int i = tid; i < ELL * D; i += EF_THREADS) fs[G::ROW_B + i] = ef_silu(red4(0, i / D, i % D)) * red4(1, i / D, i % D);
    __syncthreads();
    ef_quarter<ELL, 1>({red_at(2)}, fs + G::ROW_B, {&wa}, k0, c);
    if (!last) { ef_wcol(wa, p.w[j + 1][0], k0, c); ef_wcol(wb, p.w[j + 1][1], k0, c); ef_wcol(wc, p.w[j + 1][2], k0, c); }
    __syncthreads();
    for (int i = tid; i < ELL * D; i += EF_THREADS) {
      const float t = red4(2, i / D, i % D);
      fs[G::ROW_C + i] = t;
      fs[G::LP + i] += t;
    }
    if (last) break;
    __syncthreads();
    for (int r = warp; r < ELL; r += 8) ln_row(fs + G::ROW_C + r * D, r);
    // ---- history <- links, a tile at a time, rows replaced in place
    // (a short last tile by the variant with fewer tokens a thread)
    for (int r0 = 0; r0 < n; r0 += EF_TILE) {
      const int nr = min(EF_TILE, n - r0);
      float* const x = rows + (int64_t)r0 * ld;
      if (nr > 64) ef_update_tile<G, 8>(fs, x, ld, nr, tid, p.silu, p.ln, p.eps);
      else if (nr > 32) ef_update_tile<G, 4>(fs, x, ld, nr, tid, p.silu, p.ln, p.eps);
      else ef_update_tile<G, 2>(fs, x, ld, nr, tid, p.silu, p.ln, p.eps);
    }
  }
  __syncthreads();
  if (rank == 0)
    for (int i = tid; i < ELL * D / 4; i += EF_THREADS) *(reinterpret_cast<float4*>(p.out + (int64_t)b * ELL * D) + i) = ef_ld4(fs + G::LP + i * 4);
}

bool encode_f32_supported(int dtype, int d, int d_ff, int H, int ell, int gated_mlp) {
  return dtype == LIME_F32 && d == EF_D && d_ff == EF_D && gated_mlp && ((H == 2 && (ell == 8 || ell == 16)) || (H == 4 && ell == 8));
}

template <class G>
static lime_status launch_ef(EncodeF32Params p, int B, int64_t total, cudaStream_t st) {
  // Blocks per user: as many as run at once (a block fills an SM; clusters of two fit 148 of them, of four 132), a share of no less than
  // about 50 tokens (a smaller one does not pay for the exchange), at most the eight of a portable cluster; more where the
  // shares would not fit shared memory.
  constexpr int64_t kSmem = 232448, kRow = EF_LD * 4;
  auto fixed_bytes = [](int cl) -> int64_t { return (int64_t)(G::EX + 2 * cl * G::MSG) * 4; };
  static_assert((G::EX + 2 * 2 * G::MSG) * 4 + 128 * EF_LD * 4 <= 232448, "two blocks a user must fit with 128 rows each");
  int cl = 1;
  while (cl < 8 && fixed_bytes(2 * cl) + 128 * kRow <= kSmem &&
         (((int64_t)B * cl * 2 <= 144 && total / ((int64_t)B * cl * 2) >= EF_SHARE) || 2 * total / ((int64_t)B * cl) > (kSmem - fixed_bytes(cl)) / kRow))
    cl *= 2;
  p.B = B;
  p.longer_than = EF_LONG * cl;
  p.total = (int)total;
  p.planned = B >= EF_PLAN_FROM && B <= EF_PLAN_USERS && total >= 2ll * EF_SHARE * B && fixed_bytes(4) + 128 * kRow <= kSmem;
  if (p.planned) cl = 4;
  p.cluster = cl;
  // the host knows the mean length only: room for twice the mean share, 256 rows at least, where shared memory has it
  const int64_t fixed = fixed_bytes(cl), most = (kSmem - fixed) / kRow;
  int64_t cap = 2 * total / ((int64_t)B * cl) + 1;
  if (cap < 256 || p.planned) cap = p.planned ? most : 256;
  if (cap > total) cap = total;
  p.cap = (int)(cap < most ? cap : most);
  auto launch = [&](void (*kernel)(EncodeF32Params), bool (&smem_set)[kMaxDeviceOrdinals], int64_t blocks, int cluster, size_t smem, const EncodeF32Params& q) -> lime_status {
    const lime_status s = ensure_dynamic_smem((const void*)kernel, (int)kSmem, smem_set);
    if (s != LIME_OK) return s;
    if (cluster > 8) LIME_CUDA(cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(EF_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    ProfScope _p("k_encode_f32", st);
    cudaLaunchKernelEx(&cfg, kernel, q);
    LIME_LAUNCH_CHECK("k_encode_f32");
    return LIME_OK;
  };
  // as many clusters of sixteen as the total allows long users, which find theirs or leave; no launch where it allows none
  int64_t longs = total / (p.longer_than + 1);
  if (longs > B) longs = B;
  if (longs > EF_LONG_CLUSTERS) longs = EF_LONG_CLUSTERS;
  p.skip_long = longs > 0;
  if (longs > 0) {
    EncodeF32Params q = p;
    constexpr int64_t long_fixed = (int64_t)(G::EX + G::MSG) * 4;
    q.cap = (int)((kSmem - long_fixed) / kRow);
    static bool long_smem_set[kMaxDeviceOrdinals] = {};
    const lime_status s = launch(k_encode_f32<G, true>, long_smem_set, longs * EF_LONG_CLUSTER, EF_LONG_CLUSTER, (size_t)(long_fixed + q.cap * kRow), q);
    if (s != LIME_OK) return s;
  }
  static bool smem_set[kMaxDeviceOrdinals] = {};
  const int64_t blocks = p.planned ? 4 * (B < EF_PLAN_CLUSTERS ? B : EF_PLAN_CLUSTERS) : (int64_t)B * cl;
  return launch(k_encode_f32<G, false>, smem_set, blocks, cl, (size_t)(fixed + p.cap * kRow), p);
}

lime_status launch_encode_f32(const EncodeSmallArgs& a, int* err, cudaStream_t st) {
  EncodeF32Params p;
  p.hist = (const float*)a.hist; p.off = a.off; p.links = a.links; p.links_per_user = a.links_per_user;
  for (int j = 0; j < a.n_layers; ++j) {
    const void* w[6] = {a.w->Wq[j], a.w->Wk[j], a.w->Wv[j], a.w->Wg[j], a.w->Wu[j], a.w->Wo[j]};
    for (int m = 0; m < 6; ++m) p.w[j][m] = (const float*)w[m];
  }
  p.scratch = (float*)a.scratch; p.out = a.lp; p.n_layers = a.n_layers; p.ln = a.ln; p.hist_ln = a.hist_ln; p.silu = a.silu;
  p.eps = a.eps; p.scale = a.silu ? 1.0f : a.scale * 1.4426950408889634f; p.err = err;
  if (a.H == 4) return launch_ef<EfCfg<4, 8>>(p, a.B, a.total, st);
  return a.ell == 8 ? launch_ef<EfCfg<2, 8>>(p, a.B, a.total, st) : launch_ef<EfCfg<2, 16>>(p, a.B, a.total, st);
}

}  // namespace lime
