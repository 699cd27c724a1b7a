// Candidate scoring through a three-layer interaction network (bf16 storage, d = 32, hidden widths w0 <= 512, 128, 64):
//
//   O_c = sum_l W[c,l] LS_b[l,:]   (Eq. 4),   logit_c = w_3 . relu( relu( relu( [O_c | T_c] W_0 + b_0 ) W_1 + b_1 ) W_2 + b_2 ) + b_3
//
// About 200 k operations per candidate against 100 bytes: bound by the tensor pipe (196 KB of weights stay in shared memory).
// The hidden layers chain through registers: a warp takes 16 or 32 candidates, forms 16 hidden units of the first layer at a
// time (the accumulator becomes the A fragment of the second layer's k-step) and keeps the 128-wide second layer in its
// accumulators, so no activation touches memory.  The pipe is 60 % busy at the rate that mma.sync reaches; on tcgen05 the hidden
// blocks would go through TMEM as A operands, as U does in the history updates (k_hist_update_tmem_tc.cu).  That form has not been built.
// The first layer's input is not folded through the link states: O is formed per candidate (four products), so it needs no per-user
// operand.  O and both hidden layers enter their products as a bf16 value and its bf16 remainder.  Error of the logits against
// fp64 from the same link states (16 links, widths 512, 128, 64, four seeds): 2.0e-6 .. 5.3e-6; rounded once instead, the hidden
// layers put 1.7e-3 .. 3.0e-3 into it (the CUDA-core kernel for other widths: 2.3e-7 .. 5.6e-7; a third piece leaves 0.9e-6 ..
// 2.3e-6, what the tensor cores' sums add, and costs 18 us more).  25,600 candidates on 256 slots a block: 35 us a launch with one
// rounding, 44 with two pieces.
// Weights are read as stored ([in x out], ldmatrix.trans).  Chunk c (16 bytes) of row r sits at c ^ s(r), s(r) = (r & 7) ^
// ((r >> 3 & 3) << 1): free of conflicts both for eight consecutive rows and for the rows 8 i, 8 i + 1 (i = 0..3) that the
// permuted contraction over T needs (thread t of a quad holds features 8 t .. 8 t + 7 of a candidate row: one 16-byte load).
#include "lime_common.cuh"
#include "tc_common.cuh"

namespace lime {

constexpr int M3_D = 32, M3_N1 = 128, M3_N2 = 64;
constexpr int M3_TERMS = 2;      // bf16 pieces of a value that was fp32: the mix, the first and the second hidden layer

struct ScoreMlp3Params {
  const __nv_bfloat16* LS; const __nv_bfloat16* W; const __nv_bfloat16* T;
  const int32_t* cand_off; const int32_t* ids; int32_t* flag; float* logits;
  const __nv_bfloat16 *W0, *W1, *W2, *W3;
  const float *b0, *b1, *b2, *b3;
  int rows, total, B, C, w0, n_groups;      // groups of a warp's slots
};

__device__ __forceinline__ int m3_s(int r) { return (r & 7) ^ (((r >> 3) & 3) << 1); }
__device__ __forceinline__ uint32_t m3_at(int r, int c, int pitch) { return (uint32_t)r * pitch + ((uint32_t)(c ^ m3_s(r)) << 4); }
__device__ __forceinline__ uint32_t m3_pack(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// two fp32 values as M3_TERMS packed bf16 pairs: the values, their remainders
__device__ __forceinline__ void m3_split(float x, float y, uint32_t (&out)[M3_TERMS]) {
#pragma unroll
  for (int k = 0; k < M3_TERMS; ++k) {
    out[k] = m3_pack(x, y);
    x -= __uint_as_float(out[k] << 16);
    y -= __uint_as_float(out[k] & 0xffff0000u);
  }
}
__device__ __forceinline__ void m3_mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void m3_mma8(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ void m3_ldsm_t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}

// shared memory: W_0 [64 x w0], W_1 [w0 x 128], W_2 [128 x 64], the link states a warp works with, biases and w_3
struct M3Layout {
  uint32_t w1, w2, ls, consts, bytes;
  __host__ __device__ M3Layout(int w0, int ell, int warps) {
    w1 = 2 * M3_D * w0 * 2;
    w2 = w1 + w0 * M3_N1 * 2;
    ls = w2 + M3_N1 * M3_N2 * 2;
    consts = ls + warps * ell * M3_D * 2;
    bytes = consts + (w0 + M3_N1 + 2 * M3_N2 + 4) * 4;
  }
};

template <int ELL, int MT, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1)
k_score_mlp3(const ScoreMlp3Params p) {
  constexpr int THREADS = WARPS * 32, SLOTS = 16 * MT;           // candidates a warp scores at a time
  extern __shared__ __align__(128) uint8_t sm[];
  const M3Layout lay(p.w0, ELL, WARPS);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  pdl_launch_dependents();
  pdl_wait();
  const uint32_t sb = (uint32_t)__cvta_generic_to_shared(sm);
  {
    auto copy = [&](uint32_t at, const __nv_bfloat16* src, int rows, int cols) {
      const int cpr = cols / 8;
      for (int i = tid; i < rows * cpr; i += THREADS)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sb + at + m3_at(i / cpr, i % cpr, cols * 2)), "l"(src + (int64_t)i * 8) : "memory");
    };
    copy(0, p.W0, 2 * M3_D, p.w0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    copy(lay.w1, p.W1, p.w0, M3_N1);
    copy(lay.w2, p.W2, M3_N1, M3_N2);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  float* const c0 = reinterpret_cast<float*>(sm + lay.consts);
  float *const c1 = c0 + p.w0, *const c2 = c1 + M3_N1, *const c3 = c2 + M3_N2;
  for (int i = tid; i < p.w0; i += THREADS) c0[i] = p.b0 ? p.b0[i] : 0.f;
  for (int i = tid; i < M3_N1; i += THREADS) c1[i] = p.b1 ? p.b1[i] : 0.f;
  for (int i = tid; i < M3_N2; i += THREADS) { c2[i] = p.b2 ? p.b2[i] : 0.f; c3[i] = __bfloat162float(p.W3[i]); }
  if (tid == 0) c3[M3_N2] = p.b3 ? p.b3[0] : 0.f;

  uint8_t* const ls = sm + lay.ls + warp * (ELL * M3_D * 2);
  const uint32_t ls_a = sb + lay.ls + warp * (ELL * M3_D * 2);
  bool weights_in = false;
  for (int grp = blockIdx.x * WARPS + warp; grp < ((p.n_groups + WARPS - 1) / WARPS) * WARPS; grp += gridDim.x * WARPS) {
    // slots s0 .. s0 + here - 1 (none past the last group; slot numbers go up to 2^31 - 2, so nothing is added to one ahead of a comparison)
    const int s0 = grp < p.n_groups ? grp * SLOTS : p.total, here = min(SLOTS, p.total - s0), s1 = s0 + here;
    const bool work = here > 0;
    int row = lane < here ? s0 + lane : p.total - 1;
    bool good = lane < here;
    if (p.ids != nullptr) {
      const int32_t id = __ldg(p.ids + row);
      if (good && (id < 0 || id >= p.rows) && p.flag != nullptr) atomicMin(p.flag, row);
      good = good && id >= 0 && id < p.rows;
      row = id;
    }
    const unsigned live = __ballot_sync(0xffffffffu, good);
    // candidate rows g, g + 8, (g + 16, g + 24): features 8 t .. of T, links of W
    uint4 tv[2 * MT];
    uint32_t wv[2 * MT][ELL / 8];
#pragma unroll
    for (int i = 0; i < 2 * MT; ++i) {
      const int64_t rr = __shfl_sync(0xffffffffu, row, g + 8 * i);
      const bool on = (live >> (g + 8 * i)) & 1u;
      tv[i] = on ? __ldg(reinterpret_cast<const uint4*>(p.T + rr * M3_D + t * 8)) : make_uint4(0, 0, 0, 0);
      const uint32_t* wp = reinterpret_cast<const uint32_t*>(p.W + rr * ELL) + t;
#pragma unroll
      for (int k = 0; k < ELL / 8; ++k) wv[i][k] = on ? __ldg(wp + 4 * k) : 0u;
    }
    // O = W . LS of each slot's user
    float o[MT][4][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[m][n][e] = 0.f;
    int b = 0;
    if (work) b = p.cand_off == nullptr ? s0 / p.C : upper_user(p.cand_off, p.B, s0);
    while (work) {
      const int u0 = p.cand_off == nullptr ? b * p.C : __ldg(p.cand_off + b);
      const int u1 = p.cand_off == nullptr ? u0 + p.C : __ldg(p.cand_off + b + 1);
      if (u1 > s0) {
        __syncwarp();
        for (int i = lane; i < ELL * 4; i += 32) {
          const int l = i >> 2, c = i & 3;
          *reinterpret_cast<uint4*>(ls + l * 64 + ((c ^ ((l >> 1) & 3)) << 4)) = __ldg(reinterpret_cast<const uint4*>(p.LS + (int64_t)b * ELL * M3_D) + i);
        }
        __syncwarp();
        float q[MT][4][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
          for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) q[m][n][e] = 0.f;
        if constexpr (ELL == 8) {
          uint32_t w[4];
          m3_ldsm_t(w, ls_a + (lane & 7) * 64 + (((lane >> 3) ^ (((lane & 7) >> 1) & 3)) << 4));
#pragma unroll
          for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < 4; ++n) m3_mma8(q[m][n], wv[2 * m][0], wv[2 * m + 1][0], w[n]);
        } else {
#pragma unroll
          for (int ks = 0; ks < ELL / 16; ++ks)
#pragma unroll
            for (int n = 0; n < 4; n += 2) {
              uint32_t w[4];
              const int l = ks * 16 + (lane & 15);
              m3_ldsm_t(w, ls_a + l * 64 + (((n + (lane >> 4)) ^ ((l >> 1) & 3)) << 4));
#pragma unroll
              for (int m = 0; m < MT; ++m) {
                const uint32_t a[4] = {wv[2 * m][2 * ks], wv[2 * m + 1][2 * ks], wv[2 * m][2 * ks + 1], wv[2 * m + 1][2 * ks + 1]};
                m3_mma(q[m][n], a, w[0], w[1]);
                m3_mma(q[m][n + 1], a, w[2], w[3]);
              }
            }
        }
#pragma unroll
        for (int i = 0; i < 2 * MT; ++i) {
          const int slot = g + 8 * i;
          if (slot >= u0 - s0 && slot < u1 - s0)
#pragma unroll
            for (int n = 0; n < 4; ++n) { o[i >> 1][n][(i & 1) * 2] = q[i >> 1][n][(i & 1) * 2]; o[i >> 1][n][(i & 1) * 2 + 1] = q[i >> 1][n][(i & 1) * 2 + 1]; }
        }
      }
      if (u1 >= s1 || b + 1 >= p.B) break;
      ++b;
    }
    // O as A fragments
    uint32_t of[M3_TERMS][MT][2][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int ks = 0; ks < 2; ++ks)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          uint32_t v[M3_TERMS];
          m3_split(o[m][2 * ks + (r >> 1)][(r & 1) * 2], o[m][2 * ks + (r >> 1)][(r & 1) * 2 + 1], v);
#pragma unroll
          for (int k = 0; k < M3_TERMS; ++k) of[k][m][ks][r] = v[k];
        }
    if (!weights_in) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      weights_in = true;
    }
    if (!work) continue;
    // first two layers, 16 units of the first at a time
    float acc[MT][M3_N1 / 8][4];
#pragma unroll
    for (int n = 0; n < M3_N1 / 8; ++n) {
      const float2 bias = *reinterpret_cast<const float2*>(c1 + n * 8 + 2 * t);
#pragma unroll
      for (int m = 0; m < MT; ++m) { acc[m][n][0] = acc[m][n][2] = bias.x; acc[m][n][1] = acc[m][n][3] = bias.y; }
    }
    const int pitch0 = p.w0 * 2;
#pragma unroll 1
    for (int hb = 0; hb < p.w0 / 16; ++hb) {
      float h[MT][2][4];
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const float2 bias = *reinterpret_cast<const float2*>(c0 + hb * 16 + n * 8 + 2 * t);
#pragma unroll
        for (int m = 0; m < MT; ++m) { h[m][n][0] = h[m][n][2] = bias.x; h[m][n][1] = h[m][n][3] = bias.y; }
      }
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) {
        uint32_t w[4];
        m3_ldsm_t(w, sb + m3_at(ks * 16 + (lane & 15), 2 * hb + (lane >> 4), pitch0));
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
          for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int k = 0; k < M3_TERMS; ++k) m3_mma(h[m][n], of[k][m][ks], w[2 * n], w[2 * n + 1]);
      }
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        uint32_t w[4];
        const int i = lane & 7, which = (lane >> 3) & 1;
        m3_ldsm_t(w, sb + m3_at(M3_D + (i >> 1) * 8 + (i & 1) + 4 * s + 2 * which, 2 * hb + (lane >> 4), pitch0));
#pragma unroll
        for (int m = 0; m < MT; ++m) {
          const uint32_t a[4] = {s ? tv[2 * m].z : tv[2 * m].x, s ? tv[2 * m + 1].z : tv[2 * m + 1].x, s ? tv[2 * m].w : tv[2 * m].y,
                                 s ? tv[2 * m + 1].w : tv[2 * m + 1].y};
#pragma unroll
          for (int n = 0; n < 2; ++n) m3_mma(h[m][n], a, w[2 * n], w[2 * n + 1]);
        }
      }
      uint32_t a[M3_TERMS][MT][4];
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          uint32_t v[M3_TERMS];
          m3_split(fmaxf(h[m][r >> 1][(r & 1) * 2], 0.f), fmaxf(h[m][r >> 1][(r & 1) * 2 + 1], 0.f), v);
#pragma unroll
          for (int k = 0; k < M3_TERMS; ++k) a[k][m][r] = v[k];
        }
#pragma unroll
      for (int n = 0; n < M3_N1 / 8; n += 2) {
        uint32_t w[4];
        m3_ldsm_t(w, sb + lay.w1 + m3_at(hb * 16 + (lane & 15), n + (lane >> 4), M3_N1 * 2));
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
          for (int k = 0; k < M3_TERMS; ++k) { m3_mma(acc[m][n], a[k][m], w[0], w[1]); m3_mma(acc[m][n + 1], a[k][m], w[2], w[3]); }
      }
    }
    // third layer
    float z[MT][M3_N2 / 8][4];
#pragma unroll
    for (int n = 0; n < M3_N2 / 8; ++n) {
      const float2 bias = *reinterpret_cast<const float2*>(c2 + n * 8 + 2 * t);
#pragma unroll
      for (int m = 0; m < MT; ++m) { z[m][n][0] = z[m][n][2] = bias.x; z[m][n][1] = z[m][n][3] = bias.y; }
    }
#pragma unroll
    for (int ks = 0; ks < M3_N1 / 16; ++ks) {
      uint32_t a[M3_TERMS][MT][4];
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          uint32_t v[M3_TERMS];
          m3_split(fmaxf(acc[m][2 * ks + (r >> 1)][(r & 1) * 2], 0.f), fmaxf(acc[m][2 * ks + (r >> 1)][(r & 1) * 2 + 1], 0.f), v);
#pragma unroll
          for (int k = 0; k < M3_TERMS; ++k) a[k][m][r] = v[k];
        }
#pragma unroll
      for (int n = 0; n < M3_N2 / 8; n += 2) {
        uint32_t w[4];
        m3_ldsm_t(w, sb + lay.w2 + m3_at(ks * 16 + (lane & 15), n + (lane >> 4), M3_N2 * 2));
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
          for (int k = 0; k < M3_TERMS; ++k) { m3_mma(z[m][n], a[k][m], w[0], w[1]); m3_mma(z[m][n + 1], a[k][m], w[2], w[3]); }
      }
    }
    // output layer: rows g, g + 8 (values 0-1, 2-3) of each half
    float v[2 * MT];
#pragma unroll
    for (int i = 0; i < 2 * MT; ++i) v[i] = 0.f;
#pragma unroll
    for (int n = 0; n < M3_N2 / 8; ++n) {
      const float2 w = *reinterpret_cast<const float2*>(c3 + n * 8 + 2 * t);
#pragma unroll
      for (int i = 0; i < 2 * MT; ++i) {
        v[i] = fmaf(fmaxf(z[i >> 1][n][(i & 1) * 2], 0.f), w.x, v[i]);
        v[i] = fmaf(fmaxf(z[i >> 1][n][(i & 1) * 2 + 1], 0.f), w.y, v[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < 2 * MT; ++i) {
      v[i] += __shfl_xor_sync(0xffffffffu, v[i], 1);
      v[i] += __shfl_xor_sync(0xffffffffu, v[i], 2);
    }
    const int r = g + 8 * t;                                     // lane (g, t) writes row g + 8 t
    float mine = v[0];
#pragma unroll
    for (int i = 1; i < 2 * MT; ++i) mine = t == i ? v[i] : mine;
    mine += c3[M3_N2];
    if (r < here) p.logits[s0 + r] = ((live >> r) & 1u) ? mine : 0.f;
  }
}

bool score_mlp3_supported(const ScoreArgs& a, const lime_ffn& f) {
  if (a.dtype != LIME_BF16 || a.d != M3_D || !(a.ell == 8 || a.ell == 16 || a.ell == 32) || a.ldt || a.ldw) return false;
  if (f.n_hidden != 3 || f.widths[0] % 64 || f.widths[0] > 512 || f.widths[1] != M3_N1 || f.widths[2] != M3_N2) return false;
  if (a.cand_off == nullptr && a.C <= 0) return false;
  return M3Layout(f.widths[0], a.ell, 8).bytes <= 232448;
}

template <int ELL, int MT, int WARPS>
static lime_status launch_m3(ScoreMlp3Params p, cudaStream_t st) {
  const M3Layout lay(p.w0, ELL, WARPS);
  static bool smem_set[kMaxDeviceOrdinals] = {};
  lime_status s = ensure_dynamic_smem((const void*)k_score_mlp3<ELL, MT, WARPS>, 232448, smem_set);
  if (s != LIME_OK) return s;
  p.n_groups = (int)(((int64_t)p.total + 16 * MT - 1) / (16 * MT));
  const int blocks = (p.n_groups + WARPS - 1) / WARPS;
  ProfScope _p("k_score_mlp3", st);
  launch_pdl(k_score_mlp3<ELL, MT, WARPS>, dim3((unsigned)(blocks < kSMs ? blocks : kSMs)), dim3(WARPS * 32), (size_t)lay.bytes, st, p);
  LIME_LAUNCH_CHECK("k_score_mlp3");
  return LIME_OK;
}

// A block takes 128, 192 or 256 slots at a time: a round of the grid costs 18.4, 27.2 or 35 us (16 links, widths 512, 128, 64; the
// whole call 23.5, 32.4 and 39.6 with one), so what counts is how full the last round is.  25,600 candidates 40.2 -> 32.4 us,
// 12,800 39.0 -> 23.6, 45,000 74.4 -> 59.9, 200,000 211.9 -> 205.9 against 256 slots whatever their number.  Other shapes take less a round,
// in nearly the same proportion: with 8, 16 or 32 links, a first width of 64 to 512 and 1000 to 200,000 candidates the shape chosen is
// within 2 % of the best of the three but for first widths of 64 from 120,000 candidates on (4 %).
template <int ELL>
static lime_status launch_m3_shape(const ScoreMlp3Params& p, cudaStream_t st) {
  auto rounds = [&](int slots) { return (double)((p.total + (int64_t)slots * kSMs - 1) / ((int64_t)slots * kSMs)); };
  const double t128 = 18.4 * rounds(128), t256 = 35.0 * rounds(256);
  const double t192 = M3Layout(p.w0, ELL, 12).bytes <= 232448 ? 27.2 * rounds(192) : 1e30;
  if (t128 <= t192 && t128 <= t256) return launch_m3<ELL, 1, 8>(p, st);
  return t192 <= t256 ? launch_m3<ELL, 1, 12>(p, st) : launch_m3<ELL, 2, 8>(p, st);
}

lime_status launch_score_mlp3(const ScoreArgs& a, const lime_ffn& f, cudaStream_t st) {
  ScoreMlp3Params p;
  p.LS = (const __nv_bfloat16*)a.LS; p.W = (const __nv_bfloat16*)a.W; p.T = (const __nv_bfloat16*)a.T;
  p.cand_off = a.cand_off; p.ids = a.cand_ids; p.flag = a.dev_flag; p.logits = a.logits;
  p.W0 = (const __nv_bfloat16*)f.W[0]; p.W1 = (const __nv_bfloat16*)f.W[1]; p.W2 = (const __nv_bfloat16*)f.W[2]; p.W3 = (const __nv_bfloat16*)f.W[3];
  p.b0 = f.b[0]; p.b1 = f.b[1]; p.b2 = f.b[2]; p.b3 = f.b[3];
  p.rows = (int)(a.cand_ids ? a.corpus_rows : a.total); p.total = (int)a.total; p.B = a.B; p.C = a.C; p.w0 = f.widths[0];
  if (a.ell == 8) return launch_m3_shape<8>(p, st);
  if (a.ell == 16) return launch_m3_shape<16>(p, st);
  return launch_m3_shape<32>(p, st);
}

}  // namespace lime
