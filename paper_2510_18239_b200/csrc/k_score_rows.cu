// Candidate scoring with every warp on its own (Eq. 4, bf16 storage): candidates by id from the corpus caches, ragged
// candidate lists, and widths the streaming scorers are not built for.
//
//   logit[i] = < sum_l W[r, l] LS_b[l, :], T[r, :] >,   r = cand_ids[i] (or i), b = user of slot i
//
// What bounds it: the rate at which HBM serves random rows.  Rows by id arrive in pieces of 2 d and 2 ell bytes; the
// memory system opens about 16.5 G different 256-byte blocks a second whatever fetches them, so the kernel's part is to
// keep enough rows in flight and to add no latency of its own.  A warp takes 16 consecutive slots, reads its rows from
// global memory straight into the A fragments of mma.m16n8k16 (no shared memory, no barrier, no tensor memory to allocate:
// the first row is requested two dependent reads after the launch) and forms A = T_rows . LS^T; the ell-term dot with the
// weight row follows in registers.  The tensor work (2 ell d per candidate against 2 d + 2 ell bytes) is far below what
// mma.sync sustains, so the tcgen05 pipeline would only add set-up.  Two permutations make every access wide:
//   - of the contraction index: thread t of a quad holds columns (4 j + t) * 8 .. + 7 of a row for j = 0, 1, .. (one 16-byte
//     load gives the fragments of two k-steps); the link states are read with the same permutation;
//   - of the links: thread t owns links t * ell / 4 .. of the accumulator row, so its weights are one 8- to 32-byte piece.
// The link states come through L1: the warps of a block work on neighbouring slots, nearly always of one user.
#include "lime_common.cuh"

namespace lime {

constexpr int SR_WARPS = 4;
constexpr int SR_AHEAD = 4;      // groups of slots a warp asks L2 for before it may read the link states
// blocks an SM can hold: what a thread keeps of its rows (d / 16 words each of two), weights and accumulators sets the
// registers it needs, and the rest goes into warps
constexpr int sr_blocks(int d, int ell) { return d * ell >= 8192 ? (d == 256 && ell == 64 ? 2 : 3) : 4; }

struct ScoreRowsParams {
  const __nv_bfloat16* LS; const __nv_bfloat16* W; const __nv_bfloat16* T;
  const int32_t* cand_off; const int32_t* ids;     // both nullable
  int32_t* flag;
  float* logits;
  int ldt, ldw;            // row pitches in elements
  int rows;                // rows of W and T
  int total;               // slots
  int B, C, n_groups;      // groups of 16 slots (8 with fp32 storage)
};

__device__ __forceinline__ uint4 sr_ld_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
// link-state pieces: kept in L1, and not moved ahead of the products of the previous chunk (all of them in flight at once
// would not leave room for the candidate rows in the registers)
__device__ __forceinline__ uint4 sr_ld_keep(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ void sr_mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// user of slot `s`: the largest b with off[b] <= s (users without candidates are skipped by taking the largest), found by
// the warp together: every step narrows the range 32-fold
__device__ __forceinline__ int sr_find_user(const int32_t* __restrict__ off, int B, int s, int lane) {
  int lo = 0, hi = B;                             // off[lo] <= s, answer in [lo, hi)
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) / 32;
    const int at = lo + (lane + 1) * step;        // lane's pivot
    const unsigned le = __ballot_sync(0xffffffffu, at < hi && __ldg(off + min(at, B)) <= s);
    const int k = __popc(le);                     // pivots are increasing: the first k lie at or below s
    hi = min(hi, lo + (k + 1) * step);
    lo += k * step;
  }
  return lo;
}

template <int D, int ELL>
__global__ void __launch_bounds__(SR_WARPS * 32, sr_blocks(D, ELL))
k_score_rows(const ScoreRowsParams p) {
  constexpr int NT = ELL / 8, NL = ELL / 4, KJ = D / 32;    // n-tiles, links per thread, 32-column chunks
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int g_begin = (int)(((int64_t)blockIdx.x * p.n_groups) / gridDim.x);
  const int g_end = (int)(((int64_t)(blockIdx.x + 1) * p.n_groups) / gridDim.x);
  // What the block waits for is the link states (and the list offsets): its first rows move into L2 meanwhile, two lanes per
  // slot taking every other line of the row (memory is idle while the last link-side kernel runs on a few SMs, and all blocks of
  // this kernel fit beside it: 100 lists of 20..1500 ids, the batch 142 -> 134 us.  The tcgen05 scorers do not gain: their CTAs
  // take a whole SM, so those that wait for one of the busy SMs start late whatever the others have prefetched)
  for (int grp = g_begin + warp; grp < min(g_end, g_begin + SR_AHEAD * SR_WARPS); grp += SR_WARPS) {
    const int s0 = grp * 16;
    const bool in = (lane & 15) < p.total - s0;    // (not s0 + lane < total: slot numbers go up to 2^31 - 2)
    const int slot = in ? s0 + (lane & 15) : 0;
    const int id = in ? (p.ids != nullptr ? __ldcg(p.ids + slot) : slot) : -1;
    if (id >= 0 && id < p.rows) {
      const char* row = reinterpret_cast<const char*>(p.T + (int64_t)id * p.ldt);
      for (int o = (lane >> 4) * 128; o < D * 2; o += 256) prefetch_l2(row + o);
      if (lane < 16) prefetch_l2_row(p.W + (int64_t)id * p.ldw, ELL * 2);
    }
  }
  pdl_wait();
  int b = -1;
  for (int grp = g_begin + warp; grp < g_end; grp += SR_WARPS) {
    const int s0 = grp * 16;
    const int here = min(16, p.total - s0), s1 = s0 + here;
    // one row index per slot
    bool in = lane < here;
    int row = in ? s0 + lane : s0;
    if (p.ids != nullptr) {
      const int32_t id = in ? __ldg(p.ids + row) : 0;
      const bool good = id >= 0 && id < p.rows;
      if (in && !good && p.flag != nullptr) atomicMin(p.flag, row);
      in = in && good;
      row = id;
    }
    const unsigned live = __ballot_sync(0xffffffffu, in);
    // T rows as A fragments (all chunks requested at once), weight pieces
    uint4 a[2][KJ];
    uint32_t w[2][NL / 2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = g + 8 * i;
      const int rr = __shfl_sync(0xffffffffu, row, r);
      const bool on = (live >> r) & 1u;
      const __nv_bfloat16* tp = p.T + (int64_t)rr * p.ldt + t * 8;
#pragma unroll
      for (int j = 0; j < KJ; ++j) a[i][j] = on ? sr_ld_stream(tp + j * 32) : make_uint4(0, 0, 0, 0);
      const __nv_bfloat16* wp = p.W + (int64_t)rr * p.ldw + t * NL;
      if constexpr (NL >= 8) {
#pragma unroll
        for (int k = 0; k < NL / 8; ++k) {
          const uint4 v = on ? sr_ld_stream(wp + k * 8) : make_uint4(0, 0, 0, 0);
          w[i][4 * k] = v.x; w[i][4 * k + 1] = v.y; w[i][4 * k + 2] = v.z; w[i][4 * k + 3] = v.w;
        }
      } else if constexpr (NL == 4) {
        const uint2 v = on ? __ldg(reinterpret_cast<const uint2*>(wp)) : make_uint2(0, 0);
        w[i][0] = v.x; w[i][1] = v.y;
      } else {
        w[i][0] = on ? __ldg(reinterpret_cast<const uint32_t*>(wp)) : 0u;
      }
    }
    // the users these slots belong to (one, but for groups across a boundary)
    if (p.cand_off == nullptr) b = s0 / p.C;
    else if (b < 0) b = sr_find_user(p.cand_off, p.B, s0, lane);
    float out = 0.f;
    for (;;) {
      const int u_end = p.cand_off == nullptr ? (b + 1) * p.C : __ldg(p.cand_off + b + 1);
      if (u_end > s0) {
        float acc[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
        const __nv_bfloat16* ls = p.LS + (int64_t)b * (ELL * D) + (int64_t)((g >> 1) * NL + (g & 1)) * D + t * 8;
#pragma unroll
        for (int j = 0; j < KJ; ++j) {
          constexpr int NB = NT < 4 ? NT : 4;
#pragma unroll
          for (int n0 = 0; n0 < NT; n0 += NB) {
            uint4 bf[NB];
#pragma unroll
            for (int n = 0; n < NB; ++n) bf[n] = sr_ld_keep(ls + (2 * (n0 + n)) * D + j * 32);
#pragma unroll
            for (int n = 0; n < NB; ++n) {
              sr_mma(acc[n0 + n], a[0][j].x, a[1][j].x, a[0][j].y, a[1][j].y, bf[n].x, bf[n].y);
              sr_mma(acc[n0 + n], a[0][j].z, a[1][j].z, a[0][j].w, a[1][j].w, bf[n].z, bf[n].w);
            }
          }
        }
        // dot with the weights: links t * NL + 2 n + {0, 1} of rows g (c0, c1) and g + 8 (c2, c3)
        float v[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          float s = 0.f;
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            const uint32_t u = w[i][n];
            s = fmaf(__uint_as_float(u << 16), acc[n][i * 2], s);
            s = fmaf(__uint_as_float(u & 0xffff0000u), acc[n][i * 2 + 1], s);
          }
          s += __shfl_xor_sync(0xffffffffu, s, 1);
          s += __shfl_xor_sync(0xffffffffu, s, 2);
          v[i] = s;
        }
        // lanes t = 0, 1 keep row g + 8 t
        const float mine = t == 0 ? v[0] : v[1];
        const int u_begin = p.cand_off == nullptr ? b * p.C : __ldg(p.cand_off + b);
        if (g + 8 * t >= u_begin - s0 && g + 8 * t < u_end - s0) out = mine;
      }
      if (u_end >= s1 || b + 1 >= p.B) break;
      ++b;
    }
    if (g + 8 * t < here) p.logits[s0 + g + 8 * t] = out;       // here <= 16: threads t = 0, 1
  }
}

// ----------------------------------------------------------------------------- fp32 storage
// A quad per candidate: lane t holds columns (4 i + t) * 4 .. of its row (64 contiguous bytes a load) and the same columns of the
// user's link states in registers, which stay there for all candidates of the user a warp works through.
template <int D, int ELL>
__global__ void __launch_bounds__(SR_WARPS * 32, 2)
k_score_rows_f32(const float* __restrict__ LS, const float* __restrict__ W, const float* __restrict__ T, const ScoreRowsParams p) {
  constexpr int KI = D / 16;
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  // contiguous groups per warp: neighbouring groups share a user
  const int64_t w0 = (int64_t)blockIdx.x * SR_WARPS + warp, nw = (int64_t)gridDim.x * SR_WARPS;
  const int g_begin = (int)(w0 * p.n_groups / nw), g_end = (int)((w0 + 1) * p.n_groups / nw);
  pdl_wait();
  float4 ls[ELL][KI];
  int b = -1, loaded = -1;
  for (int grp = g_begin; grp < g_end; ++grp) {
    const int s0 = grp * 8, here = min(8, p.total - s0), s1 = s0 + here;
    bool in = g < here;
    const int slot = in ? s0 + g : p.total - 1;
    int row = slot;
    if (p.ids != nullptr) {
      const int32_t id = __ldg(p.ids + row);
      const bool good = id >= 0 && id < p.rows;
      if (in && !good && t == 0 && p.flag != nullptr) atomicMin(p.flag, row);
      in = in && good;
      row = in ? id : 0;
    }
    float4 x[KI], w[ELL / 4];
#pragma unroll
    for (int i = 0; i < KI; ++i) x[i] = in ? __ldg(reinterpret_cast<const float4*>(T + (int64_t)row * p.ldt) + 4 * i + t) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < ELL / 4; ++i) w[i] = in ? __ldg(reinterpret_cast<const float4*>(W + (int64_t)row * p.ldw) + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    if (p.cand_off == nullptr) b = s0 / p.C;
    else if (b < 0) b = sr_find_user(p.cand_off, p.B, s0, lane);
    float out = 0.f;
    for (;;) {
      const int u0 = p.cand_off == nullptr ? b * p.C : __ldg(p.cand_off + b), u1 = p.cand_off == nullptr ? u0 + p.C : __ldg(p.cand_off + b + 1);
      if (u1 > s0) {
        if (b != loaded) {
          const float4* src = reinterpret_cast<const float4*>(LS + (int64_t)b * ELL * D) + t;
#pragma unroll
          for (int l = 0; l < ELL; ++l)
#pragma unroll
            for (int i = 0; i < KI; ++i) ls[l][i] = __ldg(src + l * (D / 4) + 4 * i);
          loaded = b;
        }
        float s = 0.f;
#pragma unroll
        for (int l = 0; l < ELL; ++l) {
          float q = 0.f;
#pragma unroll
          for (int i = 0; i < KI; ++i) {
            q = fmaf(ls[l][i].x, x[i].x, q); q = fmaf(ls[l][i].y, x[i].y, q); q = fmaf(ls[l][i].z, x[i].z, q); q = fmaf(ls[l][i].w, x[i].w, q);
          }
          const float4 w4 = w[l / 4];
          s = fmaf(l % 4 == 0 ? w4.x : l % 4 == 1 ? w4.y : l % 4 == 2 ? w4.z : w4.w, q, s);
        }
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (g >= u0 - s0 && g < u1 - s0) out = s;
      }
      if (u1 >= s1 || b + 1 >= p.B) break;
      ++b;
    }
    if (t == 0 && g < here) p.logits[slot] = out;
  }
}

// ----------------------------------------------------------------------------- candidate -> link weights, narrow models
// out[m, :] = softmax_l <T_m, keff_l>, every warp on its own as above.  bf16: 16 rows a step as A fragments, the keys as a
// bf16 value and its remainder (keff_hl, [2 ell x d]) in B fragments that stay in registers.
template <int D, int ELL>
__global__ void __launch_bounds__(SR_WARPS * 32)
k_precompute_rows(const __nv_bfloat16* __restrict__ T, int64_t M, const __nv_bfloat16* __restrict__ keff_hl, __nv_bfloat16* __restrict__ out) {
  constexpr int NT = ELL / 8, NL = ELL / 4, KJ = D / 32;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  uint4 kf[2][NT][KJ];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int j = 0; j < KJ; ++j)
        kf[h][n][j] = __ldg(reinterpret_cast<const uint4*>(keff_hl + (int64_t)(h * ELL + (g >> 1) * NL + 2 * n + (g & 1)) * D + j * 32 + t * 8));
  const int64_t groups = (M + 15) / 16, stride = (int64_t)gridDim.x * SR_WARPS;
  for (int64_t grp = (int64_t)blockIdx.x * SR_WARPS + (threadIdx.x >> 5); grp < groups; grp += stride) {
    const int64_t m0 = grp * 16 + g;
    uint4 a[2][KJ];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < KJ; ++j) a[i][j] = m0 + 8 * i < M ? sr_ld_stream(T + (m0 + 8 * i) * D + j * 32 + t * 8) : make_uint4(0, 0, 0, 0);
    float acc[NT][4];
#pragma unroll
    for (int n = 0; n < NT; ++n) {
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int j = 0; j < KJ; ++j) {
          sr_mma(acc[n], a[0][j].x, a[1][j].x, a[0][j].y, a[1][j].y, kf[h][n][j].x, kf[h][n][j].y);
          sr_mma(acc[n], a[0][j].z, a[1][j].z, a[0][j].w, a[1][j].w, kf[h][n][j].z, kf[h][n][j].w);
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {                                 // rows g, g + 8: this thread's links t * NL ..
      float mx = -INFINITY, sum = 0.f;
#pragma unroll
      for (int n = 0; n < NT; ++n) mx = fmaxf(mx, fmaxf(acc[n][2 * i], acc[n][2 * i + 1]));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        acc[n][2 * i] = __expf(acc[n][2 * i] - mx); acc[n][2 * i + 1] = __expf(acc[n][2 * i + 1] - mx);
        sum += acc[n][2 * i] + acc[n][2 * i + 1];
      }
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      const float inv = 1.0f / sum;
      if (m0 + 8 * i < M) {
        uint32_t o[NT];
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const __nv_bfloat162 v = __floats2bfloat162_rn(acc[n][2 * i] * inv, acc[n][2 * i + 1] * inv);
          o[n] = *reinterpret_cast<const uint32_t*>(&v);
        }
        __nv_bfloat16* dst = out + (m0 + 8 * i) * ELL + t * NL;
        if constexpr (NT == 1) *reinterpret_cast<uint32_t*>(dst) = o[0];
        else if constexpr (NT == 2) *reinterpret_cast<uint2*>(dst) = make_uint2(o[0], o[1]);
        else
#pragma unroll
          for (int n = 0; n < NT; n += 4) *reinterpret_cast<uint4*>(dst + 2 * n) = make_uint4(o[n], o[n + 1], o[n + 2], o[n + 3]);
      }
    }
  }
}

// fp32: a quad per row, the keys' columns of a lane in registers
template <int D, int ELL>
__global__ void __launch_bounds__(SR_WARPS * 32, 2)
k_precompute_rows_f32(const float* __restrict__ T, int64_t M, const float* __restrict__ keff, float* __restrict__ out) {
  constexpr int KI = D / 16, NL = ELL / 4;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  float4 kf[ELL][KI];
#pragma unroll
  for (int l = 0; l < ELL; ++l)
#pragma unroll
    for (int i = 0; i < KI; ++i) kf[l][i] = __ldg(reinterpret_cast<const float4*>(keff + l * D) + 4 * i + t);
  const int64_t groups = (M + 7) / 8, stride = (int64_t)gridDim.x * SR_WARPS;
  // the next step's rows are requested before this one's products
  auto load = [&](float4 (&x)[KI], int64_t grp) {
    const int64_t m = grp * 8 + g;
#pragma unroll
    for (int i = 0; i < KI; ++i) x[i] = m < M ? __ldg(reinterpret_cast<const float4*>(T + m * D) + 4 * i + t) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  float4 x[KI], nx[KI], nx2[KI];
  int64_t grp = (int64_t)blockIdx.x * SR_WARPS + (threadIdx.x >> 5);
  load(nx, grp);
  load(nx2, grp + stride);
  for (; grp < groups; grp += stride) {
    const int64_t m = grp * 8 + g;
#pragma unroll
    for (int i = 0; i < KI; ++i) { x[i] = nx[i]; nx[i] = nx2[i]; }
    load(nx2, grp + 2 * stride);
    float s[ELL], mx = -INFINITY, sum = 0.f;
#pragma unroll
    for (int l = 0; l < ELL; ++l) {
      s[l] = 0.f;
#pragma unroll
      for (int i = 0; i < KI; ++i) {
        s[l] = fmaf(kf[l][i].x, x[i].x, s[l]); s[l] = fmaf(kf[l][i].y, x[i].y, s[l]); s[l] = fmaf(kf[l][i].z, x[i].z, s[l]); s[l] = fmaf(kf[l][i].w, x[i].w, s[l]);
      }
      s[l] += __shfl_xor_sync(0xffffffffu, s[l], 1);
      s[l] += __shfl_xor_sync(0xffffffffu, s[l], 2);
      mx = fmaxf(mx, s[l]);
    }
#pragma unroll
    for (int l = 0; l < ELL; ++l) { s[l] = __expf(s[l] - mx); sum += s[l]; }
    const float inv = 1.0f / sum;
    if (m < M)
#pragma unroll
      for (int k = 0; k < NL; k += 2) {                           // lane t writes links t * NL ..
        float a = s[k], bq = s[k + 1];
#pragma unroll
        for (int q = 1; q < 4; ++q) { a = t == q ? s[q * NL + k] : a; bq = t == q ? s[q * NL + k + 1] : bq; }
        *reinterpret_cast<float2*>(out + m * ELL + t * NL + k) = make_float2(a * inv, bq * inv);
      }
  }
}

bool precompute_rows_supported(int dtype, int d, int rows, int group) {
  if (rows != group) return false;                                // one softmax per row
  if (dtype == LIME_F32) return (d == 64 && rows == 8) || (d == 32 && (rows == 8 || rows == 16));
  return d == 32 && (rows == 8 || rows == 16 || rows == 32);
}

lime_status launch_precompute_rows(int dtype, const void* cand, int64_t M, int d, int ell, const float* keff, const void* keff_hl, void* out_w,
                                   cudaStream_t st) {
  if (M == 0) return LIME_OK;
  const int64_t blocks = (M / (dtype == LIME_F32 ? 8 : 16) + SR_WARPS) / SR_WARPS, cap = (int64_t)kSMs * (dtype == LIME_F32 ? 3 : 8);
  const dim3 grid((unsigned)(blocks < cap ? blocks : cap)), block(SR_WARPS * 32);
  ProfScope _p("k_precompute_rows", st);
  if (dtype == LIME_F32) {
    const float* T = (const float*)cand;
    float* o = (float*)out_w;
    if (d == 64) k_precompute_rows_f32<64, 8><<<grid, block, 0, st>>>(T, M, keff, o);
    else if (ell == 8) k_precompute_rows_f32<32, 8><<<grid, block, 0, st>>>(T, M, keff, o);
    else k_precompute_rows_f32<32, 16><<<grid, block, 0, st>>>(T, M, keff, o);
  } else {
    const __nv_bfloat16 *T = (const __nv_bfloat16*)cand, *k = (const __nv_bfloat16*)keff_hl;
    __nv_bfloat16* o = (__nv_bfloat16*)out_w;
    if (ell == 8) k_precompute_rows<32, 8><<<grid, block, 0, st>>>(T, M, k, o);
    else if (ell == 16) k_precompute_rows<32, 16><<<grid, block, 0, st>>>(T, M, k, o);
    else k_precompute_rows<32, 32><<<grid, block, 0, st>>>(T, M, k, o);
  }
  LIME_LAUNCH_CHECK("k_precompute_rows");
  return LIME_OK;
}

// ----------------------------------------------------------------------------- dispatch
static bool score_rows_supported(const ScoreArgs& a) {
  if (a.cand_off == nullptr && a.C <= 0) return false;
  if (a.dtype == LIME_F32) {
    if (!((a.d == 64 && a.ell == 8) || (a.d == 32 && (a.ell == 8 || a.ell == 16)))) return false;
    return ((reinterpret_cast<uintptr_t>(a.T) | reinterpret_cast<uintptr_t>(a.W) | reinterpret_cast<uintptr_t>(a.LS)) & 15) == 0 && a.ldt % 4 == 0 && a.ldw % 4 == 0;
  }
  const bool d_ok = a.d == 32 || a.d == 64 || a.d == 128 || a.d == 256;
  const bool l_ok = a.ell == 8 || a.ell == 16 || a.ell == 32 || a.ell == 64;
  if (!d_ok || !l_ok) return false;
  const int64_t ldt = a.ldt ? a.ldt : a.d, ldw = a.ldw ? a.ldw : a.ell;
  // 16-byte pieces of T rows; weight pieces of ell / 2 bytes, at most 16
  return (reinterpret_cast<uintptr_t>(a.T) & 15) == 0 && ldt % 8 == 0 && (reinterpret_cast<uintptr_t>(a.W) & 15) == 0 && ldw % 8 == 0 &&
         (reinterpret_cast<uintptr_t>(a.LS) & 15) == 0;
}

// Which candidates it takes.  Ragged lists always (no other tensor-core scorer serves them).  Fixed C by id: up to 32768
// slots, where the set-up of the copy pipeline (k_score_gather_tc.cu) costs more than the rows (333 slots: 2 against 6 us);
// beyond that the pipeline keeps more rows in flight (8.4 M slots at d = 256, ell = 64: 1.51 against 1.92 ms).
bool score_rows_preferred(const ScoreArgs& a) {
  if (!score_rows_supported(a)) return false;
  return a.cand_off != nullptr || a.total <= 32768 || !(score_tc_supported(a) || score_gather_tc_supported(a));
}

template <int D, int ELL>
static lime_status launch_score_rows_t(const ScoreArgs& a, cudaStream_t st) {
  ScoreRowsParams p;
  p.LS = (const __nv_bfloat16*)a.LS; p.W = (const __nv_bfloat16*)a.W; p.T = (const __nv_bfloat16*)a.T;
  p.cand_off = a.cand_off; p.ids = a.cand_ids; p.flag = a.dev_flag; p.logits = a.logits;
  p.ldt = a.ldt ? (int)a.ldt : D; p.ldw = a.ldw ? (int)a.ldw : ELL;
  p.rows = (int)(a.cand_ids ? a.corpus_rows : a.total); p.total = (int)a.total; p.B = a.B; p.C = a.C;
  p.n_groups = (int)((a.total + 15) / 16);
  const int64_t blocks = (p.n_groups + SR_WARPS - 1) / SR_WARPS, cap = 2 * kSMs;
  ProfScope _p("k_score_rows", st);
  launch_pdl(k_score_rows<D, ELL>, dim3((unsigned)(blocks < cap ? blocks : cap)), dim3(SR_WARPS * 32), 0, st, p);
  LIME_LAUNCH_CHECK("k_score_rows");
  return LIME_OK;
}

template <int D>
static lime_status launch_score_rows_d(const ScoreArgs& a, cudaStream_t st) {
  switch (a.ell) {
    case 8: return launch_score_rows_t<D, 8>(a, st);
    case 16: return launch_score_rows_t<D, 16>(a, st);
    case 32: return launch_score_rows_t<D, 32>(a, st);
    default: return launch_score_rows_t<D, 64>(a, st);
  }
}

template <int D, int ELL>
static lime_status launch_score_rows_f32_t(const ScoreArgs& a, cudaStream_t st) {
  ScoreRowsParams p{};
  p.cand_off = a.cand_off; p.ids = a.cand_ids; p.flag = a.dev_flag; p.logits = a.logits;
  p.ldt = a.ldt ? (int)a.ldt : D; p.ldw = a.ldw ? (int)a.ldw : ELL;
  p.rows = (int)(a.cand_ids ? a.corpus_rows : a.total); p.total = (int)a.total; p.B = a.B; p.C = a.C;
  p.n_groups = (int)((a.total + 7) / 8);
  const int64_t blocks = (p.n_groups + SR_WARPS - 1) / SR_WARPS, cap = 3 * kSMs;
  ProfScope _p("k_score_rows", st);
  launch_pdl(k_score_rows_f32<D, ELL>, dim3((unsigned)(blocks < cap ? blocks : cap)), dim3(SR_WARPS * 32), 0, st, (const float*)a.LS,
             (const float*)a.W, (const float*)a.T, p);
  LIME_LAUNCH_CHECK("k_score_rows");
  return LIME_OK;
}

lime_status launch_score_rows(const ScoreArgs& a, cudaStream_t st) {
  if (a.dtype == LIME_F32) {
    if (a.d == 64) return launch_score_rows_f32_t<64, 8>(a, st);
    return a.ell == 8 ? launch_score_rows_f32_t<32, 8>(a, st) : launch_score_rows_f32_t<32, 16>(a, st);
  }
  switch (a.d) {
    case 32: return launch_score_rows_d<32>(a, st);
    case 64: return launch_score_rows_d<64>(a, st);
    case 128: return launch_score_rows_d<128>(a, st);
    default: return launch_score_rows_d<256>(a, st);
  }
}

}  // namespace lime
