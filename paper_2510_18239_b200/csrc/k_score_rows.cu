// Candidate scoring with every warp on its own (Eq. 4, bf16 storage): candidates by id from the corpus caches, ragged
// candidate lists, and widths the streaming scorers are not built for.
//
//   logit[i] = < sum_l W[r, l] LS_b[l, :], T[r, :] >,   r = cand_ids[i] (or i), b = user of slot i
//
// What bounds it: the rate at which HBM serves random rows.  Rows by id arrive in pieces of 2 d and 2 ell bytes; the
// memory system opens about 16.5 G different 256-byte blocks a second whatever fetches them, so the kernel's part is to
// keep enough rows in flight and to add no latency of its own.  A warp takes 16 MT consecutive slots, reads its rows from
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
  int B, C, n_groups;      // groups of 16 * MT slots
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

template <int D, int ELL, int MT>
__global__ void __launch_bounds__(SR_WARPS * 32, sr_blocks(D, ELL))
k_score_rows(const ScoreRowsParams p) {
  constexpr int NT = ELL / 8, NL = ELL / 4, KJ = D / 32, RW = 2 * MT;    // n-tiles, links per thread, 32-column chunks, rows per thread
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int g_begin = (int)(((int64_t)blockIdx.x * p.n_groups) / gridDim.x);
  const int g_end = (int)(((int64_t)(blockIdx.x + 1) * p.n_groups) / gridDim.x);
  pdl_wait();
  int b = -1;
  for (int grp = g_begin + warp; grp < g_end; grp += SR_WARPS) {
    const int s0 = grp * (16 * MT);
    const int s1 = min(s0 + 16 * MT, p.total);
    // one row index per slot
    int row = s0 + lane;
    bool in = (MT == 2 || lane < 16) && row < s1;
    if (p.ids != nullptr) {
      const int32_t id = in ? __ldg(p.ids + row) : 0;
      const bool good = id >= 0 && id < p.rows;
      if (in && !good && p.flag != nullptr) atomicMin(p.flag, row);
      in = in && good;
      row = id;
    }
    const unsigned live = __ballot_sync(0xffffffffu, in);
    // T rows as A fragments (all chunks requested at once), weight pieces
    uint4 a[RW][KJ];
    uint32_t w[RW][NL / 2];
#pragma unroll
    for (int i = 0; i < RW; ++i) {
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
        float acc[MT][NT][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
          for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[m][n][e] = 0.f;
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
            for (int n = 0; n < NB; ++n)
#pragma unroll
              for (int m = 0; m < MT; ++m) {
                sr_mma(acc[m][n0 + n], a[2 * m][j].x, a[2 * m + 1][j].x, a[2 * m][j].y, a[2 * m + 1][j].y, bf[n].x, bf[n].y);
                sr_mma(acc[m][n0 + n], a[2 * m][j].z, a[2 * m + 1][j].z, a[2 * m][j].w, a[2 * m + 1][j].w, bf[n].z, bf[n].w);
              }
          }
        }
        // dot with the weights: links t * NL + 2 n + {0, 1} of rows g (c0, c1) and g + 8 (c2, c3)
        float v[RW];
#pragma unroll
        for (int i = 0; i < RW; ++i) {
          float s = 0.f;
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            const uint32_t u = w[i][n];
            s = fmaf(__uint_as_float(u << 16), acc[i >> 1][n][(i & 1) * 2], s);
            s = fmaf(__uint_as_float(u & 0xffff0000u), acc[i >> 1][n][(i & 1) * 2 + 1], s);
          }
          s += __shfl_xor_sync(0xffffffffu, s, 1);
          s += __shfl_xor_sync(0xffffffffu, s, 2);
          v[i] = s;
        }
        // lane (g, t) keeps row g + 8 t
        const float mine = RW == 4 ? (t == 0 ? v[0] : t == 1 ? v[1] : t == 2 ? v[2] : v[RW - 1]) : (t == 0 ? v[0] : v[1]);
        const int slot = s0 + g + 8 * t;
        const int u_begin = p.cand_off == nullptr ? b * p.C : __ldg(p.cand_off + b);
        if (slot >= u_begin && slot < u_end) out = mine;
      }
      if (u_end >= s1 || b + 1 >= p.B) break;
      ++b;
    }
    const int slot = s0 + g + 8 * t;
    if ((MT == 2 || t < 2) && slot < s1) p.logits[slot] = out;
  }
}

static bool score_rows_supported(const ScoreArgs& a) {
  if (a.dtype != LIME_BF16) return false;
  const bool d_ok = a.d == 32 || a.d == 64 || a.d == 128 || a.d == 256;
  const bool l_ok = a.ell == 8 || a.ell == 16 || a.ell == 32 || a.ell == 64;
  if (!d_ok || !l_ok) return false;
  if (a.cand_off == nullptr && a.C <= 0) return false;
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
  constexpr int MT = 1;      // 32 slots per pass while rows, accumulators and weights fit in 128 registers
  ScoreRowsParams p;
  p.LS = (const __nv_bfloat16*)a.LS; p.W = (const __nv_bfloat16*)a.W; p.T = (const __nv_bfloat16*)a.T;
  p.cand_off = a.cand_off; p.ids = a.cand_ids; p.flag = a.dev_flag; p.logits = a.logits;
  p.ldt = a.ldt ? (int)a.ldt : D; p.ldw = a.ldw ? (int)a.ldw : ELL;
  p.rows = (int)(a.cand_ids ? a.corpus_rows : a.total); p.total = (int)a.total; p.B = a.B; p.C = a.C;
  p.n_groups = (int)((a.total + 16 * MT - 1) / (16 * MT));
  const int64_t blocks = (p.n_groups + SR_WARPS - 1) / SR_WARPS, cap = 2 * kSMs;
  ProfScope _p("k_score_rows", st);
  launch_pdl(k_score_rows<D, ELL, MT>, dim3((unsigned)(blocks < cap ? blocks : cap)), dim3(SR_WARPS * 32), 0, st, p);
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

lime_status launch_score_rows(const ScoreArgs& a, cudaStream_t st) {
  switch (a.d) {
    case 32: return launch_score_rows_d<32>(a, st);
    case 64: return launch_score_rows_d<64>(a, st);
    case 128: return launch_score_rows_d<128>(a, st);
    default: return launch_score_rows_d<256>(a, st);
  }
}

}  // namespace lime
