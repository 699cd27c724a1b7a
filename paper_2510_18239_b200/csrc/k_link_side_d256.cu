// The link side of one XOR layer at d = d_ff = 256 with 32 links (bf16 storage), one cluster of four blocks per one or two users:
//
//   Ohat (merged over the history's chunks)  ->  O = Ohat W_V,  T = (SiLU(O W_g) * (O W_u)) W_o,  L^P += T          (Eq. 5, Eq. 8)
//   LN(T) -> Q | K | V = LN(T) [W_Q | W_K | W_V] of the next layer -> folded queries Q2_h = Q_h W_K,h^T * scale, folded keys
//   K2_h = K_h W_Q,h^T * scale, link values V (transposed): the operands the streaming kernels take               (Eq. 7)
//
// A user has 32 link rows, so a step is a 32 x 256 x 256 product and what bounds it is the latency of a chain of five
// dependent products, each of which reads its weights (128 to 384 KB) from L2.  One 128-row tcgen05 tile would hold four
// users and leave a batch of 64 users on 16 SMs (MLP 33 us, operands 13 us, merge 10 us per layer); here a block takes a
// quarter of the columns of every product, and the B fragments of mma.m16n8k16 go from global memory straight to registers
// through a ring per warp - with two or four 16-row tiles there is next to nothing to share between warps - which is filled
// before the exchange that a step waits for.  The blocks exchange O, U and T through distributed shared memory.  Two users
// per cluster once one per cluster no longer fits the GPU: the weights then cross L2 half as often.
// Weights are taken unfolded (4 + 5 d^2 products per row instead of 9 + 9), exact as stored; the activations that everything
// depends on - O, U, LN(T), Q, K - enter as a bf16 value and its bf16 remainder, which leaves the error of the link states
// where fp32 link rows had it (0.6 % of their norm; operands rounded once: 0.9 %).
// The contraction index is permuted so that thread t of a quad holds columns (4 j + t) * 8 .. + 7 of both operands (one 16-byte
// read gives the fragments of two k-steps).  Activations in shared memory: row pitch 512 bytes, 16-byte chunk c at
// c ^ ((row & 1) << 2), so that the eight threads of a read phase (two rows, four chunks) cover all banks.
#include "lime_common.cuh"
#include "tc_common.cuh"

namespace lime {

constexpr int LS2_D = 256, LS2_ELL = 32, LS2_WARPS = 16, LS2_THREADS = LS2_WARPS * 32;

template <int H_, int UPC_>
struct Ls2Cfg {
  static constexpr int H = H_, UPC = UPC_, CL = 4, DH = LS2_D / H, HC = H / CL, NS = LS2_D / CL;   // users of a cluster; heads and columns of a block
  static constexpr int ROWS = 32 * UPC, MB = UPC;                // link rows of a cluster; 16-row tiles per warp (8 n-tiles x 2 row halves)
  static constexpr uint32_t ABUF = ROWS * 512;                   // [rows x 256] bf16
  static constexpr int T_LD = 260;
  // Ohat [HC][rows x 256] and O (value | remainder); over both, once read, T (fp32) and then Q | K of the block's columns
  static constexpr uint32_t OFF_OHAT = 0, OFF_O = OFF_OHAT + HC * ABUF, OFF_T = 0, OFF_QK = 0;
  static constexpr uint32_t OFF_U = OFF_O + 2 * ABUF;            // U, later LN(T): value | remainder
  static constexpr uint32_t OFF_V = OFF_U + 2 * ABUF;            // V^T [NS x rows] bf16
  static constexpr int V_LD = ROWS * 2 + 16;
  static constexpr uint32_t OFF_BAR = OFF_V + NS * V_LD;         // [3] what the peers sent of O, U and T has arrived
  static constexpr uint32_t SMEM = OFF_BAR + 32;
  static_assert(ROWS * T_LD * 4 <= (int)OFF_U && 4 * ROWS * NS * 2 <= (int)OFF_U, "what lies over Ohat and O");
  static_assert(SMEM <= 232448, "shared memory budget of one block");
};

struct LinkSide256Params {
  int users;
  const __nv_bfloat16* Ohat; const float *part_m, *part_s, *part_acc; const int32_t* chunk_start;   // MLP half (Ohat nullable: none)
  const float* T_in; int t_shared;                               // without the MLP half: T, fp32 [users x 32 x d] (or one block)
  const __nv_bfloat16 *WvT, *WguT, *WoT;
  const __nv_bfloat16 *WqT, *WkT, *WvT_next, *Wq, *Wk;           // operand half (WqT nullable: none)
  int need_hist, lp_accumulate, ln;
  float *T_out, *LP;
  __nv_bfloat16 *link_states, *Q2, *K2, *V2t;
  float scale, eps;
  int* err;
};

__device__ __forceinline__ uint32_t l2_at(int row, int chunk, int pitch) { return (uint32_t)row * pitch + ((uint32_t)(chunk ^ ((row & 1) << 2)) << 4); }
__device__ __forceinline__ uint32_t l2_pack(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ void l2_split(float x, float y, uint32_t& hi, uint32_t& lo) {
  hi = l2_pack(x, y);
  lo = l2_pack(x - __uint_as_float(hi << 16), y - __uint_as_float(hi & 0xffff0000u));
}
__device__ __forceinline__ void l2_mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t l2_peer(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// 16 bytes to a peer's shared memory, counted on the barrier beside it there
__device__ __forceinline__ void l2_st_peer(uint32_t addr, const uint4& v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ void l2_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void l2_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// One warp's share of a product: NB n-tiles against MB 16-row tiles, contraction over KB blocks of 32.  The B rows of n-tile i
// start at b[i] (this thread's row, this thread's chunk of block 0).  begin() requests the first R blocks, run() goes through
// all of them and keeps R in flight.
template <int NB, int R>
struct L2Stream {
  const __nv_bfloat16* b[NB];
  uint4 f[R][NB];
  __device__ __forceinline__ void load(int kb) {
#pragma unroll
    for (int n = 0; n < NB; ++n) f[kb % R][n] = __ldg(reinterpret_cast<const uint4*>(b[n] + kb * 32));
  }
  __device__ __forceinline__ void begin() {
#pragma unroll
    for (int kb = 0; kb < R; ++kb) load(kb);
  }
  // A: value at a, remainder at a + rem (REM); rows m0 * 16 .. of pitch `pitch`, block 0 at chunk c0
  template <int MB, int KB, bool REM>
  __device__ __forceinline__ void run(float (&acc)[MB][NB][4], const uint8_t* a, uint32_t rem, int m0, int pitch, int c0, int g, int t) {
#pragma unroll
    for (int kb = 0; kb < KB; ++kb) {
#pragma unroll
      for (int m = 0; m < MB; ++m) {
        const uint32_t at = l2_at((m0 + m) * 16 + g, c0 + kb * 4 + t, pitch);
#pragma unroll
        for (int r = 0; r < (REM ? 2 : 1); ++r) {
          const uint4 x = *reinterpret_cast<const uint4*>(a + at + r * rem), y = *reinterpret_cast<const uint4*>(a + at + 8 * pitch + r * rem);
#pragma unroll
          for (int n = 0; n < NB; ++n) {
            const uint4 w = f[kb % R][n];
            l2_mma(acc[m][n], x.x, y.x, x.y, y.y, w.x, w.y);
            l2_mma(acc[m][n], x.z, y.z, x.w, y.w, w.z, w.w);
          }
        }
      }
      if (kb + R < KB) load(kb + R);
    }
  }
};
template <int MB, int NB>
__device__ __forceinline__ void l2_zero(float (&acc)[MB][NB][4]) {
#pragma unroll
  for (int m = 0; m < MB; ++m)
#pragma unroll
    for (int n = 0; n < NB; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[m][n][e] = 0.f;
}

template <class G>
__global__ void __launch_bounds__(LS2_THREADS, 1)
k_link_side_d256(const LinkSide256Params p) {
  constexpr int H = G::H, CL = G::CL, DH = G::DH, HC = G::HC, NS = G::NS, MB = G::MB, ROWS = G::ROWS, D = LS2_D;
  extern __shared__ __align__(1024) uint8_t sm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int rank = (int)(blockIdx.x % CL), u0 = (int)(blockIdx.x / CL) * G::UPC;
  const int rows = min(ROWS, (p.users - u0) * 32);               // link rows that exist
  const int n0 = rank * NS;                                      // this block's first column of every product
  // this warp's n-tile within the block's columns, and its first 16-row tile
  const int wn = warp & 7, m0 = (warp >> 3) * MB;
  const uint32_t sb = (uint32_t)__cvta_generic_to_shared(sm);
  float* const Ts = reinterpret_cast<float*>(sm + G::OFF_T);
  uint64_t* const bars = reinterpret_cast<uint64_t*>(sm + G::OFF_BAR);
  if (tid == 0) {
    for (int i = 0; i < 3; ++i) {
      tc::mbar_init(&bars[i], 1);
      tc::mbar_arrive_expect_tx(&bars[i], (CL - 1) * (uint32_t)(ROWS * NS * 4));
    }
    tc::fence_barrier_init();
  }
  l2_arrive();                                                   // this block runs and its barriers exist: it may be written to
  pdl_wait();
  pdl_launch_dependents();                                       // behind the wait: lime_common.cuh, the update beside the link side

  // c (columns col, col + 1 of rows m * 16 + g and + 8) to this block's operand buffer at `off`, as value and remainder
  auto store_split = [&](uint32_t off, int m, int col, const float (&c)[4]) {
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      uint32_t hi, lo;
      l2_split(c[2 * hf], c[2 * hf + 1], hi, lo);
      uint8_t* at = sm + off + l2_at(m * 16 + g + 8 * hf, col >> 3, 512) + (col & 7) * 2;
      *reinterpret_cast<uint32_t*>(at) = hi;
      *reinterpret_cast<uint32_t*>(at + G::ABUF) = lo;
    }
  };
  // this block's columns of a buffer to the other blocks of the cluster, 16 bytes at a time (4-byte stores from the
  // accumulators to every block were measured: the exchanges then took longer than the products).  `per` chunks per row
  // from chunk c0, at(row, chunk) the position.  Data and arrival travel together, no fence or cluster barrier follows.  A
  // buffer is only written over once its readers are done: whoever sends U has read all of O, and T (over O) is sent by
  // blocks that have every U.
  auto push = [&](int which, int n_rows, int per, int c0, auto at) {
    __syncthreads();
    for (int i = tid; i < n_rows * per; i += LS2_THREADS) {
      const uint32_t o = at(i / per, c0 + i % per);
      const uint4 v = *reinterpret_cast<const uint4*>(sm + o);
#pragma unroll
      for (int r = 1; r < CL; ++r) l2_st_peer(l2_peer(sb + o, (rank + r) % CL), v, l2_peer(sb + G::OFF_BAR + which * 8, (rank + r) % CL));
    }
  };
  auto push_split = [&](int which, uint32_t off) {
    push(which, 2 * ROWS, NS / 8, n0 / 8, [&](int row, int c) { return off + (row >= ROWS ? G::ABUF : 0) + l2_at(row % ROWS, c, 512); });
  };

  if (p.Ohat != nullptr) {
    L2Stream<1, 8> s1;
    s1.b[0] = p.WvT + (int64_t)(n0 + wn * 8 + g) * D + t * 8;
    s1.begin();
    // ---- attention rows of this block's heads -> shared memory (chunks merged with log-sum-exp weights, normalised)
    constexpr int HL = H * LS2_ELL;
    for (int i = tid; i < HC * ROWS * 32; i += LS2_THREADS) {
      const int c = i & 31, lr = (i >> 5) % ROWS, hc = i / (ROWS * 32), h = rank * HC + hc, l = lr & 31, u = u0 + (lr >> 5);
      uint4 v = make_uint4(0, 0, 0, 0);
      if (lr < rows) {
        const int ck0 = __ldg(p.chunk_start + u), ck1 = __ldg(p.chunk_start + u + 1);
        if (ck1 - ck0 == 1) {
          v = __ldg(reinterpret_cast<const uint4*>(p.Ohat + ((int64_t)u * 32 + l) * (H * D) + h * D) + c);
        } else if (ck1 > ck0) {
          const int row = h * 32 + l;
          float M = -INFINITY, S = 0.f, a[8];
          for (int k = ck0; k < ck1; ++k) M = fmaxf(M, __ldg(p.part_m + (int64_t)k * HL + row));
#pragma unroll
          for (int e = 0; e < 8; ++e) a[e] = 0.f;
          for (int k = ck0; k < ck1; ++k) {
            const float w = exp2f(__ldg(p.part_m + (int64_t)k * HL + row) - M);
            S = fmaf(w, __ldg(p.part_s + (int64_t)k * HL + row), S);
            const float4* src = reinterpret_cast<const float4*>(p.part_acc + ((int64_t)k * HL + row) * D + c * 8);
            const float4 x = __ldg(src), y = __ldg(src + 1);
            a[0] = fmaf(w, x.x, a[0]); a[1] = fmaf(w, x.y, a[1]); a[2] = fmaf(w, x.z, a[2]); a[3] = fmaf(w, x.w, a[3]);
            a[4] = fmaf(w, y.x, a[4]); a[5] = fmaf(w, y.y, a[5]); a[6] = fmaf(w, y.z, a[6]); a[7] = fmaf(w, y.w, a[7]);
          }
          const float inv = 1.0f / S;
          v = make_uint4(l2_pack(a[0] * inv, a[1] * inv), l2_pack(a[2] * inv, a[3] * inv), l2_pack(a[4] * inv, a[5] * inv), l2_pack(a[6] * inv, a[7] * inv));
        }
      }
      *reinterpret_cast<uint4*>(sm + G::OFF_OHAT + hc * G::ABUF + l2_at(lr, c, 512)) = v;
    }
    __syncthreads();
    // ---- O = Ohat W_V: column n belongs to head n / d_h
    {
      float acc[MB][1][4];
      l2_zero(acc);
      s1.template run<MB, 8, false>(acc, sm + G::OFF_OHAT + (wn * 8 / DH) * G::ABUF, 0, m0, 512, 0, g, t);
#pragma unroll
      for (int m = 0; m < MB; ++m) store_split(G::OFF_O, m0 + m, n0 + wn * 8 + 2 * t, acc[m][0]);
      l2_wait();                                                  // every block of the cluster runs
      push_split(0, G::OFF_O);
    }
    // ---- [gate | up] = O [W_g | W_u], U = SiLU(gate) * up
    {
      L2Stream<2, 8> s2;
      s2.b[0] = p.WguT + (int64_t)(n0 + wn * 8 + g) * D + t * 8;
      s2.b[1] = s2.b[0] + (int64_t)D * D;
      s2.begin();
      tc::mbar_wait(&bars[0], 0, p.err, 85);
      float acc[MB][2][4];
      l2_zero(acc);
      s2.template run<MB, 8, true>(acc, sm + G::OFF_O, G::ABUF, m0, 512, 0, g, t);
#pragma unroll
      for (int m = 0; m < MB; ++m) {
        float x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = __fdividef(acc[m][0][e], 1.0f + __expf(-acc[m][0][e])) * acc[m][1][e];
        store_split(G::OFF_U, m0 + m, n0 + wn * 8 + 2 * t, x);
      }
      push_split(1, G::OFF_U);
    }
    // ---- T = U W_o
    {
      L2Stream<1, 8> s3;
      s3.b[0] = p.WoT + (int64_t)(n0 + wn * 8 + g) * D + t * 8;
      s3.begin();
      tc::mbar_wait(&bars[1], 0, p.err, 86);
      float acc[MB][1][4];
      l2_zero(acc);
      s3.template run<MB, 8, true>(acc, sm + G::OFF_U, G::ABUF, m0, 512, 0, g, t);
#pragma unroll
      for (int m = 0; m < MB; ++m)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf)
          *reinterpret_cast<float2*>(Ts + ((m0 + m) * 16 + g + 8 * hf) * G::T_LD + n0 + wn * 8 + 2 * t) = make_float2(acc[m][0][2 * hf], acc[m][0][2 * hf + 1]);
      push(2, ROWS, NS / 4, n0 / 4, [&](int row, int c) { return G::OFF_T + (uint32_t)(row * G::T_LD + c * 4) * 4; });
    }
  } else {
    const float* src = p.T_in + (p.t_shared ? 0 : (int64_t)u0 * 32 * D);
    for (int i = tid; i < rows * D / 4; i += LS2_THREADS)
      *reinterpret_cast<float4*>(Ts + (i >> 6) * G::T_LD + (i & 63) * 4) = __ldg(reinterpret_cast<const float4*>(src) + i);
  }
  // ---- next layer's operands
  L2Stream<3, 4> s4;
  const bool operands = p.WqT != nullptr;
  if (operands) {
    const int64_t at = (int64_t)(n0 + wn * 8 + g) * D + t * 8;
    s4.b[0] = p.WqT + at;
    s4.b[1] = p.need_hist ? p.WkT + at : s4.b[0];
    s4.b[2] = p.need_hist ? p.WvT_next + at : s4.b[0];
    s4.begin();
  }
  if (p.Ohat != nullptr) tc::mbar_wait(&bars[2], 0, p.err, 87);
  else { l2_wait(); __syncthreads(); }
  // T of this block's columns leaves: fp32 rows, the running sum of Eq. 8, the link states
  if (p.Ohat != nullptr) {
    for (int i = tid; i < rows * NS / 4; i += LS2_THREADS) {
      const int l = i / (NS / 4), c = n0 + (i % (NS / 4)) * 4;
      float4 v = *reinterpret_cast<const float4*>(Ts + l * G::T_LD + c);
      const int64_t o = ((int64_t)u0 * 32 + l) * D + c;
      if (p.T_out) *reinterpret_cast<float4*>(p.T_out + o) = v;
      if (p.LP) {
        if (p.lp_accumulate) {
          const float4 x = *reinterpret_cast<const float4*>(p.LP + o);
          v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
        }
        if (p.link_states) *reinterpret_cast<uint2*>(p.link_states + o) = make_uint2(l2_pack(v.x, v.y), l2_pack(v.z, v.w));
        else *reinterpret_cast<float4*>(p.LP + o) = v;
      }
    }
  }
  if (!operands) return;                                         // uniform over the cluster; nobody writes to a peer from here on
  // LN(T) -> value | remainder over the U buffer (eight columns per lane)
#pragma unroll
  for (int k = 0; k < ROWS / LS2_WARPS; ++k) {
    const int l = warp * (ROWS / LS2_WARPS) + k;
    float x[8];
    *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(Ts + l * G::T_LD + lane * 8);
    *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(Ts + l * G::T_LD + lane * 8 + 4);
    if (p.ln) {
      float s = 0.f, v = 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) s += x[e];
      const float mu = warp_sum(s) * (1.0f / D);
#pragma unroll
      for (int e = 0; e < 8; ++e) { x[e] -= mu; v = fmaf(x[e], x[e], v); }
      const float rstd = rsqrtf(warp_sum(v) * (1.0f / D) + p.eps);
#pragma unroll
      for (int e = 0; e < 8; ++e) x[e] *= rstd;
    }
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) l2_split(x[2 * e], x[2 * e + 1], hi[e], lo[e]);
    *reinterpret_cast<uint4*>(sm + G::OFF_U + l2_at(l, lane, 512)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(sm + G::OFF_U + G::ABUF + l2_at(l, lane, 512)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
  __syncthreads();
  // Q | K | V of this block's columns (its heads); Q and K as value | remainder where T was
  constexpr int QP = NS * 2;                                     // row pitch of Q and K
  constexpr uint32_t QBUF = ROWS * QP;
  {
    float acc[MB][3][4];
    l2_zero(acc);
    s4.template run<MB, 8, true>(acc, sm + G::OFF_U, G::ABUF, m0, 512, 0, g, t);
#pragma unroll
    for (int m = 0; m < MB; ++m) {
      const int col = wn * 8 + 2 * t;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int l = (m0 + m) * 16 + g + 8 * hf;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          uint32_t hi, lo;
          l2_split(acc[m][q][2 * hf], acc[m][q][2 * hf + 1], hi, lo);
          uint8_t* dst = sm + G::OFF_QK + q * 2 * QBUF + l2_at(l, col >> 3, QP) + (col & 7) * 2;
          *reinterpret_cast<uint32_t*>(dst) = hi;
          *reinterpret_cast<uint32_t*>(dst + QBUF) = lo;
        }
        if (p.need_hist) {
          *reinterpret_cast<__nv_bfloat16*>(sm + G::OFF_V + col * G::V_LD + l * 2) = __float2bfloat16_rn(acc[m][2][2 * hf]);
          *reinterpret_cast<__nv_bfloat16*>(sm + G::OFF_V + (col + 1) * G::V_LD + l * 2) = __float2bfloat16_rn(acc[m][2][2 * hf + 1]);
        }
      }
    }
  }
  // folded queries and keys: units of (operand, head, user, 32 columns); the n order is permuted so that a thread ends with eight
  // adjacent columns (n-tile q, column g <-> column (g >> 1) * 8 + 2 q + (g & 1))
  const int per_user = (p.need_hist ? 2 : 1) * HC * 8, n_units = per_user * (rows / 32);
  L2Stream<4, DH / 32> s5;
  auto aim = [&](int unit) {
    const int k = unit % per_user, op = k / (HC * 8), h = rank * HC + (k / 8) % HC, i0 = (k & 7) * 32;
    const __nv_bfloat16* W = op ? p.Wq : p.Wk;
#pragma unroll
    for (int q = 0; q < 4; ++q) s5.b[q] = W + (int64_t)(i0 + (g >> 1) * 8 + 2 * q + (g & 1)) * D + h * DH + t * 8;
  };
  if (warp < n_units) { aim(warp); s5.begin(); }
  __syncthreads();
  if (p.need_hist)
    for (int i = tid; i < NS * rows / 8; i += LS2_THREADS) {
      const int c = i & 3, n = (i >> 2) % NS, k = i / (NS * 4);
      *(reinterpret_cast<uint4*>(p.V2t + ((int64_t)(u0 + k) * D + n0 + n) * 32) + c) = *reinterpret_cast<const uint4*>(sm + G::OFF_V + n * G::V_LD + k * 64 + c * 16);
    }
  for (int unit = warp; unit < n_units; unit += LS2_WARPS) {
    const int k = unit % per_user, usr = unit / per_user, op = k / (HC * 8), hc = (k / 8) % HC, h = rank * HC + hc, i0 = (k & 7) * 32;
    if (unit != warp) { aim(unit); s5.begin(); }
    float acc[2][4][4];
    l2_zero(acc);
    s5.template run<2, DH / 32, true>(acc, sm + G::OFF_QK + op * 2 * QBUF, QBUF, usr * 2, QP, hc * (DH / 8), g, t);
    __nv_bfloat16* dst = (op ? p.K2 : p.Q2) + ((int64_t)(u0 + usr) * (H * 32) + h * 32) * D + i0 + t * 8;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        uint32_t o[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) o[q] = l2_pack(acc[m][q][2 * hf] * p.scale, acc[m][q][2 * hf + 1] * p.scale);
        *reinterpret_cast<uint4*>(dst + (int64_t)(m * 16 + g + 8 * hf) * D) = make_uint4(o[0], o[1], o[2], o[3]);
      }
  }
}

// Any number of users: this is the only link side of the shape.  A layer takes 21 us for 16 users, 35 for 64, 64 for 128, and from
// there 0.47 us a user (256: 121, 512: 240, 1024: 478 us; 0.3 on the last layer), a quarter of an encode at 256 users of 1000 tokens and
// two thirds at 1024 users of 200.  The CUDA-core path is no alternative at any of them (1024 users of 200 tokens, three layers: 29.4 ms,
// 1.76 ms here); 128-row tcgen05 tiles would be full from about 512 users on.
bool link_side_d256_supported(int d, int d_ff, int H, int ell) { return d == LS2_D && d_ff == LS2_D && ell == LS2_ELL && (H == 4 || H == 8); }

// one user per cluster while the clusters run at once (32 of four blocks do, whatever the SMs per GPC), two beyond
static int link_side_d256_users(int users) { return users <= 32 ? 1 : 2; }
int link_side_d256_blocks(int users) { const int per = link_side_d256_users(users); return (users + per - 1) / per * 4; }

template <class G>
static lime_status launch_ls2(const LinkSide256Params& p, cudaStream_t st) {
  static bool smem_set[kMaxDeviceOrdinals] = {};
  lime_status s = ensure_dynamic_smem((const void*)k_link_side_d256<G>, (int)G::SMEM, smem_set);
  if (s != LIME_OK) return s;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((p.users + G::UPC - 1) / G::UPC) * G::CL);
  cfg.blockDim = dim3(LS2_THREADS);
  cfg.dynamicSmemBytes = G::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = G::CL; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  ProfScope _p("k_link_side_d256", st);
  cudaLaunchKernelEx(&cfg, k_link_side_d256<G>, p);
  LIME_LAUNCH_CHECK("k_link_side_d256");
  return LIME_OK;
}

lime_status launch_link_side_d256(const LinkSide256Args& a, cudaStream_t st) {
  if (a.users == 0) return LIME_OK;
  LinkSide256Params p;
  p.users = a.users;
  typedef const __nv_bfloat16* B16;
  p.Ohat = (B16)a.Ohat; p.part_m = a.part_m; p.part_s = a.part_s; p.part_acc = a.part_acc; p.chunk_start = a.chunk_start;
  p.T_in = a.T_in; p.t_shared = a.t_shared;
  p.WvT = (B16)a.WvT; p.WguT = (B16)a.WguT; p.WoT = (B16)a.WoT;
  p.WqT = (B16)a.WqT; p.WkT = (B16)a.WkT; p.WvT_next = (B16)a.WvT_next; p.Wq = (B16)a.Wq; p.Wk = (B16)a.Wk;
  p.need_hist = a.need_hist; p.lp_accumulate = a.lp_accumulate; p.ln = a.ln; p.T_out = a.T_out; p.LP = a.LP;
  p.link_states = (__nv_bfloat16*)a.link_states; p.Q2 = (__nv_bfloat16*)a.Q2; p.K2 = (__nv_bfloat16*)a.K2; p.V2t = (__nv_bfloat16*)a.V2t;
  p.scale = a.scale; p.eps = a.eps; p.err = a.err;
  if (link_side_d256_users(a.users) == 1) return a.H == 4 ? launch_ls2<Ls2Cfg<4, 1>>(p, st) : launch_ls2<Ls2Cfg<8, 1>>(p, st);
  return a.H == 4 ? launch_ls2<Ls2Cfg<4, 2>>(p, st) : launch_ls2<Ls2Cfg<8, 2>>(p, st);
}

}  // namespace lime
