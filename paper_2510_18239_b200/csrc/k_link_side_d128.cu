// The link side of one XOR layer at d = d_ff = 128 with four heads for batches of few link rows (bf16 storage): a cluster of four
// blocks per ROWS link rows (one or more users), instead of the merge, GatedMLP and operand kernels.
//
//   Ohat (merged over the history's chunks) -> [gate | up] = Ohat . [Mvg | Mvu],  U = SiLU(gate) * up,  T = U W_o,  L^P += T
//   LN(T) -> [Q2 | K2 | G2 | U2] = LN(T) . Wprep of the next layer                             (Eq. 5, Eq. 8, Eq. 7; k_link_prep.cu)
//
// The three kernels it stands in for stream 800 KB of weights through tcgen05 tiles of 128 link rows, which is the right shape
// for thousands of rows; a batch of 60 users has 2000, and what it pays for is three launches and three pipeline fills on a
// few SMs (64 users: 25 us a layer with the merge, one user: 14 us; here 14 and 8 us).  Here block r of a cluster takes head r: its part of the
// contraction of [gate | up], a quarter of the columns of U and T, and the operands of head r; B fragments of mma.m16n8k16 go
// from global memory straight to registers, requested before the exchange that a step waits for.  Same folded weights and
// the same places of rounding as the tcgen05 kernels.  Exchanges through distributed shared memory, data and arrival
// together (st.async): partial [gate | up] to the column's owner, then U and T to everyone.
// Contraction order and shared-memory layout of the activations as in k_link_side_d256.cu (row pitch 256 bytes here).
#include "lime_common.cuh"
#include "tc_common.cuh"

namespace lime {

constexpr int L1_D = 128, L1_H = 4, L1_CL = 4, L1_WARPS = 16, L1_THREADS = L1_WARPS * 32;

template <int ROWS_>
struct L1Cfg {
  static constexpr int ROWS = ROWS_, MT = ROWS / 16;
  static constexpr uint32_t ABUF = ROWS * 256;                   // [rows x 128] bf16
  static constexpr int T_LD = 132, V_LD = ROWS * 2 + 16;
  static constexpr uint32_t OFF_A = 0;                           // Ohat of this block's head, later LN(T)
  static constexpr uint32_t OFF_U = OFF_A + ABUF;                // U, all columns
  static constexpr uint32_t OFF_PIN = OFF_U + ABUF;              // [4 sources][rows][gate 32 | up 32] fp32
  static constexpr uint32_t OFF_T = OFF_PIN;                     // over it, once U is formed everywhere: T fp32 [rows x T_LD]
  static constexpr uint32_t OFF_V = OFF_PIN;                     // over that: G2^T | U2^T of head r [2][128 x rows] bf16
  static constexpr uint32_t PIN_BYTES = 4 * ROWS * 256, T_BYTES = ROWS * T_LD * 4, V_BYTES = 2 * 128 * V_LD;
  static constexpr uint32_t R_BYTES = PIN_BYTES > T_BYTES ? (PIN_BYTES > V_BYTES ? PIN_BYTES : V_BYTES) : (T_BYTES > V_BYTES ? T_BYTES : V_BYTES);
  static constexpr uint32_t OFF_BAR = OFF_PIN + R_BYTES;         // [3]: partial sums, U, T of the peers
  static constexpr uint32_t SMEM = OFF_BAR + 32;
  static_assert(SMEM <= 232448, "shared memory budget of one block");
};

struct LinkSide128Params {
  int users, ell;
  const __nv_bfloat16* Ohat; const float *part_m, *part_s, *part_acc; const int32_t* chunk_start;
  const __nv_bfloat16 *WpostT, *WoT, *WprepT;                    // WprepT nullable: no operands
  int need_hist, lp_accumulate, ln;
  float* LP;
  __nv_bfloat16 *link_states, *Q2, *K2, *G2t, *U2t;
  float eps;
  int* err;
};

__device__ __forceinline__ uint32_t l1_at(int row, int chunk) { return (uint32_t)row * 256u + ((uint32_t)(chunk ^ ((row & 1) << 2)) << 4); }
__device__ __forceinline__ uint32_t l1_pack(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ void l1_mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float l1_silu(float x) {              // the tanh form of the tcgen05 kernels
  const float hx = 0.5f * x;
  float th;
  asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(hx));
  return fmaf(hx, th, hx);
}
__device__ __forceinline__ uint32_t l1_peer(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void l1_push(uint32_t addr, const uint4& v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
// four adjacent columns of one row from the accumulators of a quad's lane pair: even lanes end with row g, odd ones with g + 8
__device__ __forceinline__ uint4 l1_four(const float (&c)[4], int t) {
  const bool odd = t & 1;
  const float a = __shfl_xor_sync(0xffffffffu, odd ? c[0] : c[2], 1), b = __shfl_xor_sync(0xffffffffu, odd ? c[1] : c[3], 1);
  return odd ? make_uint4(__float_as_uint(a), __float_as_uint(b), __float_as_uint(c[2]), __float_as_uint(c[3]))
             : make_uint4(__float_as_uint(c[0]), __float_as_uint(c[1]), __float_as_uint(a), __float_as_uint(b));
}
// B fragments of NB n-tiles over the whole contraction of 128 (four blocks of 32), requested by load()
template <int NB>
struct L1Weights {
  uint4 f[4][NB];
  __device__ __forceinline__ void load(const __nv_bfloat16* const (&b)[NB]) {
#pragma unroll
    for (int kb = 0; kb < 4; ++kb)
#pragma unroll
      for (int n = 0; n < NB; ++n) f[kb][n] = __ldg(reinterpret_cast<const uint4*>(b[n] + kb * 32));
  }
  // acc[n] += 16 rows from row0 of the operand at a
  __device__ __forceinline__ void run(float (&acc)[NB][4], const uint8_t* a, int row0, int g, int t) const {
#pragma unroll
    for (int kb = 0; kb < 4; ++kb) {
      const uint8_t* at = a + l1_at(row0 + g, kb * 4 + t);
      const uint4 x = *reinterpret_cast<const uint4*>(at), y = *reinterpret_cast<const uint4*>(at + 8 * 256);
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        l1_mma(acc[n], x.x, y.x, x.y, y.y, f[kb][n].x, f[kb][n].y);
        l1_mma(acc[n], x.z, y.z, x.w, y.w, f[kb][n].z, f[kb][n].w);
      }
    }
  }
};
template <int NB>
__device__ __forceinline__ void l1_zero(float (&acc)[NB][4]) {
#pragma unroll
  for (int n = 0; n < NB; ++n)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
}

template <class G>
__global__ void __launch_bounds__(L1_THREADS, 1)
k_link_side_d128(const LinkSide128Params p) {
  constexpr int ROWS = G::ROWS, MT = G::MT, D = L1_D, H = L1_H, CL = L1_CL;
  extern __shared__ __align__(1024) uint8_t sm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int rank = (int)(blockIdx.x % CL);
  const int row_first = (int)(blockIdx.x / CL) * ROWS;           // first link row (users x ell) of the cluster
  const int rows = min(ROWS, p.users * p.ell - row_first);
  const int HL = H * p.ell;
  const uint32_t sb = (uint32_t)__cvta_generic_to_shared(sm);
  uint64_t* const bars = reinterpret_cast<uint64_t*>(sm + G::OFF_BAR);
  const uint32_t bar_a = sb + G::OFF_BAR;
  float* const Ts = reinterpret_cast<float*>(sm + G::OFF_T);
  if (tid == 0) {
    const uint32_t bytes[3] = {(CL - 1) * ROWS * 256u, (CL - 1) * ROWS * 64u, (CL - 1) * ROWS * 128u};
    for (int i = 0; i < 3; ++i) {
      tc::mbar_init(&bars[i], 1);
      tc::mbar_arrive_expect_tx(&bars[i], bytes[i]);
    }
    tc::fence_barrier_init();
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  pdl_wait();
  pdl_launch_dependents();                                       // behind the wait: lime_common.cuh, the update beside the link side

  // ---- [gate | up], the part of head `rank`: warp = hidden columns warp * 8 .. (gate and up)
  {
    L1Weights<2> w;
    const __nv_bfloat16* wp = p.WpostT + (int64_t)(warp * 8 + g) * (H * D) + rank * D + t * 8;
    w.load({wp, wp + (int64_t)D * (H * D)});
    for (int i = tid; i < ROWS * 16; i += L1_THREADS) {
      const int c = i & 15, lr = i >> 4;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (lr < rows) {
        const int u = (row_first + lr) / p.ell, l = (row_first + lr) % p.ell;
        const int c0 = __ldg(p.chunk_start + u), c1 = __ldg(p.chunk_start + u + 1);
        if (c1 - c0 == 1) {
          v = *(reinterpret_cast<const uint4*>(p.Ohat + ((int64_t)(row_first + lr) * H + rank) * D) + c);
        } else if (c1 > c0) {
          // chunks combined with log-sum-exp weights (maxima in the log2 domain), as k_link_attn_merge_norm does
          const int row = rank * p.ell + l;
          float M = -INFINITY, S = 0.f, a[8];
          for (int k = c0; k < c1; ++k) M = fmaxf(M, __ldg(p.part_m + (int64_t)k * HL + row));
#pragma unroll
          for (int e = 0; e < 8; ++e) a[e] = 0.f;
#pragma unroll 2
          for (int k = c0; k < c1; ++k) {
            const float wt = exp2f(__ldg(p.part_m + (int64_t)k * HL + row) - M);
            S = fmaf(wt, __ldg(p.part_s + (int64_t)k * HL + row), S);
            const float4* src = reinterpret_cast<const float4*>(p.part_acc + ((int64_t)k * HL + row) * D + c * 8);
            const float4 x = __ldg(src), y = __ldg(src + 1);
            a[0] = fmaf(wt, x.x, a[0]); a[1] = fmaf(wt, x.y, a[1]); a[2] = fmaf(wt, x.z, a[2]); a[3] = fmaf(wt, x.w, a[3]);
            a[4] = fmaf(wt, y.x, a[4]); a[5] = fmaf(wt, y.y, a[5]); a[6] = fmaf(wt, y.z, a[6]); a[7] = fmaf(wt, y.w, a[7]);
          }
          const float inv = 1.0f / S;
          v = make_uint4(l1_pack(a[0] * inv, a[1] * inv), l1_pack(a[2] * inv, a[3] * inv), l1_pack(a[4] * inv, a[5] * inv), l1_pack(a[6] * inv, a[7] * inv));
        }
      }
      *reinterpret_cast<uint4*>(sm + G::OFF_A + l1_at(lr, c)) = v;
    }
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");      // every block of the cluster runs, its barriers exist
    const int owner = warp >> 2;                                 // of these hidden columns
    const uint32_t at = sb + G::OFF_PIN + (rank * ROWS + g + 8 * (t & 1)) * 256 + ((warp & 3) * 8 + (t >> 1) * 4) * 4;
    const uint32_t peer = l1_peer(at, owner), peer_bar = l1_peer(bar_a, owner);
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      float acc[2][4];
      l1_zero(acc);
      w.run(acc, sm + G::OFF_A, m * 16, g, t);
      const uint4 gt = l1_four(acc[0], t), up = l1_four(acc[1], t);
      if (owner == rank) {
        *reinterpret_cast<uint4*>(sm + (at - sb) + m * 16 * 256) = gt;
        *reinterpret_cast<uint4*>(sm + (at - sb) + m * 16 * 256 + 128) = up;
      } else {
        l1_push(peer + m * 16 * 256, gt, peer_bar);
        l1_push(peer + m * 16 * 256 + 128, up, peer_bar);
      }
    }
  }
  // ---- U of this block's 32 hidden columns -> everyone.  (W_o is requested first: warp = (n-tile, row tiles) of T)
  L1Weights<1> wo;
  const int tn = warp & 3, tm0 = warp >> 2;                      // n-tile of T within the block's columns; row tiles tm0, tm0 + 4, ..
  wo.load({p.WoT + (int64_t)(rank * 32 + tn * 8 + g) * D + t * 8});
  __syncthreads();
  tc::mbar_wait(&bars[0], 0, p.err, 89);
  for (int i = tid; i < ROWS * 4; i += L1_THREADS) {
    const int lr = i >> 2, c8 = (i & 3) * 8;
    const float* src = reinterpret_cast<const float*>(sm + G::OFF_PIN) + lr * 64 + c8;
    float x[8], y[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = y[e] = 0.f;
#pragma unroll
    for (int q = 0; q < CL; ++q)
#pragma unroll
      for (int e = 0; e < 8; e += 4) {
        const float4 a = *reinterpret_cast<const float4*>(src + q * ROWS * 64 + e), b = *reinterpret_cast<const float4*>(src + q * ROWS * 64 + 32 + e);
        x[e] += a.x; x[e + 1] += a.y; x[e + 2] += a.z; x[e + 3] += a.w;
        y[e] += b.x; y[e + 1] += b.y; y[e + 2] += b.z; y[e + 3] += b.w;
      }
    uint4 v;
    v.x = l1_pack(l1_silu(x[0]) * y[0], l1_silu(x[1]) * y[1]); v.y = l1_pack(l1_silu(x[2]) * y[2], l1_silu(x[3]) * y[3]);
    v.z = l1_pack(l1_silu(x[4]) * y[4], l1_silu(x[5]) * y[5]); v.w = l1_pack(l1_silu(x[6]) * y[6], l1_silu(x[7]) * y[7]);
    const uint32_t at = G::OFF_U + l1_at(lr, rank * 4 + (i & 3));
    *reinterpret_cast<uint4*>(sm + at) = v;
    // (the pushes follow a barrier: T may land over the partial sums as soon as every block's U is out)
  }
  __syncthreads();
  for (int i = tid; i < ROWS * 4; i += L1_THREADS) {
    const uint32_t at = G::OFF_U + l1_at(i >> 2, rank * 4 + (i & 3));
    const uint4 v = *reinterpret_cast<const uint4*>(sm + at);
#pragma unroll
    for (int r = 1; r < CL; ++r) l1_push(l1_peer(sb + at, (rank + r) % CL), v, l1_peer(bar_a + 8, (rank + r) % CL));
  }
  tc::mbar_wait(&bars[1], 0, p.err, 90);
  // ---- T of this block's 32 columns -> everyone
#pragma unroll
  for (int m = 0; m < (MT + 3) / 4; ++m) {
    const int mt = tm0 + 4 * m;
    if (mt < MT) {
      float acc[1][4];
      l1_zero(acc);
      wo.run(acc, sm + G::OFF_U, mt * 16, g, t);
      const uint4 v = l1_four(acc[0], t);
      const uint32_t at = sb + G::OFF_T + ((mt * 16 + g + 8 * (t & 1)) * G::T_LD + rank * 32 + tn * 8 + (t >> 1) * 4) * 4;
      *reinterpret_cast<uint4*>(sm + (at - sb)) = v;
#pragma unroll
      for (int r = 1; r < CL; ++r) l1_push(l1_peer(at, (rank + r) % CL), v, l1_peer(bar_a + 16, (rank + r) % CL));
    }
  }
  // ---- the next layer's operands of head `rank`: warp = segment (Q2, K2, G2, U2) x 32 columns.  The n order is permuted so that
  // a thread ends with eight adjacent columns (n-tile q, column g <-> column (g >> 1) * 8 + 2 q + (g & 1))
  const int seg = warp >> 2, i0 = (warp & 3) * 32;
  const bool operands = p.WprepT != nullptr, mine = operands && (p.need_hist || seg == 0);
  L1Weights<4> wn;
  if (mine) {
    const __nv_bfloat16* wp = p.WprepT + ((int64_t)seg * (H * D) + rank * D + i0 + (g >> 1) * 8 + (g & 1)) * D + t * 8;
    wn.load({wp, wp + 2 * D, wp + 4 * D, wp + 6 * D});
  }
  __syncthreads();
  tc::mbar_wait(&bars[2], 0, p.err, 91);
  // T of this block's columns leaves: the running sum of Eq. 8, the link states
  for (int i = tid; i < rows * 8; i += L1_THREADS) {
    const int lr = i >> 3, c = rank * 32 + (i & 7) * 4;
    float4 v = *reinterpret_cast<const float4*>(Ts + lr * G::T_LD + c);
    const int64_t o = (int64_t)(row_first + lr) * D + c;
    if (p.LP) {
      if (p.lp_accumulate) {
        const float4 x = *reinterpret_cast<const float4*>(p.LP + o);
        v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
      }
      if (p.link_states) *reinterpret_cast<uint2*>(p.link_states + o) = make_uint2(l1_pack(v.x, v.y), l1_pack(v.z, v.w));
      else *reinterpret_cast<float4*>(p.LP + o) = v;
    }
  }
  if (!operands) return;
  // LN(T) -> bf16 where Ohat was: a warp per row, four columns a lane
#pragma unroll
  for (int k = 0; k < ROWS / L1_WARPS; ++k) {
    const int lr = warp * (ROWS / L1_WARPS) + k;
    float4 x = *reinterpret_cast<const float4*>(Ts + lr * G::T_LD + lane * 4);
    if (p.ln) {
      const float mu = warp_sum((x.x + x.y) + (x.z + x.w)) * (1.0f / D);
      x.x -= mu; x.y -= mu; x.z -= mu; x.w -= mu;
      const float rstd = rsqrtf(warp_sum(fmaf(x.x, x.x, x.y * x.y) + fmaf(x.z, x.z, x.w * x.w)) * (1.0f / D) + p.eps);
      x.x *= rstd; x.y *= rstd; x.z *= rstd; x.w *= rstd;
    }
    *reinterpret_cast<uint2*>(sm + G::OFF_A + l1_at(lr, lane >> 1) + (lane & 1) * 8) = make_uint2(l1_pack(x.x, x.y), l1_pack(x.z, x.w));
  }
  __syncthreads();
  if (mine) {
#pragma unroll 1
    for (int m = 0; m < MT; ++m) {
      float acc[4][4];
      l1_zero(acc);
      wn.run(acc, sm + G::OFF_A, m * 16, g, t);
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int lr = m * 16 + g + 8 * hf;
        uint32_t o[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) o[q] = l1_pack(acc[q][2 * hf], acc[q][2 * hf + 1]);
        if (seg < 2) {
          if (lr < rows) {
            const int u = (row_first + lr) / p.ell, l = (row_first + lr) % p.ell;
            *reinterpret_cast<uint4*>((seg ? p.K2 : p.Q2) + ((int64_t)u * HL + rank * p.ell + l) * D + i0 + t * 8) = make_uint4(o[0], o[1], o[2], o[3]);
          }
        } else {
          uint8_t* dst = sm + G::OFF_V + ((seg - 2) * 128 + i0 + t * 8) * G::V_LD + lr * 2;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            *reinterpret_cast<uint16_t*>(dst + (2 * q) * G::V_LD) = (uint16_t)o[q];
            *reinterpret_cast<uint16_t*>(dst + (2 * q + 1) * G::V_LD) = (uint16_t)(o[q] >> 16);
          }
        }
      }
    }
  }
  if (!p.need_hist) return;
  __syncthreads();
  // G2^T | U2^T: per user and hidden unit the links of head `rank` in a row of 2 ell bytes
  const int per_row = ROWS / 8;                                  // 16-byte pieces of eight links
  for (int i = tid; i < 2 * 128 * per_row; i += L1_THREADS) {
    const int c = i % per_row, f = (i / per_row) & 127, which = i / (per_row * 128), lr = c * 8;
    if (lr < rows) {
      const int u = (row_first + lr) / p.ell, l = (row_first + lr) % p.ell;
      *reinterpret_cast<uint4*>((which ? p.U2t : p.G2t) + ((int64_t)u * D + f) * HL + rank * p.ell + l) =
          *reinterpret_cast<const uint4*>(sm + G::OFF_V + (which * 128 + f) * G::V_LD + lr * 2);
    }
  }
}

// Rows a cluster takes: the fewest for which all clusters run at once (32 of four blocks do); 0: too many rows.  128 rows a
// cluster were measured as well: mma.sync then takes as long as the three kernels, whose tcgen05 tiles are full enough by
// then (3200 and 4096 rows: 21-27 against 20-25 us a layer).
static int link_side_d128_rows(int64_t rows) { return rows <= 32 * 32 ? 32 : rows <= 32 * 64 ? 64 : 0; }
bool link_side_d128_wanted(int d, int d_ff, int H, int ell, int64_t users) {
  return d == L1_D && d_ff == L1_D && H == L1_H && ell % 8 == 0 && link_side_d128_rows(users * ell) != 0;
}

int link_side_d128_blocks(int64_t rows) {
  const int per = link_side_d128_rows(rows);
  return per == 0 ? 0 : (int)((rows + per - 1) / per) * L1_CL;
}

template <class G>
static lime_status launch_l1(const LinkSide128Params& p, cudaStream_t st) {
  static bool smem_set[kMaxDeviceOrdinals] = {};
  lime_status s = ensure_dynamic_smem((const void*)k_link_side_d128<G>, (int)G::SMEM, smem_set);
  if (s != LIME_OK) return s;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((p.users * p.ell + G::ROWS - 1) / G::ROWS) * L1_CL);
  cfg.blockDim = dim3(L1_THREADS);
  cfg.dynamicSmemBytes = G::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = L1_CL; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  ProfScope _p("k_link_side_d128", st);
  cudaLaunchKernelEx(&cfg, k_link_side_d128<G>, p);
  LIME_LAUNCH_CHECK("k_link_side_d128");
  return LIME_OK;
}

lime_status launch_link_side_d128(const LinkSide128Args& a, cudaStream_t st) {
  if (a.users == 0) return LIME_OK;
  LinkSide128Params p;
  typedef const __nv_bfloat16* B16;
  p.users = a.users; p.ell = a.ell; p.Ohat = (B16)a.Ohat; p.part_m = a.part_m; p.part_s = a.part_s; p.part_acc = a.part_acc;
  p.chunk_start = a.chunk_start; p.WpostT = (B16)a.WpostT; p.WoT = (B16)a.WoT; p.WprepT = (B16)a.WprepT;
  p.need_hist = a.need_hist; p.lp_accumulate = a.lp_accumulate; p.ln = a.ln; p.LP = a.LP;
  p.link_states = (__nv_bfloat16*)a.link_states; p.Q2 = (__nv_bfloat16*)a.Q2; p.K2 = (__nv_bfloat16*)a.K2;
  p.G2t = (__nv_bfloat16*)a.G2t; p.U2t = (__nv_bfloat16*)a.U2t; p.eps = a.eps; p.err = a.err;
  switch (link_side_d128_rows((int64_t)a.users * a.ell)) {
    case 32: return launch_l1<L1Cfg<32>>(p, st);
    case 64: return launch_l1<L1Cfg<64>>(p, st);
  }
  return LIME_UNSUPPORTED_SHAPE;
}

}  // namespace lime
