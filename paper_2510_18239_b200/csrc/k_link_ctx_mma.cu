// Link contextualisation with one hidden layer (Eq. 2: L^C_b = MLP(L (+) E^C_b); bf16 storage) on tensor cores:
//
//   x[l, :] = ReLU( first[l, :] + E^C_b W_0[d:] ),  first = (L W_0[:d]) + b_0 from set-up;   L^C_b[l, :] = x[l, :] W_1 + b_1
//
// A block takes one user and 64 output columns.  The second product (ell x w0 x 64 per block) is a few hundred thousand
// multiply-adds, so what bounds the kernel is latency: the weights come in by cp.async under the user's term, and a warp's eight
// columns for all link rows are a chain of mma.m16n8k16.  The activations are fp32 sums, so they enter as a bf16 value and its bf16
// remainder (two products): the accuracy of the CUDA-core kernel (k_ffn_simt.cu), whose single thread per column walked the
// contraction alone (128 users x 32 links, w0 = d = 128: 20 us, here 5).
#include "lime_common.cuh"
#include "tc_common.cuh"

namespace lime {

constexpr int CX_THREADS = 256, CX_COLS = 64;

__device__ __forceinline__ void cx_ldsm(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void cx_ldsm_t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void cx_mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// 16-byte chunk c of a row sits at c ^ (row & 7): eight rows of one chunk cover all banks
__device__ __forceinline__ uint32_t cx_at(int row, int chunk, int pitch) { return (uint32_t)row * pitch + ((uint32_t)(chunk ^ (row & 7)) << 4); }

__global__ void __launch_bounds__(CX_THREADS)
k_link_ctx_mma(const float* __restrict__ first, const __nv_bfloat16* __restrict__ user_ctx, int d_c, const __nv_bfloat16* __restrict__ W0c,
               int w0, int ell, int d, const __nv_bfloat16* __restrict__ W1, const float* __restrict__ b1, float* __restrict__ out) {
  extern __shared__ __align__(128) uint8_t sm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int b = blockIdx.x, n0 = blockIdx.y * CX_COLS;
  const uint32_t sb = (uint32_t)__cvta_generic_to_shared(sm);
  const uint32_t w_bytes = (uint32_t)w0 * CX_COLS * 2, x_bytes = (uint32_t)ell * w0 * 2;     // W_1 columns | x value | x remainder
  float* const u = reinterpret_cast<float*>(sm + w_bytes + 2 * x_bytes);                     // [w0] user's term, then [d_c] features
  float* const ec = u + w0;
  pdl_launch_dependents();
  pdl_wait();
  for (int i = tid; i < w0 * (CX_COLS / 8); i += CX_THREADS) {
    const int k = i / (CX_COLS / 8), c = i % (CX_COLS / 8);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sb + cx_at(k, c, CX_COLS * 2)), "l"(W1 + (int64_t)k * d + n0 + c * 8) : "memory");
  }
  for (int c = tid; c < d_c; c += CX_THREADS) ec[c] = __bfloat162float(user_ctx[(int64_t)b * d_c + c]);
  __syncthreads();
  for (int j = tid; j < w0; j += CX_THREADS) {
    float s = 0.f;
#pragma unroll 8
    for (int c = 0; c < d_c; ++c) s = fmaf(ec[c], __bfloat162float(W0c[(int64_t)c * w0 + j]), s);
    u[j] = s;
  }
  __syncthreads();
  for (int i = tid; i < ell * w0 / 8; i += CX_THREADS) {
    const int l = i / (w0 / 8), c = i % (w0 / 8);
    const float* f = first + (int64_t)l * w0 + c * 8;
    float x[8];
    *reinterpret_cast<float4*>(x) = __ldg(reinterpret_cast<const float4*>(f));
    *reinterpret_cast<float4*>(x + 4) = __ldg(reinterpret_cast<const float4*>(f) + 1);
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float y0 = fmaxf(x[2 * e] + u[c * 8 + 2 * e], 0.f), y1 = fmaxf(x[2 * e + 1] + u[c * 8 + 2 * e + 1], 0.f);
      const __nv_bfloat162 h = __floats2bfloat162_rn(y0, y1);
      const __nv_bfloat162 r = __floats2bfloat162_rn(y0 - __low2float(h), y1 - __high2float(h));
      hi[e] = *reinterpret_cast<const uint32_t*>(&h);
      lo[e] = *reinterpret_cast<const uint32_t*>(&r);
    }
    uint8_t* dst = sm + w_bytes + cx_at(l, c, w0 * 2);
    *reinterpret_cast<uint4*>(dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(dst + x_bytes) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const int n = n0 + warp * 8 + 2 * t;
  const float2 bias = b1 ? *reinterpret_cast<const float2*>(b1 + n) : make_float2(0.f, 0.f);
  for (int m = 0; m < ell; m += 32) {                             // two 16-row tiles at a time
    const int mt = min(2, (ell - m) / 16);
    float acc[2][4] = {};
#pragma unroll 2
    for (int k = 0; k < w0; k += 32) {
      uint32_t w[4];
      cx_ldsm_t(w, sb + cx_at(k + lane, warp, CX_COLS * 2));
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (q < mt)
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) {
            const uint32_t at = sb + w_bytes + cx_at(m + q * 16 + (lane & 15), k / 8 + ks * 2 + (lane >> 4), w0 * 2);
            uint32_t a[4];
            cx_ldsm(a, at);
            cx_mma(acc[q], a, w[2 * ks], w[2 * ks + 1]);
            cx_ldsm(a, at + x_bytes);
            cx_mma(acc[q], a, w[2 * ks], w[2 * ks + 1]);
          }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (q < mt) {
        float* o = out + ((int64_t)b * ell + m + q * 16 + g) * d + n;
        *reinterpret_cast<float2*>(o) = make_float2(acc[q][0] + bias.x, acc[q][1] + bias.y);
        *reinterpret_cast<float2*>(o + 8 * d) = make_float2(acc[q][2] + bias.x, acc[q][3] + bias.y);
      }
  }
}

static size_t link_ctx_mma_smem(int w0, int ell, int d_c) { return (size_t)w0 * CX_COLS * 2 + 2 * (size_t)ell * w0 * 2 + ((size_t)w0 + d_c) * 4; }

// one hidden layer; rows of 16-byte pieces in groups of eight (the swizzle): w0 and d multiples of 64
bool link_ctx_mma_supported(int dtype, int d_c, int w0, int ell, int d, const FfnArgs& f) {
  return dtype == LIME_BF16 && f.n_layers == 1 && w0 % 64 == 0 && d % CX_COLS == 0 && ell % 16 == 0 &&
         (reinterpret_cast<uintptr_t>(f.b[0]) & 7) == 0 && link_ctx_mma_smem(w0, ell, d_c) <= 200 * 1024;
}

lime_status launch_link_ctx_mma(const float* first, const void* user_ctx, int d_c, const void* W0c, int w0, int B, int ell, int d,
                                const FfnArgs& f, float* out, cudaStream_t st) {
  if (B == 0) return LIME_OK;
  static bool smem_set[kMaxDeviceOrdinals] = {};
  lime_status s = ensure_dynamic_smem((const void*)k_link_ctx_mma, 200 * 1024, smem_set);
  if (s != LIME_OK) return s;
  ProfScope _p("k_link_ctx_mma", st);
  launch_pdl(k_link_ctx_mma, dim3((unsigned)B, (unsigned)(d / CX_COLS)), dim3(CX_THREADS), link_ctx_mma_smem(w0, ell, d_c), st, first,
             (const __nv_bfloat16*)user_ctx, d_c, (const __nv_bfloat16*)W0c, w0, ell, d, (const __nv_bfloat16*)f.W[0], f.b[0], out);
  LIME_LAUNCH_CHECK("k_link_ctx_mma");
  return LIME_OK;
}

}  // namespace lime
