// Shared declarations of the CUDA side of the LIME hot path (sm_100a).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lime.h"

namespace lime {

constexpr int kSMs = 148;  // B200: 2 dies x 74 SMs; grids of persistent kernels are sized from this

// ----------------------------------------------------------------------------- storage helpers
template <typename T> struct Store;
template <> struct Store<float> {
  static __device__ __forceinline__ float ld(const float* p) { return *p; }
  static __device__ __forceinline__ void st(float* p, float v) { *p = v; }
};
template <> struct Store<__nv_bfloat16> {
  static __device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
  static __device__ __forceinline__ void st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
};

__device__ __forceinline__ float silu_f(float x) { return x / (1.0f + __expf(-x)); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Largest b in [0, B) with start[b] <= x, for a non-decreasing start[0..B] (start[0] = 0).
__device__ __forceinline__ int upper_user(const int32_t* __restrict__ start, int B, int x) {
  int lo = 0, hi = B;  // invariant: start[lo] <= x, answer in [lo, hi)
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (start[mid] <= x) lo = mid; else hi = mid;
  }
  return lo;
}

// Which users get a cluster of blocks each: those of more than `base` tokens, the line doubling until at most `most` are left.  The
// host knows the total length only, so the blocks find the line.  Every thread of the block calls these; `word` is a word of its
// shared memory (a static one would not fit beside all of it taken dynamically).
__device__ __forceinline__ int long_user_line(const int32_t* __restrict__ off, int B, int base, int most, int* word) {
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {
    int line = base;
    for (;; line *= 2) {
      int n = 0;
      for (int b = lane; b < B; b += 32) n += off[b + 1] - off[b] > line;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
      if (n <= most || line > (1 << 29)) break;
    }
    if (lane == 0) *word = line;
  }
  __syncthreads();
  const int line = *word;
  __syncthreads();
  return line;
}
// the k-th of those users (from 0); -1: there are not that many
__device__ __forceinline__ int nth_long_user(const int32_t* __restrict__ off, int B, int base, int most, int k, int* word) {
  const int line = long_user_line(off, B, base, most, word), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) *word = -1;
  __syncthreads();
  if (threadIdx.x < 32)
    for (int b0 = 0; b0 < B && k >= 0; b0 += 32) {
      const int b = min(b0 + lane, B - 1);
      const unsigned m = __ballot_sync(0xffffffffu, b0 + lane < B && off[b + 1] - off[b] > line);
      if (((m >> lane) & 1u) && __popc(m & ((1u << lane) - 1u)) == k) *word = b;
      k -= __popc(m);
    }
  __syncthreads();
  return *word;
}
// barrier of all threads of a cluster; what they wrote before it is visible behind it, to the cluster
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the same shared-memory address in block `rank` of the cluster, as a generic pointer
template <typename T>
__device__ __forceinline__ const T* cluster_peer(const T* p, int rank) {
  uint64_t r;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"((uint64_t)p), "r"(rank));
  return reinterpret_cast<const T*>(r);
}

// ----------------------------------------------------------------------------- context
struct Ctx {
  lime_config cfg;
  lime_weights w;
  bool have_weights;
  int device;
  int cand_heads;   // heads of the candidate side: 1 (one weight row per candidate) or H (one per head)
  int ell_c;        // weight columns per candidate = cand_heads * ell; also the rows of a user's link states
  float* keff;      // [ell x d] fp32: (L W_K^c) W_Q^c^T * cand_scale, the effective link keys of Eq. 4
  void* keff_hl;    // [2 ell x d] bf16: keff split into a rounded part and its remainder (tensor-core precompute)
  float* links32;   // [ell x d] fp32 copy of L (layer-1 link rows when no L^C is given)
  int tc_mode;                   // 0: generic kernels; 1: tensor-core layer kernels at d = 128; 2: at d = 256
  void* WoT[LIME_MAX_LAYERS];    // tensor-core path, per layer (NULL otherwise): W_o transposed [d x d_ff] bf16,
  void* WprepT[LIME_MAX_LAYERS]; //   folded PREP operand (k_link_prep.cu), folded link-row GLU operand [2*d_ff x H*d],
  void* WpostT[LIME_MAX_LAYERS]; //   and (tc_mode 2) [W_g | W_u] transposed [2*d_ff x d]
  void* WguT[LIME_MAX_LAYERS];
  bool side256;                  // d = 256 with 32 links: link side by k_link_side_d256.cu, weights unfolded:
  void* side_w;                  //   one buffer, per layer W_Q^T | W_K^T | W_V^T | W_g^T | W_u^T | W_o^T, then the sh_ operands
  // link-side operands of the first layer for the shared links T^0 = L (weights only, formed at lime_set_weights)
  void *sh_That, *sh_Q2, *sh_K2, *sh_G2t, *sh_U2t, *sh_V2t;
  float *sh_cQ, *sh_cK;
  // feed-forward networks (k_ffn_simt.cu, k_score_head_tc.cu): the caller's description plus derived device data
  bool have_head, have_ctx_mlp;
  lime_ffn head, ctx_mlp;
  int ctx_dc;            // context features per user
  void* head_W1bT;       // [w0 x d] bf16: the T half of the head's first layer, transposed (tensor-core path)
  void* head_W1aT;       // [w0 x d] bf16: its O half, transposed (B operand of the per-user link-state product)
  float* head_w2;        // [w_last] fp32 copy of the head's last layer
  float* ctx_first;      // [ell x w0] fp32: (L W_0[:d]) + b_0 of the context MLP
  int* dev_err;     // device word: 0, or the code of the first bounded wait that gave up in a kernel of this context
  float attn_scale, cand_scale, ln_eps;
  int d_ff, d_h;
};

// record a CUDA error for lime_last_cuda_error(); returns LIME_CUDA_ERROR
lime_status cuda_fail(cudaError_t e, const char* where);
#define LIME_CUDA(expr)                                          \
  do {                                                           \
    cudaError_t _e = (expr);                                     \
    if (_e != cudaSuccess) return ::lime::cuda_fail(_e, #expr);  \
  } while (0)
#define LIME_LAUNCH_CHECK(name)                                  \
  do {                                                           \
    cudaError_t _e = cudaGetLastError();                         \
    if (_e != cudaSuccess) return ::lime::cuda_fail(_e, name);   \
  } while (0)

// ----------------------------------------------------------------------------- programmatic dependent launch
// The kernels of one step run back to back on one stream.  Launched with the programmatic-serialization attribute, a
// kernel's CTAs may become resident while its predecessor still runs (as soon as every CTA of the predecessor has
// executed pdl_launch_dependents() or exited), set up their barriers and tensor memory, and then block in pdl_wait()
// until the predecessor has completed and its writes are visible.  Rules kept by every kernel launched this way:
//  - nothing produced by an earlier kernel is read, and no global memory is written, before pdl_wait().  Two scorers (k_score_rows.cu,
//    k_score_tc.cu) do ask L2 for candidate rows before it: prefetches hold no value, and ids read that early only choose
//    what to prefetch, past L1, and are read again afterwards;
//  - a kernel that allocates tensor memory calls pdl_launch_dependents() only after its allocation, so a dependent CTA
//    that shares the SM can never hold the columns a CTA of the running kernel still waits for.
//  - no thread leaves a kernel ahead of pdl_wait(), on an error either: a kernel all of whose CTAs have left is complete although its
//    predecessor may still run, and whoever waits for it would take that predecessor for complete too.
// A kernel launched the ordinary way after such a kernel still waits for its completion, as always.
//
// A history update may run BESIDE the link side of its layer, launched right before it (`early`): the two read the attention's
// result and the layer's operands and write different things.  It reads what the kernels up to the attention wrote without a wait of
// its own, and waits at its end, so that whoever waits for the update has waited for the link side as well.  The programming model
// gives a dependent no view of anything before its own wait; that the early reads are sound rests on three things here:
//  - order: the launch right before the update is a kernel of the link side (the merge of the partials comes ahead of that one), every
//    thread of which signals behind its own wait.  So when the update's CTAs start, a wait for everything up to the attention has
//    returned, which is to say those kernels are complete and their writes have been flushed to L2;
//  - place: what it reads that early comes from L2, by TMA or by loads past L1, never through a line that L1 may have kept from before;
//  - buffers: nothing that runs beside it writes what it reads (operands of consecutive layers alternate or are written behind it).
// A kernel put between the attention and the update, or an exit of a link-side kernel ahead of its wait, breaks the first.
// (tests/test_launch_order.py holds the sources against these rules.)
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// the 128-byte line at `p` into L2
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// a row of `bytes`
__device__ __forceinline__ void prefetch_l2_row(const void* p, int bytes) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p);
  for (uintptr_t l = a & ~(uintptr_t)127; l < a + bytes; l += 128) prefetch_l2(reinterpret_cast<const void*>(l < a ? a : l));
}
#endif
#ifdef __CUDACC__
// First tile of block `cta` when the `n` tiles are split in order among `grid` blocks, of which the last `late` start when the others
// are `late_by` tiles ahead (they wait for the SMs that the link side holds).
__device__ __forceinline__ int early_first_tile(int cta, int grid, int n, int late, int late_by) {
  const int64_t first = grid - late, share = n + (int64_t)late * late_by;                    // share / grid: tiles of an early block
  if (share < (int64_t)grid * late_by) return cta >= first ? n : (int)(cta * (int64_t)n / first);
  const int64_t behind = cta > first ? (cta - first) * (int64_t)grid * late_by : 0;
  return (int)((cta * share - behind) / grid);
}
#endif
bool pdl_enabled();      // environment LIME_PDL=0 turns the attribute off (every launch then serialises fully)
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ----------------------------------------------------------------------------- per-kernel event timing
// While a profile is open (lime_profile_start .. lime_profile_stop) every launcher brackets its kernel with two
// CUDA events on the launching stream.  Closed, a scope costs one predictable branch.
struct ProfScope {
  ProfScope(const char* name, cudaStream_t st);
  ~ProfScope();
  int slot;
  cudaStream_t st;
};

// ----------------------------------------------------------------------------- kernel launchers (host)
// Each returns LIME_OK or a status; all launch on `st` and never synchronise.

lime_status launch_offsets(const int32_t* len, int B, int32_t* off, cudaStream_t st);

lime_status launch_gather(int dtype, const void* table, int64_t V, int d, const int32_t* ids, int64_t total,
                          void* out, int32_t* dev_flag, cudaStream_t st);
// the same lookup with the non-affine LayerNorm of the row applied before it is stored
lime_status launch_gather_ln(int dtype, const void* table, int64_t V, int d, float eps, const int32_t* ids, int64_t total,
                             void* out, int32_t* dev_flag, cudaStream_t st);

// Work lists of the XOR layers in one launch: chunk_start[b] = sum_{b' < b} ceil(len_b' / chunk) and
// tile_start[b] = sum_{b' < b} ceil(len_b' / tile) for b = 0..B; chunk_user[item] = user of the chunk item (may be NULL);
// *merge_needed (may be NULL) = 1 if any user has several chunks or none (its attention rows come from the merge step)
// Optional: the chunk items dealt to n_groups groups of CTAs with even token-tile counts (tiles of att_tile tokens);
// group_start == NULL: not wanted.  group_start[n_groups + 1], group_items[items], scratch[4 x items].
struct GroupSchedule {
  int n_groups = 0, att_tile = 0;
  bool walk = false;                // a single user may have many items: they are listed by its warp
  int32_t* group_start = nullptr; int32_t* group_items = nullptr; int32_t* scratch = nullptr;
};
// How long the work items of the links <- history attention are: `tokens`, or `short_tokens` (0: never) where some history is over
// twice as long as that and the histories longer than it make no more than `short_items` such chunks.
// Where some history is longer than `tokens` and not the short ones are taken, the length of up to 64 tiles of 128 that fits
// the `fit_groups` groups of CTAs best, of at most `fit_items` items (fit_groups 0: `tokens` as it is).
struct ChunkRule { int tokens = 0, short_tokens = 0, short_items = 0, fit_groups = 0, fit_items = 0; };
lime_status launch_layer_schedules(const int32_t* off, int B, const ChunkRule& chunk, int32_t* chunk_out, int32_t* chunk_start, int tile, int32_t* tile_start,
                                   int32_t* chunk_user, int32_t* merge_needed, const GroupSchedule& gs, cudaStream_t st);

// Y[r, n] (+)= epilogue( LN?(X[r, :]) . W[:, n] ) for up to three weight matrices sharing X.
struct LinearArgs {
  const void* X; int x_dtype;   // [M x K], lime_dtype
  int64_t M; int K; int N;      // every W is [K x N], stored w_dtype; a NULL W means identity (K == N)
  const void* W[3]; int w_dtype;
  void* Y[3]; int y_dtype;      // outputs [M x N] each (ldy = N)
  int n_out;                    // 1..3 (ignored when glu)
  int ln; float ln_eps;         // LayerNorm rows of X first
  int glu;                      // 1: Y[0] = SiLU(X W[0]) * (X W[1])
  int accumulate;               // 1: Y[0] += result (y_dtype must be F32, n_out == 1)
  const float* also_add_to;     // unused (reserved)
};
lime_status launch_linear_simt(const LinearArgs& a, cudaStream_t st);

// link <- history attention partials: per (user, chunk of `chunk` tokens, head, link row): running max, sum,
// un-normalised weighted values.
struct AttnLinkArgs {
  const float* QT; int64_t qt_user_stride;   // [B x ell x d] fp32 (stride 0: shared)
  const void* KS; const void* VS; int s_dtype; // [total x d]
  const int32_t* off; int B; int64_t total;
  int ell, d, H; int phi; float scale;
  int chunk; const int32_t* chunk_start; int n_chunk_upper;  // work list from launch_layer_schedules
  float* part_m; float* part_s; float* part_acc;             // [n_chunk_upper x H x ell], same, [.. x d_h]
  float* AT;                                                  // out [B x ell x d] fp32
};
lime_status launch_attn_link_simt(const AttnLinkArgs& a, cudaStream_t st);
lime_status launch_attn_link_merge(const AttnLinkArgs& a, cudaStream_t st);

// history <- links attention: AS[t, :] = phi(Q[S]_t K[T]^T) V[T] per head, over the ell links of t's user
struct AttnHistArgs {
  const void* QS; void* AS; int s_dtype;     // [total x d]; AS may alias QS
  const float* KT; const float* VT; int64_t t_user_stride;  // [B x ell x d] fp32
  const int32_t* off; int B; int64_t total;
  int ell, d, H; int phi; float scale;
  int tile; const int32_t* tile_start; int n_tile_upper;
};
lime_status launch_attn_hist_simt(const AttnHistArgs& a, cudaStream_t st);

// out[r, :] (storage dtype) = in[r, :] fp32, optionally accumulate into acc fp32 first
lime_status launch_cast_rows(const float* in, int64_t n, void* out, int dtype, cudaStream_t st);
lime_status launch_axpy(const float* x, float* y, int64_t n, int zero_first, cudaStream_t st);
lime_status launch_widen(const void* in, int dtype, float* out, int64_t n, cudaStream_t st);

// candidate -> link weights: W[c, :] = softmax_l( <T_c, keff_l> )  (keff already carries cand_scale); `rows` keys
// in groups of `ell` (one group per head of the candidate side), the softmax inside each group
lime_status launch_precompute(int dtype, const void* cand, int64_t M, int d, int rows, int ell, const float* keff,
                              void* out_w, cudaStream_t st);
// keff = ((L Wk) Wq^T) * scale, fp32 [heads * ell x d]: one key per link, or per (head, link) restricted to the
// head's columns; the buffer holds 2 * heads * ell * d floats
lime_status launch_keff(int dtype, const void* L, const void* Wk, const void* Wq, int ell, int d, int heads, float scale,
                        float* keff, cudaStream_t st);
// link states for the per-head candidate side: out[b, h * ell + l, :] = src[b, l, :] on head h's columns, 0 elsewhere
lime_status launch_expand_heads(const float* src, int64_t rows_in, int ell, int d, int heads, void* out, int dtype, cudaStream_t st);

// bf16 precompute on tcgen05 tensor cores (ell in {16,32,64,128}, d % 64 == 0); keff_hl from launch_keff_split
// `ell` keys in all, softmax per group of `group` consecutive keys (group == ell: one softmax per row)
bool precompute_tc_supported(int dtype, int d, int ell, int group);
lime_status launch_keff_split(const float* keff, int ell, int d, void* keff_hl, cudaStream_t st);
lime_status launch_precompute_tc(const void* cand, int64_t M, int d, int rows, int group, const void* keff_hl, void* out_w,
                                 int* err, cudaStream_t st);

struct ScoreArgs {
  const void* LS; const void* W; const void* T; int dtype;
  int B; int ell, d;
  const int32_t* cand_off; int C; int64_t total;
  const int32_t* cand_ids;      // nullable; with ids, W and T have `corpus_rows` rows and ids outside [0, corpus_rows) score 0
  int64_t corpus_rows;
  int32_t* dev_flag;            // nullable: lowered to the smallest slot whose id was out of range
  float* logits;
  int64_t ldw, ldt;             // row pitch of W and T in elements; 0 = dense (ell, d).  Packed corpus records: d + ell both
};
// out[v, :] = [ emb[v, 0..d) | w[v, 0..ell) ]: one record per item of the corpus caches (k_cand_simt.cu)
lime_status launch_pack_corpus(int dtype, const void* emb, const void* w, int64_t V, int d, int ell, void* out, cudaStream_t st);
lime_status launch_score_simt(const ScoreArgs& a, cudaStream_t st);
// bf16 streaming scorer on tcgen05 tensor cores (fixed C per user, dense rows, ell in {16,32,64,128}, d % 64 == 0)
bool score_tc_supported(const ScoreArgs& a);
lime_status launch_score_tc(const ScoreArgs& a, int* err, cudaStream_t st);
// the same with rows taken from corpus-level caches by cand_ids (fixed C per user), k_score_gather_tc.cu
bool score_gather_tc_supported(const ScoreArgs& a);
lime_status launch_score_gather_tc(const ScoreArgs& a, int* err, cudaStream_t st);

// warp-level scorer: by id, ragged lists, small widths (bf16, d in {32, 64, 128, 256}, ell in {8, 16, 32, 64}; fp32, d in {32, 64}), k_score_rows.cu
bool score_rows_preferred(const ScoreArgs& a);
// candidate -> link weights of narrow models, same design (bf16 d = 32; fp32 d = 32, 64)
bool precompute_rows_supported(int dtype, int d, int rows, int group);
lime_status launch_precompute_rows(int dtype, const void* cand, int64_t M, int d, int ell, const float* keff, const void* keff_hl, void* out_w, cudaStream_t st);
lime_status launch_score_rows(const ScoreArgs& a, cudaStream_t st);

// the whole encode of a narrow model (bf16, d = d_ff = 32) in one launch, one block per user (k_encode_small.cu)
struct EncodeSmallArgs {
  const void* hist; const int32_t* off; int B; int64_t total;
  const float* links; int links_per_user;      // T^0: [ell x d] fp32, or [B x ell x d]
  const lime_weights* w;                       // as the caller gave them
  int H, ell, n_layers, ln, hist_ln, silu; float eps, scale;
  void* scratch;                               // [total x d] bf16, for histories beyond shared memory
  void* link_states; float* lp;                // bf16 link states, or (link_states NULL) L^P in fp32
};
bool encode_small_supported(int dtype, int d, int d_ff, int H, int ell, int gated_mlp);
lime_status launch_encode_small(const EncodeSmallArgs& a, cudaStream_t st);
// the same for fp32 storage at d = d_ff = 64, a cluster of blocks per user; L^P to a.lp (k_encode_f32.cu)
bool encode_f32_supported(int dtype, int d, int d_ff, int H, int ell, int gated_mlp);
lime_status launch_encode_f32(const EncodeSmallArgs& a, int* err, cudaStream_t st);

// one-thread kernel whose only wait can never be satisfied (self-test of the bounded waits, tc_host.cu)
lime_status launch_wait_expiry(int* err, uint64_t limit_ns, int code, cudaStream_t st);

// ---- feed-forward networks: Eq. 2 and the interaction network of Sec. 3.3 ------------------------------------------
// layers after the first (whose input is a concatenation and is handled split): W[i] [in_w[i] x out_w[i]], b[i] nullable
struct FfnArgs {
  int n_layers;
  int in_w[LIME_FFN_MAX_HIDDEN + 1], out_w[LIME_FFN_MAX_HIDDEN + 1];
  const void* W[LIME_FFN_MAX_HIDDEN + 1];
  const float* b[LIME_FFN_MAX_HIDDEN + 1];
};
// Y = X . W (+ bias) for a few rows: fp32 [M x N]
lime_status launch_rows_times_w(const void* X, int x_dtype, int64_t M, int K, const void* W, int w_dtype, int ldw, int N,
                                const float* bias, float* Y, const char* name, cudaStream_t st);
lime_status launch_link_ctx_mlp(int dtype, const float* first, const void* user_ctx, int d_c, const void* W0c, int w0, int B,
                                int ell, const FfnArgs& f, float* out, cudaStream_t st);
// the same with one hidden layer on tensor cores (k_link_ctx_mma.cu)
bool link_ctx_mma_supported(int dtype, int d_c, int w0, int ell, int d, const FfnArgs& f);
lime_status launch_link_ctx_mma(const float* first, const void* user_ctx, int d_c, const void* W0c, int w0, int B, int ell, int d,
                                const FfnArgs& f, float* out, cudaStream_t st);
// generic scorer through the interaction network; LSW fp32 [B x ell x w0], W0t = rows d.. of the first layer [d x w0]
lime_status launch_score_head_simt(const ScoreArgs& a, const float* LSW, const void* W0t, const float* b0, int w0,
                                   const FfnArgs& f, cudaStream_t st);
// one hidden layer of n1 units on tensor cores; LSWt bf16 [B x n1 x ell], W1bT bf16 [n1 x d], w2 fp32 [n1]
struct ScoreHeadArgs {
  const void* LSWt; const void* W1bT; const float* b1; const float* w2; const float* b2; int n1;
};
bool score_head_tc_supported(const ScoreArgs& a, int n1);
int score_head_tc_terms(const ScoreArgs& a, int n1);      // bf16 pieces per value of LSWt [B][n1][terms][ell]
lime_status launch_score_head_tc(const ScoreArgs& a, const ScoreHeadArgs& h, int* err, cudaStream_t st);

// three hidden layers (w0 <= 512, 128, 64) at d = 32, any candidate form (k_score_mlp3.cu)
bool score_mlp3_supported(const ScoreArgs& a, const lime_ffn& f);
lime_status launch_score_mlp3(const ScoreArgs& a, const lime_ffn& f, cudaStream_t st);

// ---- tensor-core XOR layer (bf16, d = d_ff = 128, H * ell = 128) ----------------------------------------------
// plain_v: WprepT's third segment is W_V^T (link values formed as they stand) instead of the folded gate / up products
lime_status launch_fold_weights(const void* Wq, const void* Wk, const void* Wv, const void* Wg, const void* Wu, int d,
                                int H, int f, float scale, int plain_v, void* WprepT, void* WpostT, cudaStream_t st);
lime_status launch_ln_rows_bf16(const float* T, int64_t rows, int d, int ln, float eps, void* out, cudaStream_t st);
lime_status launch_link_attn_merge_norm(const int32_t* chunk_start, const int32_t* merge_needed, int B, int ell, int d, int H,
                                        const float* part_m, const float* part_s, const float* part_acc, void* Ohat, cudaStream_t st);
// n square matrices [d x d] (NULL: identity), transposed one after the other into out
lime_status launch_transpose_square_bf16(const void* const* W, int n, int d, void* out, cudaStream_t st);
lime_status launch_transpose_bf16(const void* W, int rows, int cols, void* WT, cudaStream_t st);

// link-row GEMMs on tensor cores (k_gemm_tc.cu); A [M x K] bf16 row-major, Bt [N x K] bf16 (weights, pre-folded)
struct LinkGemmArgs {
  const void* A; int64_t M; int K; const void* Bt; void* out;   // K = d
  int ell, H, need_hist;                       // PREP: rows are (user, link); need_hist = also K2 and G2t / U2t (or V2t)
  int f, plain_v;                              // GatedMLP width; plain_v: V2t [users x d x ell] instead of G2t / U2t
  void *Q2, *K2, *G2t, *U2t, *V2t; float *cQ, *cK;   // PREP outputs (cQ / cK nullable; only formed with d = 128)
  int* err;
};
lime_status launch_gemm_prep(const LinkGemmArgs& a, cudaStream_t st);
// A [M x K] . Bt^T, Bt [n_cols x K] (bf16, K % 64 == 0, 16-byte aligned): `terms` bf16 pieces per value, transposed per group
// of rows: out_t [M / group][n_cols][terms][group]
lime_status launch_gemm_rows_t(const void* A, int64_t M, int K, const void* Bt, int n_cols, int group, int terms, void* out_t, int* err,
                               const char* name, cudaStream_t st);

// GatedMLP on link rows fused with its consumers (k_link_mlp_tc.cu); d = d_ff in {128, 256}
struct LinkMlpArgs {
  const void* Ohat; int64_t M; int K; int d;   // attention rows [M x K = H*d] bf16
  const void* WpostT; const void* WoT;         // folded [2f x H*d] (d = 128) and transposed [d x f] weights, bf16
  const void *WvT, *WguT;                      // d = 256: W_V transposed [d x d], [W_g | W_u] transposed [2f x d]
  float* T_out;                                // nullable: the layer's link rows, fp32 [M x d]
  float* LP; int lp_accumulate;                // nullable running sum of Eq. 8 (0: assign, 1: add)
  void* That_next;                             // nullable: bf16 LN(T) for the next layer's link-side GEMM
  void* Q2; const void* WprepT; int ell;       // d = 128, nullable: instead of it the next layer's queries [M / ell x K/d*ell x d]
  void* link_states;                           // nullable: bf16 copy of LP after this layer, which is then not stored
  int ln; float ln_eps;
  int* err;
};
lime_status launch_link_mlp_tc(const LinkMlpArgs& a, cudaStream_t st);

struct LinkAttnArgs {
  const void* hist; int64_t total;          // [total x d] bf16
  const void* Q2; const float* cQ;          // folded link queries [users x H*ell x d] bf16 and their row sums
  const int32_t* off; const int32_t* chunk_start; const int32_t* chunk; int B, n_chunk_upper;   // chunk: tokens per work item
  const int32_t* chunk_user;                // [items] user of each (user, chunk) work item
  const int32_t* group_start; const int32_t* group_items; int n_groups;   // balanced deal of the items (d = 256 kernel)
  int ell, d, H, shared, ln; float ln_eps;
  int silu;                                 // 1: SiLU(s) / N(U) instead of softmax (Algorithm 2)
  float *part_m, *part_s, *part_acc;        // scratch: [items x H*ell], same, [items x H*ell x d]
  void* Ohat;                               // [B*ell x H*d] bf16: rows of users whose history is one chunk
  float2* stats_out;                        // nullable, ln only: {rstd, mean} of every history row, for the history update
  int* err;
};
bool link_attn_tc_supported(int dtype, int d, int H, int ell, int phi);
int link_attn_d256_groups(int n_chunk_upper, int H, int ell);   // groups of CTAs (one CTA per 128-row block) of that kernel
lime_status launch_link_attn_tc(const LinkAttnArgs& a, cudaStream_t st);
lime_status launch_link_attn_d128_tmem(const LinkAttnArgs& a, cudaStream_t st);   // the same for rows LayerNorm-ed already (a.ln must be 0)

// An update that runs beside the link side of its layer: 1, and how many of its blocks start later and by how much (see above).
struct BesideLinkSide { int early, late, late_by; };
constexpr int kEarlyUsers = 1024;         // at most: their offsets are staged in shared memory, past L1
struct HistUpdateArgs {
  const void* hist_in; void* hist_out; int64_t total;
  const void *K2, *G2t, *U2t; const float* cK; const void* WoT;   // WoT [d x f] bf16 (W_o transposed)
  const int32_t* off; const int32_t* tile_start; int B, n_tile_upper;
  int ell, shared, ln; float ln_eps;    // ln: apply LayerNorm to the rows read (0 when they were stored normalised)
  int out_ln;                           // 1: store LayerNorm(S') instead of S'
  int silu;                             // 1: SiLU(s) / ell instead of the per-head softmax (Algorithm 2)
  const float2* stats_in;               // nullable, ln only: {rstd, mean} of every row read, as left by the attention kernel
  BesideLinkSide beside;                // k_hist_update_tmem_tc.cu only
  int* err;
};
bool hist_update_tmem_supported(int dtype, int d, int f, int H, int ell, int phi, int gated_mlp);     // H * ell = 128 or 256
lime_status launch_hist_update_tmem(const HistUpdateArgs& a, int H, cudaStream_t st);                 // a.ln: with stats_in and cK
// the same step for H * ell = 512 (link-side operands streamed per tile, k_hist_update2_tc.cu)
bool hist_update2_tc_supported(int dtype, int d, int f, int H, int ell, int phi, int gated_mlp);
lime_status launch_hist_update2_tc(const HistUpdateArgs& a, cudaStream_t st);

// ---- tensor-core XOR layer at d = d_ff = 256 (bf16; ell = 64 with H in {2, 4, 8}, ell = 32 with H in {4, 8}; history rows LayerNorm-ed already) ----
bool link_attn_d256_tc_supported(int dtype, int d, int H, int ell, int phi);
lime_status launch_link_attn_d256_tc(const LinkAttnArgs& a, cudaStream_t st);   // a.ln must be 0

// link side of a layer at d = 256, 32 links: merged attention rows -> T and its consumers, and (or) T -> the next layer's operands
struct LinkSide256Args {
  int users, H;
  const void* Ohat; const float *part_m, *part_s, *part_acc; const int32_t* chunk_start;   // Ohat NULL: T is given
  const float* T_in; int t_shared;
  const void *WvT, *WguT, *WoT;                             // this layer's, transposed (needed with Ohat)
  const void *WqT, *WkT, *WvT_next, *Wq, *Wk;               // next layer's, transposed and as stored (WqT NULL: no operands)
  int need_hist, lp_accumulate, ln;
  float *T_out, *LP;                                        // nullable
  void *link_states, *Q2, *K2, *V2t;                        // link_states (nullable): bf16 L^P instead of LP
  float scale, eps;
  int* err;
};
bool link_side_d256_supported(int d, int d_ff, int H, int ell);
lime_status launch_link_side_d256(const LinkSide256Args& a, cudaStream_t st);
int link_side_d256_blocks(int users);

// the same for d = 128 with four heads and few link rows: merge, GatedMLP and the next layer's operands (k_link_side_d128.cu)
struct LinkSide128Args {
  int users, ell;
  const void* Ohat; const float *part_m, *part_s, *part_acc; const int32_t* chunk_start;
  const void *WpostT, *WoT, *WprepT;                        // this layer's GatedMLP; next layer's operands (NULL: none wanted)
  int need_hist, lp_accumulate, ln;
  float* LP;                                                // nullable
  void *link_states, *Q2, *K2, *G2t, *U2t;                  // link_states (nullable): bf16 L^P instead of LP
  float eps;
  int* err;
};
bool link_side_d128_wanted(int d, int d_ff, int H, int ell, int64_t users);
lime_status launch_link_side_d128(const LinkSide128Args& a, cudaStream_t st);
int link_side_d128_blocks(int64_t rows);

struct HistUpdate256Args {
  const void* hist_in; void* hist_out; int64_t total;
  const void* K2;                       // folded link keys [users x H*ell x d] bf16
  const void* V2t;                      // link values, transposed [users x d x ell] bf16
  const void* WguT; const void* WoT;    // [W_g | W_u]^T [2f x d] and W_o^T [d x f], bf16
  const int32_t* off; const int32_t* tile_start; int B, n_tile_upper;
  int H, ell, shared;
  int out_ln;                           // 1: store LayerNorm(S') instead of S'
  int silu;                             // 1: SiLU(s) / ell instead of the per-head softmax (Algorithm 2)
  float ln_eps;
  BesideLinkSide beside;
  int* err;
};
bool hist_update_d256_tc_supported(int dtype, int d, int f, int H, int ell, int phi, int gated_mlp);
lime_status launch_hist_update_d256_tc(const HistUpdate256Args& a, cudaStream_t st);

}  // namespace lime
