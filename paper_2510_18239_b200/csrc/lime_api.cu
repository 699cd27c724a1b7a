// C-ABI entry points: argument validation, workspace carving and launch sequencing.  No arithmetic of the
// method lives here; every step runs in the kernels of this directory.
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>

#include "lime_common.cuh"
#include "tc_common.cuh"

namespace lime {

static thread_local char g_err[256] = "";

lime_status cuda_fail(cudaError_t e, const char* where) {
  snprintf(g_err, sizeof(g_err), "%s: %s (%s)", where, cudaGetErrorName(e), cudaGetErrorString(e));
  return LIME_CUDA_ERROR;
}

// ---- per-kernel event timing (process-wide, single-threaded use) -------------------------------------------
struct ProfState {
  bool open = false;
  int capacity = 0, count = 0;
  cudaEvent_t* ev = nullptr;      // 2 per record
  const char** names = nullptr;
};
static ProfState g_prof;

ProfScope::ProfScope(const char* name, cudaStream_t s) : slot(-1), st(s) {
  if (!g_prof.open || g_prof.count >= g_prof.capacity) return;
  slot = g_prof.count++;
  g_prof.names[slot] = name;
  cudaEventRecord(g_prof.ev[2 * slot], st);
}
ProfScope::~ProfScope() {
  if (slot >= 0) cudaEventRecord(g_prof.ev[2 * slot + 1], st);
}

static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
static inline size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }
// Memory of weight copies comes from a pool per device: a cudaMalloc of 2 MB or more maps fresh pages every time (0.34 ms).
// The pool keeps at most 64 MB that no context uses, and gives all of it back when the device's last context with such
// copies goes.
struct WeightPool {
  std::mutex lock;
  cudaMemPool_t pool = nullptr;
  int users = 0;
};
static WeightPool g_weight_pool[kMaxDeviceOrdinals];
static cudaError_t weight_alloc(int device, void** p, size_t bytes, cudaStream_t st) {
  if (device < 0 || device >= kMaxDeviceOrdinals) return cudaErrorInvalidDevice;
  WeightPool& w = g_weight_pool[device];
  std::lock_guard<std::mutex> hold(w.lock);
  if (w.pool == nullptr) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    cudaError_t e = cudaMemPoolCreate(&w.pool, &props);
    uint64_t keep = 64ull << 20;
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(w.pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) return e;
  }
  const cudaError_t e = cudaMallocFromPoolAsync(p, bytes, w.pool, st);
  if (e == cudaSuccess) ++w.users;
  return e;
}
static void weight_free(int device, void* p) {
  if (p == nullptr) return;
  // Memory of a pool is freed in stream order: cudaFree of it does not wait for kernels that may still read it, as that of a plain
  // allocation does.  So this waits, on the device that owns it.
  int current = device;
  cudaGetDevice(&current);
  if (current != device) cudaSetDevice(device);
  cudaDeviceSynchronize();
  cudaFree(p);
  if (current != device) cudaSetDevice(current);
  WeightPool& w = g_weight_pool[device];
  std::lock_guard<std::mutex> hold(w.lock);
  if (--w.users == 0) cudaMemPoolTrimTo(w.pool, 0);
}
static inline int elem_size(int dtype) { return dtype == LIME_F32 ? 4 : 2; }

// Tokens per work item of the link<-history attention: a power of two in [lo, hi] giving about three work items per
// SM (`row_blocks` items per chunk).  Every chunk of a multi-chunk history costs a set of fp32 partials and a pipeline
// refill, so long histories take long chunks.
static int pick_chunk(int64_t total_tokens, int row_blocks, int lo, int hi = 2048) {
  const int64_t target = total_tokens * row_blocks / (3 * kSMs);
  int c = lo;
  while (c < hi && c < target) c <<= 1;
  return c;
}

// Which kernels serve the XOR layers of this shape: 1 = the tensor-core kernels built for d = d_ff = 128, 2 = those
// built for d = d_ff = 256, 0 = the generic CUDA-core path.
static int tensor_core_mode(const lime_config& g, int d_ff) {
  if (link_attn_tc_supported(g.dtype, g.d, g.H, g.ell, g.phi) &&
      (hist_update_tmem_supported(g.dtype, g.d, d_ff, g.H, g.ell, g.phi, g.gated_mlp) ||
       hist_update2_tc_supported(g.dtype, g.d, d_ff, g.H, g.ell, g.phi, g.gated_mlp)))
    return 1;
  if (link_attn_d256_tc_supported(g.dtype, g.d, g.H, g.ell, g.phi) &&
      hist_update_d256_tc_supported(g.dtype, g.d, d_ff, g.H, g.ell, g.phi, g.gated_mlp))
    return 2;
  return 0;
}
// One launch for the whole encode, a block or a cluster per user, up to 2048 tokens a user on average (at that mean, 32 users: d = 32
// 178 us, generic kernels 1601; fp32 174 us, 815).  Single users may be far longer: these are given more blocks on the device, which
// knows the lengths (k_encode_small.cu, k_encode_f32.cu).
static bool encode_small_wanted(const Ctx* c, int32_t B, int64_t total) {
  const lime_config& g = c->cfg;
  return (encode_small_supported(g.dtype, g.d, c->d_ff, g.H, g.ell, g.gated_mlp) ||
          encode_f32_supported(g.dtype, g.d, c->d_ff, g.H, g.ell, g.gated_mlp)) && total <= 2048ll * B;
}
// d = 128 with few link rows: the link side of a layer is one kernel (k_link_side_d128.cu)
static bool few_link_rows(const Ctx* c, int64_t B) {
  return c->tc_mode == 1 && link_side_d128_wanted(c->cfg.d, c->d_ff, c->cfg.H, c->cfg.ell, B);
}
constexpr int kHistTile = 128;  // tokens per block of the history<-links attention

struct Workspace {
  // history rows, storage dtype
  void *S, *Q, *K, *V, *U;
  // link rows, fp32
  float *T, *QT, *KT, *VT, *AT, *UT, *LP, *LS32;
  int32_t *chunk_start, *tile_start, *chunk_user, *merge_needed;
  GroupSchedule groups;          // balanced deal of the chunk items (d = 256 kernels only)
  float *part_m, *part_s, *part_acc;
  // tensor-core path: folded link-side operands (bf16) and their row sums
  void *Q2, *K2, *G2t, *U2t, *V2t;
  void *K2b, *G2tb, *U2tb;       // few link rows: the history update's operands of every other layer
  float *cQ, *cK;
  float2* row_stats;   // LayerNorm {rstd, mean} of the history rows of the layer being processed
  void *That, *Ohat, *UTb;   // LN(T) [B*ell x d], merged attention rows [B*ell x H*d], GLU output [B*ell x d_ff] (bf16)
  ChunkRule chunk;
  int32_t* chunk_dev;            // the length that k_layer_schedules chose
  int n_chunk_upper, n_tile_upper;
  size_t bytes;
};

static Workspace carve(const Ctx* c, void* base, int32_t B, int64_t total) {
  Workspace w;
  const lime_config& g = c->cfg;
  const size_t es = elem_size(g.dtype);
  size_t o = 0;
  char* p = static_cast<char*>(base);
  auto take = [&](size_t nbytes) { void* r = p ? p + o : nullptr; o += align_up(nbytes); return r; };
  const size_t hd = (size_t)total * g.d * es, hf = (size_t)total * c->d_ff * es;
  w.S = take(hd); w.Q = take(hd); w.K = take(hd); w.V = take(hd); w.U = take(hf);
  const size_t ld = (size_t)B * g.ell * g.d * 4, lf = (size_t)B * g.ell * c->d_ff * 4;
  w.T = (float*)take(ld); w.QT = (float*)take(ld); w.KT = (float*)take(ld); w.VT = (float*)take(ld);
  w.AT = (float*)take(ld); w.UT = (float*)take(lf); w.LP = (float*)take(ld); w.LS32 = (float*)take(ld);
  w.chunk_start = (int32_t*)take((size_t)(B + 1) * 4);
  w.tile_start = (int32_t*)take((size_t)(B + 1) * 4);
  w.merge_needed = (int32_t*)take(4);
  const bool tc_link = c->tc_mode != 0;
  // tensor-core path: at least 4 token tiles per work item, one item per 128-row block of H * ell (at d = 256 a set of
  // partials is 4 x larger and the batches served have many users, so chunks may be longer still)
  // At least 2048 tokens once the users alone make 64 work items: splitting histories of some hundred tokens then evens out less
  // than the merge of the partials costs (100 users of 250..1000 tokens, two layers: 105 -> 87 us with 32 links, 142 -> 113 us
  // with 64).  With fewer users the split is what occupies the SMs (16 users of 375..1500 tokens: 57 us, 64 us unsplit).
  // But 512 where few histories are longer, however many users there are: one user of 2000 or 4000 tokens among 64 of 100 takes 74
  // and 76 us unsplit, 59 and 61 us split (with 64 links 80 -> 69, 85 -> 70 us; d = 256 187 -> 175, 204 -> 189 us).  Up to 64 such
  // work items the split wins or is even (100 users, 8 of them of 2000: 79 -> 69 us, 20 of 1500: 78 -> 74 us; with 64 links 91 -> 82
  // and 91 -> 93 us), beyond it loses (30 of 2000, 64 links: 114 -> 128 us; d = 256, 8 of 2000: 239 -> 246 us).
  // Only the device knows the lengths: k_layer_schedules decides.
  const int row_blocks = (g.H * g.ell + 127) / 128;
  const bool many = tc_link && (int64_t)B * row_blocks >= 64;
  w.chunk = ChunkRule{};
  w.chunk.tokens = tc_link ? pick_chunk(total, row_blocks, many ? 2048 : 512, c->tc_mode == 2 ? 4096 : 2048) : pick_chunk(total, 1, 64);
  if (many) { w.chunk.short_tokens = 512; w.chunk.short_items = 64 / row_blocks; }
  w.chunk_dev = (int32_t*)take(4);
  // d = 128: the items go round-robin to the groups of CTAs that run at once, so k_layer_schedules fits their length to these where the
  // histories are half an item long on average and the items more than the groups (one user of 30000 tokens, one round, three layers
  // with 64 links: 117.5 us, 122 fitted; 4 of 32768: 202.7, 184.8)
  const bool fit = c->tc_mode == 1 && 2 * total >= (int64_t)w.chunk.tokens * B && total * row_blocks > (int64_t)w.chunk.tokens * kSMs;
  const int64_t split_items = (total + w.chunk.tokens - 1) / w.chunk.tokens;
  w.n_chunk_upper = (int)((split_items > w.chunk.short_items ? split_items : w.chunk.short_items) + B);
  if (fit) { w.chunk.fit_groups = link_attn_d256_groups(w.n_chunk_upper, g.H, g.ell); w.chunk.fit_items = w.n_chunk_upper; }
  w.n_tile_upper = (int)((total + kHistTile - 1) / kHistTile + B);
  w.chunk_user = (int32_t*)take((size_t)w.n_chunk_upper * 4);
  if (c->tc_mode == 2) {
    w.groups.n_groups = link_attn_d256_groups(w.n_chunk_upper, g.H, g.ell);
    w.groups.att_tile = 96;
    w.groups.walk = split_items > 32;
    w.groups.group_start = (int32_t*)take((size_t)(w.groups.n_groups + 1) * 4);
    w.groups.group_items = (int32_t*)take((size_t)w.n_chunk_upper * 4);
    w.groups.scratch = (int32_t*)take((size_t)w.n_chunk_upper * 16);
  }
  const size_t rows = (size_t)w.n_chunk_upper * g.H * g.ell;
  w.part_m = (float*)take(rows * 4);
  w.part_s = (float*)take(rows * 4);
  w.part_acc = (float*)take(rows * (tc_link ? g.d : c->d_h) * 4);
  const size_t HL = (size_t)g.H * g.ell;
  w.Q2 = take((size_t)B * HL * g.d * 2); w.K2 = take((size_t)B * HL * g.d * 2);
  w.G2t = take((size_t)B * c->d_ff * HL * 2); w.U2t = take((size_t)B * c->d_ff * HL * 2);
  w.V2t = take((size_t)B * g.d * g.ell * 2);
  const size_t second = few_link_rows(c, B) ? (size_t)B * HL * 2 : 0;
  w.K2b = take(second * g.d); w.G2tb = take(second * c->d_ff); w.U2tb = take(second * c->d_ff);
  w.cQ = (float*)take((size_t)B * HL * 4); w.cK = (float*)take((size_t)B * HL * 4);
  w.row_stats = (float2*)take((size_t)total * 8);
  w.That = take((size_t)B * g.ell * g.d * 2); w.Ohat = take((size_t)B * g.ell * g.H * g.d * 2);
  w.UTb = take((size_t)B * g.ell * c->d_ff * 2);
  w.bytes = o;
  return w;
}

// True when the whole layer runs on the tensor-core kernels (their set-up data exists for this layer).
static bool layer_on_tensor_cores(const Ctx* c, int layer) {
  if (c->side256) return c->side_w && c->WoT[layer] && c->WguT[layer];
  return c->tc_mode != 0 && c->WoT[layer] && c->WprepT[layer] && (c->tc_mode == 1 ? c->WpostT[layer] : c->WguT[layer]);
}

// One XOR layer, tensor-core path: three link-row GEMMs around the two streaming attention kernels.
// Link-side operands of one layer's two attention directions (folded through the weights, k_link_prep.cu).
struct LinkOperands {
  const void *Q2, *K2, *G2t, *U2t, *V2t;   // G2t / U2t with tc_mode 1, V2t with tc_mode 2
  const float *cQ, *cK;
  int shared;                 // one set for every user (T^0 = L) or one per user
};

// The weights half of LinkSide256Args: the GatedMLP of `layer` (-1: none) and the operands of layer `next` (-1: none).
static LinkSide256Args side256_args(const Ctx* c, int layer, int next, int users) {
  LinkSide256Args a{};
  const size_t dd = (size_t)c->cfg.d * c->cfg.d * 2;
  a.users = users; a.H = c->cfg.H; a.ln = c->cfg.ln; a.eps = c->ln_eps; a.err = c->dev_err;
  a.scale = c->cfg.phi == LIME_PHI_SILU ? 1.0f : c->attn_scale * 1.4426950408889634f;
  if (layer >= 0) {
    a.WvT = static_cast<const char*>(c->side_w) + ((size_t)layer * 6 + 2) * dd;
    a.WguT = c->WguT[layer]; a.WoT = c->WoT[layer];
  }
  if (next >= 0) {
    const char* at = static_cast<const char*>(c->side_w) + (size_t)next * 6 * dd;
    a.WqT = at; a.WkT = at + dd; a.WvT_next = at + 2 * dd;
    a.Wq = c->w.Wq[next] ? c->w.Wq[next] : a.WqT;          // NULL stands for the identity, its own transpose
    a.Wk = c->w.Wk[next] ? c->w.Wk[next] : a.WkT;
  }
  return a;
}

// LN(links_in) -> bf16 -> PREP GEMM: the operands of `layer` for `rows` link rows, written to the given buffers.
static lime_status make_link_operands(Ctx* c, int layer, const void* That, int64_t rows, int need_hist, void* Q2, void* K2,
                                      void* G2t, void* U2t, void* V2t, float* cQ, float* cK, cudaStream_t st) {
  const lime_config& g = c->cfg;
  LinkGemmArgs gp{};
  gp.A = That; gp.M = rows; gp.K = g.d; gp.Bt = c->WprepT[layer]; gp.ell = g.ell; gp.H = g.H;
  gp.f = c->d_ff; gp.plain_v = c->tc_mode == 2;
  gp.need_hist = need_hist; gp.Q2 = Q2; gp.K2 = K2; gp.G2t = G2t; gp.U2t = U2t; gp.V2t = V2t;
  // the row sums serve the LayerNorm folded into the d = 128 kernels; the d = 256 kernels read normalised rows
  gp.cQ = c->tc_mode == 1 ? cQ : nullptr; gp.cK = c->tc_mode == 1 ? cK : nullptr;
  gp.err = c->dev_err;
  return launch_gemm_prep(gp, st);
}

// How the update of `tiles` tiles at most shares the SMs with a link side of `blocks` blocks, one per SM: the update's blocks that find no
// free SM (those of the highest index) start when the others are `late_by` tiles ahead.
static BesideLinkSide beside_link_side(int64_t blocks, int late_by, int tiles, int B) {
  if (B > kEarlyUsers) return BesideLinkSide{};
  const int last = blocks > 0 ? (int)((blocks - 1) % kSMs) + 1 : 0, grid = tiles < kSMs ? tiles : kSMs;      // blocks of its last wave
  const int late = grid - (kSMs - last);
  return BesideLinkSide{1, late > 0 ? late : 0, late_by};
}

// The streaming part of one XOR layer on tensor cores: links<-history attention, GatedMLP on the link rows with its
// fused consumers (`mlp` carries the outputs wanted), and the history update.  `hist_ln`: apply LayerNorm to the rows
// read (0 when they were stored normalised by the previous layer); `out_ln`: store LayerNorm(S').
static lime_status tc_layer_core(Ctx* c, int layer, const void* hist_in, const int32_t* off, int32_t B, int64_t total,
                                 const LinkOperands& ops, void* hist_out, int hist_ln, int out_ln, LinkMlpArgs mlp,
                                 const LinkSide256Args* side, const LinkSide128Args* side1, const Workspace& w, cudaStream_t st) {
  const lime_config& g = c->cfg;
  lime_status s;
  if (c->tc_mode == 2 && hist_ln && total > 0) {
    // the d = 256 kernels read LayerNorm-ed rows only: normalise the raw rows once into a scratch copy (what the
    // fused lookup + LayerNorm would have stored)
    if ((s = launch_gather_ln(g.dtype, hist_in, total, g.d, c->ln_eps, nullptr, total, w.Q, nullptr, st)) != LIME_OK) return s;
    hist_in = w.Q;
    hist_ln = 0;
  }
  // O[T]: links attend over the stored history (keys = values = history rows), chunks merged and normalised
  LinkAttnArgs la{};
  la.hist = hist_in; la.total = total; la.Q2 = ops.Q2; la.cQ = ops.cQ; la.off = off; la.chunk_start = w.chunk_start; la.chunk_user = w.chunk_user; la.B = B;
  la.group_start = w.groups.group_start; la.group_items = w.groups.group_items; la.n_groups = w.groups.n_groups;
  la.chunk = w.chunk_dev; la.n_chunk_upper = w.n_chunk_upper; la.ell = g.ell; la.d = g.d; la.H = g.H; la.shared = ops.shared;
  la.ln = hist_ln; la.ln_eps = c->ln_eps; la.silu = g.phi == LIME_PHI_SILU; la.part_m = w.part_m; la.part_s = w.part_s; la.part_acc = w.part_acc; la.Ohat = w.Ohat;
  la.err = c->dev_err;
  // the attention kernel forms the LayerNorm statistics of every history row anyway; the history update reuses them
  const bool two_tiles = c->tc_mode == 1 && hist_update_tmem_supported(g.dtype, g.d, c->d_ff, g.H, g.ell, g.phi, g.gated_mlp);
  const bool pass_stats = hist_ln && hist_out && two_tiles && total > 0;
  la.stats_out = pass_stats ? w.row_stats : nullptr;
  // The link side and the history update need nothing of each other: the update runs beside it (lime_common.cuh), which takes the
  // shorter of the two off the layer where SMs are free and evens out the tiles where they are not.  A block of the link side takes about
  // 15 us at d = 128 and 25 at d = 256, whichever of the kernels it is: two tiles of the update (13 us each at d = 256, 7 at d = 128 with
  // 256 stacked rows), or four where a tile is half as long (4 us, 128 stacked rows).  Whole tiles and one number a kind of tile: what a
  // batch takes is a step function of how many tiles move, so a finer number follows the steps of the batch it was read from.  Mean gain of
  // 27 to 33 batches of each kind over blocks that all take the same, in %, late blocks behind by 1 / 1.5 / 2 / 2.5 / 3 / 4 / 5 / 6 tiles:
  // 128 stacked rows 1.5 / 3.5 / 4.3 / 4.9 / 5.8 / 7.0 / 6.3 / 5.8; 256 stacked rows 1.8 / 4.0 / 6.9 / 6.7 / 6.3 / 5.8 / 4.8 / 3.5; d = 256
  // 4.2 / 5.3 / 6.2 / 5.4 / 5.7 / 3.9 / 2.3 / 1.0.
  const int late_by = c->tc_mode == 1 && g.H * g.ell <= 128 ? 4 : 2;
  const int64_t side_blocks = c->side256 ? link_side_d256_blocks(B) : side1 != nullptr ? link_side_d128_blocks((int64_t)B * g.ell) : ((int64_t)B * g.ell + 127) / 128;
  const BesideLinkSide beside = beside_link_side(side_blocks, late_by, w.n_tile_upper, B);
  if ((s = c->tc_mode == 2 ? launch_link_attn_d256_tc(la, st) : launch_link_attn_tc(la, st)) != LIME_OK) return s;
  if (c->side256) {
    // merge, T^j and what follows from it - the next layer's operands included - in one kernel; `side` says what is wanted
    LinkSide256Args a = *side;
    a.Ohat = w.Ohat; a.part_m = w.part_m; a.part_s = w.part_s; a.part_acc = w.part_acc; a.chunk_start = w.chunk_start;
    if ((s = launch_link_side_d256(a, st)) != LIME_OK) return s;
  } else if (side1 != nullptr) {
    // few link rows: merge, T^j and the next layer's operands in one kernel
    LinkSide128Args a = *side1;
    a.users = B; a.ell = g.ell; a.Ohat = w.Ohat; a.part_m = w.part_m; a.part_s = w.part_s; a.part_acc = w.part_acc;
    a.chunk_start = w.chunk_start; a.WpostT = c->WpostT[layer]; a.WoT = c->WoT[layer]; a.ln = g.ln; a.eps = c->ln_eps; a.err = c->dev_err;
    if ((s = launch_link_side_d128(a, st)) != LIME_OK) return s;
  } else {
  if ((s = launch_link_attn_merge_norm(w.chunk_start, w.merge_needed, B, g.ell, g.d, g.H, w.part_m, w.part_s, w.part_acc, w.Ohat, st)) != LIME_OK)
    return s;
  // T^j = GatedMLP(O[T]) and what the next step needs from it
  mlp.Ohat = w.Ohat; mlp.M = (int64_t)B * g.ell; mlp.K = g.H * g.d; mlp.d = g.d; mlp.WpostT = c->WpostT[layer]; mlp.WoT = c->WoT[layer];
  mlp.WguT = c->WguT[layer]; mlp.WvT = static_cast<const char*>(c->WprepT[layer]) + (size_t)2 * g.H * g.d * g.d * 2;     // (d = 256: k_link_prep.cu)
  mlp.ln = g.ln; mlp.ln_eps = c->ln_eps; mlp.err = c->dev_err;
  if ((s = launch_link_mlp_tc(mlp, st)) != LIME_OK) return s;
  }
  if (hist_out && c->tc_mode == 2) {
    HistUpdate256Args hu{};
    hu.hist_in = hist_in; hu.hist_out = hist_out; hu.total = total; hu.K2 = ops.K2; hu.V2t = ops.V2t; hu.WguT = c->WguT[layer];
    hu.WoT = c->WoT[layer]; hu.off = off; hu.tile_start = w.tile_start; hu.B = B; hu.n_tile_upper = w.n_tile_upper; hu.H = g.H; hu.ell = g.ell;
    hu.shared = ops.shared; hu.out_ln = out_ln; hu.silu = g.phi == LIME_PHI_SILU; hu.ln_eps = c->ln_eps; hu.beside = beside; hu.err = c->dev_err;
    if ((s = launch_hist_update_d256_tc(hu, st)) != LIME_OK) return s;
  } else if (hist_out) {
    // history attends back over the links; scores, per-head softmax, value mix and GatedMLP in one fused kernel
    HistUpdateArgs hu{};
    hu.hist_in = hist_in; hu.hist_out = hist_out; hu.total = total; hu.K2 = ops.K2; hu.G2t = ops.G2t; hu.U2t = ops.U2t;
    hu.cK = ops.cK; hu.WoT = c->WoT[layer]; hu.off = off; hu.tile_start = w.tile_start; hu.B = B;
    hu.n_tile_upper = w.n_tile_upper; hu.ell = g.ell; hu.shared = ops.shared; hu.ln = hist_ln; hu.ln_eps = c->ln_eps;
    hu.out_ln = out_ln; hu.silu = g.phi == LIME_PHI_SILU; hu.err = c->dev_err;
    hu.stats_in = pass_stats ? w.row_stats : nullptr; hu.beside = beside;
    if (two_tiles) s = launch_hist_update_tmem(hu, g.H, st);
    else s = launch_hist_update2_tc(hu, st);
    if (s != LIME_OK) return s;
  }
  return LIME_OK;
}

// One XOR layer, tensor-core path, for the public layer call: link rows in and out as fp32.
static lime_status xor_layer_tc(Ctx* c, int layer, const void* hist_in, const int32_t* off, int32_t B, int64_t total,
                                const float* links_in, int links_shared, void* hist_out, float* links_out,
                                const Workspace& w, cudaStream_t st) {
  const lime_config& g = c->cfg;
  lime_status s;
  if (c->side256) {
    LinkSide256Args prep = side256_args(c, -1, layer, links_shared ? 1 : B), side = side256_args(c, layer, -1, B);
    prep.T_in = links_in; prep.t_shared = links_shared; prep.need_hist = hist_out != nullptr;
    prep.Q2 = w.Q2; prep.K2 = w.K2; prep.V2t = w.V2t;
    if ((s = launch_link_side_d256(prep, st)) != LIME_OK) return s;
    side.T_out = links_out;
    return tc_layer_core(c, layer, hist_in, off, B, total, LinkOperands{w.Q2, w.K2, nullptr, nullptr, w.V2t, nullptr, nullptr, links_shared},
                         hist_out, g.ln, 0, LinkMlpArgs{}, &side, nullptr, w, st);
  }
  const int64_t link_rows = links_shared ? g.ell : (int64_t)B * g.ell;
  if ((s = launch_ln_rows_bf16(links_in, link_rows, g.d, g.ln, c->ln_eps, w.That, st)) != LIME_OK) return s;
  if ((s = make_link_operands(c, layer, w.That, link_rows, hist_out != nullptr, w.Q2, w.K2, w.G2t, w.U2t, w.V2t, w.cQ, w.cK, st)) != LIME_OK)
    return s;
  LinkOperands ops{w.Q2, w.K2, w.G2t, w.U2t, w.V2t, w.cQ, w.cK, links_shared};
  LinkMlpArgs mlp{};
  mlp.T_out = links_out;
  return tc_layer_core(c, layer, hist_in, off, B, total, ops, hist_out, g.ln, 0, mlp, nullptr, nullptr, w, st);
}

// lime_encode_user on the tensor-core path: per layer one link-side GEMM (none on the first layer when the links are
// the shared L: its operands are weights-only and were formed at lime_set_weights), then the streaming kernels.
// Between layers the history is kept LayerNorm-ed (every consumer normalises it first, Eq. 1 with App. C's LayerNorm),
// so only the first layer pays for the statistics.
static lime_status encode_user_tc(Ctx* c, const void* hist, bool hist_normalized, const int32_t* off, int32_t B, int64_t total,
                                  const float* link_ctx, void* link_states, const Workspace& w, cudaStream_t st) {
  const lime_config& g = c->cfg;
  lime_status s;
  const int64_t BL = (int64_t)B * g.ell;
  if (c->side256) {
    // operands of consecutive layers alternate between two sets: layer j's history update still reads its own while the
    // link side has written those of layer j + 1
    const LinkOperands set[2] = {{w.Q2, w.K2, nullptr, nullptr, w.V2t, nullptr, nullptr, 0}, {w.G2t, w.U2t, nullptr, nullptr, w.UTb, nullptr, nullptr, 0}};
    if (link_ctx) {
      LinkSide256Args prep = side256_args(c, -1, 0, B);
      prep.T_in = link_ctx; prep.need_hist = g.n_layers > 1; prep.Q2 = w.Q2; prep.K2 = w.K2; prep.V2t = w.V2t;
      if ((s = launch_link_side_d256(prep, st)) != LIME_OK) return s;
    }
    for (int j = 0; j < g.n_layers; ++j) {
      const bool last = j == g.n_layers - 1;
      LinkSide256Args side = side256_args(c, j, last ? -1 : j + 1, B);
      side.LP = w.LP; side.lp_accumulate = j > 0; side.need_hist = j + 1 < g.n_layers - 1;
      side.link_states = (last && !c->w.cand_Wv && c->cand_heads == 1) ? link_states : nullptr;
      const LinkOperands& nx = set[(j + 1) & 1];
      side.Q2 = const_cast<void*>(nx.Q2); side.K2 = const_cast<void*>(nx.K2); side.V2t = const_cast<void*>(nx.V2t);
      const LinkOperands ops = (j == 0 && !link_ctx) ? LinkOperands{c->sh_Q2, c->sh_K2, nullptr, nullptr, c->sh_V2t, nullptr, nullptr, 1} : set[j & 1];
      s = tc_layer_core(c, j, j == 0 ? hist : w.S, off, B, total, ops, last ? nullptr : w.S, (g.ln && j == 0 && !hist_normalized) ? 1 : 0,
                        (g.ln && !last) ? 1 : 0, LinkMlpArgs{}, &side, nullptr, w, st);
      if (s != LIME_OK) return s;
    }
    return LIME_OK;
  }
  // few link rows: the link side of layer j writes the operands of layer j + 1 while the update of layer j reads its own, so these
  // alternate between two sets (Q2 is the attention's, complete by then)
  const bool few_rows = few_link_rows(c, B);
  const LinkOperands set[2] = {{w.Q2, w.K2, w.G2t, w.U2t, w.V2t, w.cQ, w.cK, 0}, {w.Q2, w.K2b, w.G2tb, w.U2tb, w.V2t, w.cQ, w.cK, 0}};
  // The last layer needs its queries only: the GatedMLP kernel of the layer before makes them along with its rows.  With more than 256
  // stacked rows the update (k_hist_update2_tc.cu) does not run beside that kernel, so what it takes longer is not hidden, and a GEMM of
  // its own is shorter while the rows are few (H * ell = 512, two layers, us with a GEMM / along: 20 users of 100..1000 tokens 80.6 / 86.4, 33
  // 94.0 / 98.2, 100 149.7 / 150.6, 200 of 100..500 181.9 / 179.3).  More users than kEarlyUsers gain although the update waits there too
  // (1100 users of 100..200 tokens 239.0 / 231.7).
  const bool along = c->tc_mode == 1 && !few_rows && (g.H * g.ell <= 256 || BL > 8192);
  auto queries_along = [&](int j) { return along && j > 0 && j == g.n_layers - 1; };
  for (int j = 0; j < g.n_layers; ++j) {
    const bool last = j == g.n_layers - 1;
    const bool raw = g.ln && j == 0 && !hist_normalized;      // rows that still need their LayerNorm want the operands' row sums
    LinkOperands ops;
    if (j == 0 && !link_ctx) {
      ops = LinkOperands{c->sh_Q2, c->sh_K2, c->sh_G2t, c->sh_U2t, c->sh_V2t, c->sh_cQ, c->sh_cK, 1};
    } else {
      if (j == 0 && (s = launch_ln_rows_bf16(link_ctx, BL, g.d, g.ln, c->ln_eps, w.That, st)) != LIME_OK) return s;
      if ((j == 0 || !(few_rows || queries_along(j))) &&
          (s = make_link_operands(c, j, w.That, BL, !last, w.Q2, w.K2, w.G2t, w.U2t, w.V2t, raw ? w.cQ : nullptr, raw ? w.cK : nullptr, st)) != LIME_OK)
        return s;
      ops = set[few_rows ? j & 1 : 0];
    }
    LinkSide128Args side1{};
    if (few_rows) {
      side1.LP = w.LP; side1.lp_accumulate = j > 0; side1.need_hist = j + 1 < g.n_layers - 1;
      side1.WprepT = last ? nullptr : c->WprepT[j + 1];
      side1.link_states = (last && !c->w.cand_Wv && c->cand_heads == 1) ? link_states : nullptr;
      const LinkOperands& nx = set[(j + 1) & 1];
      side1.Q2 = w.Q2; side1.K2 = const_cast<void*>(nx.K2); side1.G2t = const_cast<void*>(nx.G2t); side1.U2t = const_cast<void*>(nx.U2t);
    }
    LinkMlpArgs mlp{};
    mlp.LP = w.LP; mlp.lp_accumulate = j > 0;                                   // L^P = sum_j T^j  (Eq. 8)
    mlp.That_next = last || queries_along(j + 1) ? nullptr : w.That;
    if (queries_along(j + 1)) { mlp.Q2 = w.Q2; mlp.WprepT = c->WprepT[j + 1]; mlp.ell = g.ell; }
    mlp.link_states = (last && !c->w.cand_Wv && c->cand_heads == 1) ? link_states : nullptr;
    s = tc_layer_core(c, j, j == 0 ? hist : w.S, off, B, total, ops, last ? nullptr : w.S, raw ? 1 : 0,
                      (g.ln && !last) ? 1 : 0, mlp, nullptr, few_rows ? &side1 : nullptr, w, st);
    if (s != LIME_OK) return s;
  }
  return LIME_OK;
}

// One XOR layer on a carved workspace (see lime_xor_layer in lime.h for the contract).
static lime_status xor_layer_impl(Ctx* c, int layer, const void* hist_in, const int32_t* off, int32_t B,
                                  int64_t total, const float* links_in, int links_shared, void* hist_out,
                                  float* links_out, const Workspace& w, bool schedules_ready, int hist_ln, cudaStream_t st) {
  // hist_ln: LayerNorm the history rows read (config.ln, except on the first layer of an encode whose rows arrive
  // normalised).  The tensor-core branch is only taken by the single-layer call, whose input is never normalised.
  const lime_config& g = c->cfg;
  lime_status s;
  if (!schedules_ready) {
    if ((s = launch_layer_schedules(off, B, w.chunk, w.chunk_dev, w.chunk_start, kHistTile, w.tile_start, w.chunk_user, w.merge_needed, w.groups, st)) != LIME_OK) return s;
  }
  if (layer_on_tensor_cores(c, layer))
    return xor_layer_tc(c, layer, hist_in, off, B, total, links_in, links_shared, hist_out, links_out, w, st);

  // ---- generic path on CUDA cores (fp32 storage, other shapes, SiLU attention, no GatedMLP) ----
  const int64_t link_rows = links_shared ? g.ell : (int64_t)B * g.ell;

  // link rows: Q[T], K[T], V[T] = LN(T) W_{Q,K,V}
  LinearArgs la{};
  la.X = links_in; la.x_dtype = LIME_F32; la.M = link_rows; la.K = g.d; la.N = g.d;
  la.W[0] = c->w.Wq[layer]; la.W[1] = c->w.Wk[layer]; la.W[2] = c->w.Wv[layer]; la.w_dtype = g.dtype;
  la.Y[0] = w.QT; la.Y[1] = w.KT; la.Y[2] = w.VT; la.y_dtype = LIME_F32; la.n_out = 3;
  la.ln = g.ln; la.ln_eps = c->ln_eps;
  if ((s = launch_linear_simt(la, st)) != LIME_OK) return s;

  // history rows: K[S], V[S] (and Q[S] when the history is updated) = LN(S) W
  LinearArgs lh{};
  lh.X = hist_in; lh.x_dtype = g.dtype; lh.M = total; lh.K = g.d; lh.N = g.d; lh.w_dtype = g.dtype; lh.y_dtype = g.dtype;
  lh.W[0] = c->w.Wk[layer]; lh.W[1] = c->w.Wv[layer]; lh.W[2] = c->w.Wq[layer];
  lh.Y[0] = w.K; lh.Y[1] = w.V; lh.Y[2] = w.Q; lh.n_out = hist_out ? 3 : 2;
  lh.ln = hist_ln; lh.ln_eps = c->ln_eps;
  if ((s = launch_linear_simt(lh, st)) != LIME_OK) return s;

  // O[T] = phi(Q[T] K[S]^T) V[S]
  AttnLinkArgs al{};
  al.QT = w.QT; al.qt_user_stride = links_shared ? 0 : (int64_t)g.ell * g.d;
  al.KS = w.K; al.VS = w.V; al.s_dtype = g.dtype; al.off = off; al.B = B; al.total = total;
  al.ell = g.ell; al.d = g.d; al.H = g.H; al.phi = g.phi; al.scale = c->attn_scale;
  al.chunk = w.chunk.tokens; al.chunk_start = w.chunk_start; al.n_chunk_upper = w.n_chunk_upper;
  al.part_m = w.part_m; al.part_s = w.part_s; al.part_acc = w.part_acc; al.AT = w.AT;
  if ((s = launch_attn_link_simt(al, st)) != LIME_OK) return s;
  if ((s = launch_attn_link_merge(al, st)) != LIME_OK) return s;

  // links_out = GatedMLP(O[T])
  const int64_t BL = (int64_t)B * g.ell;
  if (g.gated_mlp) {
    LinearArgs lg{};
    lg.X = w.AT; lg.x_dtype = LIME_F32; lg.M = BL; lg.K = g.d; lg.N = c->d_ff; lg.w_dtype = g.dtype;
    lg.W[0] = c->w.Wg[layer]; lg.W[1] = c->w.Wu[layer]; lg.Y[0] = w.UT; lg.y_dtype = LIME_F32; lg.n_out = 1; lg.glu = 1;
    if ((s = launch_linear_simt(lg, st)) != LIME_OK) return s;
    LinearArgs lo{};
    lo.X = w.UT; lo.x_dtype = LIME_F32; lo.M = BL; lo.K = c->d_ff; lo.N = g.d; lo.w_dtype = g.dtype;
    lo.W[0] = c->w.Wo[layer]; lo.Y[0] = links_out; lo.y_dtype = LIME_F32; lo.n_out = 1;
    if ((s = launch_linear_simt(lo, st)) != LIME_OK) return s;
  } else {
    if ((s = launch_axpy(w.AT, links_out, BL * g.d, 1, st)) != LIME_OK) return s;
  }

  if (hist_out) {
    // O[S] = phi(Q[S] K[T]^T) V[T], written over Q[S]; then hist_out = GatedMLP(O[S])
    AttnHistArgs ah{};
    ah.QS = w.Q; ah.AS = w.Q; ah.s_dtype = g.dtype; ah.KT = w.KT; ah.VT = w.VT;
    ah.t_user_stride = links_shared ? 0 : (int64_t)g.ell * g.d;
    ah.off = off; ah.B = B; ah.total = total; ah.ell = g.ell; ah.d = g.d; ah.H = g.H; ah.phi = g.phi;
    ah.scale = c->attn_scale; ah.tile = kHistTile; ah.tile_start = w.tile_start; ah.n_tile_upper = w.n_tile_upper;
    if ((s = launch_attn_hist_simt(ah, st)) != LIME_OK) return s;
    if (g.gated_mlp) {
      LinearArgs lg{};
      lg.X = w.Q; lg.x_dtype = g.dtype; lg.M = total; lg.K = g.d; lg.N = c->d_ff; lg.w_dtype = g.dtype;
      lg.W[0] = c->w.Wg[layer]; lg.W[1] = c->w.Wu[layer]; lg.Y[0] = w.U; lg.y_dtype = g.dtype; lg.n_out = 1; lg.glu = 1;
      if ((s = launch_linear_simt(lg, st)) != LIME_OK) return s;
      LinearArgs lo{};
      lo.X = w.U; lo.x_dtype = g.dtype; lo.M = total; lo.K = c->d_ff; lo.N = g.d; lo.w_dtype = g.dtype;
      lo.W[0] = c->w.Wo[layer]; lo.Y[0] = hist_out; lo.y_dtype = g.dtype; lo.n_out = 1;
      if ((s = launch_linear_simt(lo, st)) != LIME_OK) return s;
    } else if (total > 0) {
      LIME_CUDA(cudaMemcpyAsync(hist_out, w.Q, (size_t)total * g.d * elem_size(g.dtype), cudaMemcpyDeviceToDevice, st));
    }
  }
  return LIME_OK;
}

static lime_status check_layer_weights(const Ctx* c, int layer) {
  if (c->cfg.gated_mlp && (!c->w.Wg[layer] || !c->w.Wu[layer] || !c->w.Wo[layer])) return LIME_INVALID_ARG;
  return LIME_OK;
}

}  // namespace lime

using namespace lime;

extern "C" {

const char* lime_last_cuda_error(void) { return g_err; }
const char* lime_version(void) { return "lime-b200 0.1 sm_100a"; }

lime_status lime_profile_start(int32_t capacity) {
  if (capacity <= 0 || g_prof.open) return LIME_INVALID_ARG;
  g_prof.ev = new (std::nothrow) cudaEvent_t[2 * (size_t)capacity];
  g_prof.names = new (std::nothrow) const char*[capacity];
  if (!g_prof.ev || !g_prof.names) return LIME_INVALID_ARG;
  for (int i = 0; i < 2 * capacity; ++i) {
    cudaError_t e = cudaEventCreate(&g_prof.ev[i]);
    if (e != cudaSuccess) {
      for (int j = 0; j < i; ++j) cudaEventDestroy(g_prof.ev[j]);
      delete[] g_prof.ev; delete[] g_prof.names;
      g_prof = ProfState();
      return cuda_fail(e, "lime_profile_start");
    }
  }
  g_prof.capacity = capacity; g_prof.count = 0; g_prof.open = true;
  return LIME_OK;
}

lime_status lime_profile_stop(char* names, size_t names_bytes, float* ms, int32_t ms_capacity, int32_t* count) {
  if (!g_prof.open || !count) return LIME_INVALID_ARG;
  g_prof.open = false;
  lime_status ret = LIME_OK;
  const int n = g_prof.count < ms_capacity ? g_prof.count : ms_capacity;
  size_t pos = 0;
  if (names && names_bytes) names[0] = 0;
  for (int i = 0; i < n; ++i) {
    cudaError_t e = cudaEventSynchronize(g_prof.ev[2 * i + 1]);
    float t = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&t, g_prof.ev[2 * i], g_prof.ev[2 * i + 1]);
    if (e != cudaSuccess) ret = cuda_fail(e, "lime_profile_stop");
    if (ms) ms[i] = t;
    if (names) {
      const size_t len = strlen(g_prof.names[i]);
      if (pos + len + 2 <= names_bytes) {
        memcpy(names + pos, g_prof.names[i], len);
        pos += len;
        names[pos++] = '\n';
        names[pos] = 0;
      }
    }
  }
  *count = g_prof.count;
  for (int i = 0; i < 2 * g_prof.capacity; ++i) cudaEventDestroy(g_prof.ev[i]);
  delete[] g_prof.ev; delete[] g_prof.names;
  g_prof = ProfState();
  return ret;
}

lime_status lime_create(const lime_config* cfg, lime_ctx** out) {
  if (!cfg || !out) return LIME_INVALID_ARG;
  *out = nullptr;
  const lime_config& g = *cfg;
  if (g.d <= 0 || g.H <= 0 || g.ell <= 0 || g.n_layers <= 0 || g.d_ff < 0) return LIME_INVALID_ARG;
  if (g.dtype != LIME_F32 && g.dtype != LIME_BF16) return LIME_INVALID_ARG;
  if (g.phi != LIME_PHI_SOFTMAX && g.phi != LIME_PHI_SILU) return LIME_INVALID_ARG;
  if (g.attn_scale < 0.f || g.cand_scale < 0.f || g.ln_eps < 0.f) return LIME_INVALID_ARG;
  if (g.cand_heads != 0 && g.cand_heads != 1 && g.cand_heads != g.H) return LIME_INVALID_ARG;
  const int cand_heads = g.cand_heads == g.H ? g.H : 1;
  if (cand_heads * g.ell > 256) return LIME_UNSUPPORTED_SHAPE;
  const int d_ff = g.d_ff ? g.d_ff : g.d;
  if (g.d % 8 || d_ff % 8 || g.d % g.H || g.d / g.H > 128 || g.ell > 256 || g.n_layers > LIME_MAX_LAYERS ||
      g.d > 1024 || d_ff > 1024)
    return LIME_UNSUPPORTED_SHAPE;
  // a user's K[T], V[T] (fp32) must fit in one SM's shared memory for the history<-links attention
  if (sizeof(float) * ((size_t)2 * g.ell * (g.d + 1) + 4 * (size_t)g.d) > 200 * 1024) return LIME_UNSUPPORTED_SHAPE;
  Ctx* c = new (std::nothrow) Ctx();
  if (!c) return LIME_INVALID_ARG;
  c->cfg = g;
  memset(&c->w, 0, sizeof(c->w));
  c->have_weights = false;
  c->d_ff = d_ff;
  c->d_h = g.d / g.H;
  c->attn_scale = g.attn_scale > 0.f ? g.attn_scale : 1.0f / sqrtf((float)c->d_h);
  c->cand_heads = cand_heads;
  c->ell_c = cand_heads * g.ell;
  // per-head scores are scaled like any head of Eq. 1; the single-row form by the full width
  c->cand_scale = g.cand_scale > 0.f ? g.cand_scale : 1.0f / sqrtf((float)(cand_heads > 1 ? c->d_h : g.d));
  c->ln_eps = g.ln_eps > 0.f ? g.ln_eps : 1e-5f;
  c->keff = nullptr; c->keff_hl = nullptr; c->links32 = nullptr; c->dev_err = nullptr;
  c->have_head = c->have_ctx_mlp = false; c->ctx_dc = 0;
  c->head_W1bT = nullptr; c->head_W1aT = nullptr; c->head_w2 = nullptr; c->ctx_first = nullptr;
  c->tc_mode = tensor_core_mode(g, d_ff);
  c->side256 = c->tc_mode == 2 && link_side_d256_supported(g.d, d_ff, g.H, g.ell);
  c->side_w = nullptr;
  for (int j = 0; j < LIME_MAX_LAYERS; ++j) c->WoT[j] = c->WprepT[j] = c->WpostT[j] = c->WguT[j] = nullptr;
  c->sh_That = c->sh_Q2 = c->sh_K2 = c->sh_G2t = c->sh_U2t = c->sh_V2t = nullptr; c->sh_cQ = c->sh_cK = nullptr;
  cudaError_t e = cudaGetDevice(&c->device);
  if (e == cudaSuccess) e = cudaMalloc(&c->keff, sizeof(float) * 2 * (size_t)c->ell_c * g.d);
  if (e == cudaSuccess) e = cudaMalloc(&c->keff_hl, 2 * (size_t)2 * c->ell_c * g.d);
  if (e == cudaSuccess) e = cudaMalloc(&c->links32, sizeof(float) * (size_t)g.ell * g.d);
  if (e == cudaSuccess) e = cudaMalloc(&c->dev_err, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(c->dev_err, 0, sizeof(int));
  if (e != cudaSuccess) {
    if (c->keff) cudaFree(c->keff);
    if (c->keff_hl) cudaFree(c->keff_hl);
    if (c->links32) cudaFree(c->links32);
    if (c->dev_err) cudaFree(c->dev_err);
    delete c;
    return cuda_fail(e, "lime_create");
  }
  *out = reinterpret_cast<lime_ctx*>(c);
  return LIME_OK;
}

lime_status lime_destroy(lime_ctx* ctx) {
  if (!ctx) return LIME_OK;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  cudaFree(c->keff);
  cudaFree(c->keff_hl);
  cudaFree(c->links32);
  cudaFree(c->dev_err);
  if (c->side256) {                                    // these lie inside side_w
    for (int j = 0; j < LIME_MAX_LAYERS; ++j) c->WoT[j] = c->WguT[j] = nullptr;
    c->sh_Q2 = c->sh_K2 = c->sh_V2t = nullptr;
  }
  for (int j = 0; j < LIME_MAX_LAYERS; ++j) { cudaFree(c->WoT[j]); cudaFree(c->WprepT[j]); cudaFree(c->WpostT[j]); cudaFree(c->WguT[j]); }
  cudaFree(c->sh_That); cudaFree(c->sh_Q2); cudaFree(c->sh_K2); cudaFree(c->sh_G2t); cudaFree(c->sh_U2t); cudaFree(c->sh_V2t);
  cudaFree(c->sh_cQ); cudaFree(c->sh_cK);
  cudaFree(c->head_W1bT); cudaFree(c->head_W1aT); cudaFree(c->head_w2); cudaFree(c->ctx_first); weight_free(c->device, c->side_w);
  delete c;
  return LIME_OK;
}

lime_status lime_set_weights(lime_ctx* ctx, const lime_weights* w, void* stream) {
  if (!ctx || !w || !w->links) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  const lime_config& g = c->cfg;
  if (!aligned16(w->links)) return LIME_INVALID_ARG;
  for (int j = 0; j < g.n_layers; ++j) {
    const void* ps[6] = {w->Wq[j], w->Wk[j], w->Wv[j], w->Wg[j], w->Wu[j], w->Wo[j]};
    for (const void* p : ps) if (!aligned16(p)) return LIME_INVALID_ARG;
    if (g.gated_mlp && (!w->Wg[j] || !w->Wu[j] || !w->Wo[j])) return LIME_INVALID_ARG;
  }
  if (!aligned16(w->cand_Wq) || !aligned16(w->cand_Wk) || !aligned16(w->cand_Wv)) return LIME_INVALID_ARG;
  c->w = *w;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  lime_status s = launch_widen(w->links, g.dtype, c->links32, (int64_t)g.ell * g.d, st);
  if (s != LIME_OK) return s;
  s = launch_keff(g.dtype, w->links, w->cand_Wk, w->cand_Wq, g.ell, g.d, c->cand_heads, c->cand_scale, c->keff, st);
  if (s != LIME_OK) return s;
  if ((precompute_tc_supported(g.dtype, g.d, c->ell_c, g.ell) ||
       (g.dtype == LIME_BF16 && precompute_rows_supported(g.dtype, g.d, c->ell_c, g.ell))) &&
      (s = launch_keff_split(c->keff, c->ell_c, g.d, c->keff_hl, st)) != LIME_OK)
    return s;
  if (c->side256) {
    // weights transposed, none folded; the first layer's operands for the shared links T^0 = L follow them in one buffer
    const size_t dd = (size_t)g.d * g.d * 2, HLd = (size_t)g.H * g.ell * g.d * 2;
    if (!c->side_w) {
      LIME_CUDA(weight_alloc(c->device, &c->side_w, (size_t)g.n_layers * 6 * dd + 2 * HLd + (size_t)g.d * g.ell * 2, st));
      char* at = static_cast<char*>(c->side_w);
      for (int j = 0; j < g.n_layers; ++j, at += 6 * dd) { c->WguT[j] = at + 3 * dd; c->WoT[j] = at + 5 * dd; }
      c->sh_Q2 = at; c->sh_K2 = at + HLd; c->sh_V2t = at + 2 * HLd;
    }
    const void* src[6 * LIME_MAX_LAYERS];
    for (int j = 0; j < g.n_layers; ++j) {
      const void* m[6] = {w->Wq[j], w->Wk[j], w->Wv[j], w->Wg[j], w->Wu[j], w->Wo[j]};
      memcpy(src + 6 * j, m, sizeof(m));
    }
    if ((s = launch_transpose_square_bf16(src, 6 * g.n_layers, g.d, c->side_w, st)) != LIME_OK) return s;
    LinkSide256Args prep = side256_args(c, -1, 0, 1);
    prep.T_in = c->links32; prep.t_shared = 1; prep.need_hist = g.n_layers > 1; prep.Q2 = c->sh_Q2; prep.K2 = c->sh_K2; prep.V2t = c->sh_V2t;
    if ((s = launch_link_side_d256(prep, st)) != LIME_OK) return s;
  } else if (c->tc_mode != 0) {
    // tensor-core path: per layer, W_o as a K-major B operand ([d x d_ff], contraction index contiguous) and the
    // weight-only products that fold the history-side projections into the link rows
    const bool plain_v = c->tc_mode == 2;
    const size_t prep_rows = 2 * (size_t)g.H * g.d + (plain_v ? (size_t)g.d : 2 * (size_t)g.H * c->d_ff);
    auto need = [](void** p, size_t bytes) -> cudaError_t { return *p ? cudaSuccess : cudaMalloc(p, bytes); };
    for (int j = 0; j < g.n_layers; ++j) {
      LIME_CUDA(need(&c->WoT[j], (size_t)g.d * c->d_ff * 2));
      LIME_CUDA(need(&c->WprepT[j], prep_rows * g.d * 2));
      if (!plain_v) LIME_CUDA(need(&c->WpostT[j], (size_t)2 * c->d_ff * g.H * g.d * 2));
      if ((s = launch_transpose_bf16(w->Wo[j], c->d_ff, g.d, c->WoT[j], st)) != LIME_OK) return s;
      if (plain_v) {
        // [W_g | W_u]^T [2f x d]: the history update applies the GatedMLP weights as they stand
        LIME_CUDA(need(&c->WguT[j], (size_t)2 * c->d_ff * g.d * 2));
        if ((s = launch_transpose_bf16(w->Wg[j], g.d, c->d_ff, c->WguT[j], st)) != LIME_OK) return s;
        if ((s = launch_transpose_bf16(w->Wu[j], g.d, c->d_ff, (char*)c->WguT[j] + (size_t)c->d_ff * g.d * 2, st)) != LIME_OK) return s;
      }
      if ((s = launch_fold_weights(w->Wq[j], w->Wk[j], w->Wv[j], w->Wg[j], w->Wu[j], g.d, g.H, c->d_ff,
                                   // softmax: scores leave the fold scaled and in the log2 domain; SiLU(s) takes the raw scores
                                   g.phi == LIME_PHI_SILU ? 1.0f : c->attn_scale * 1.4426950408889634f, plain_v ? 1 : 0,
                                   c->WprepT[j], c->WpostT[j], st)) != LIME_OK)
        return s;
    }
    // first-layer operands for the shared links T^0 = L: LN(L) through the PREP GEMM, once
    const size_t HL = (size_t)g.H * g.ell;
    LIME_CUDA(need(&c->sh_That, (size_t)g.ell * g.d * 2));
    LIME_CUDA(need(&c->sh_Q2, HL * g.d * 2));
    LIME_CUDA(need(&c->sh_K2, HL * g.d * 2));
    if (plain_v) {
      LIME_CUDA(need(&c->sh_V2t, (size_t)g.d * g.ell * 2));
    } else {
      LIME_CUDA(need(&c->sh_G2t, (size_t)c->d_ff * HL * 2));
      LIME_CUDA(need(&c->sh_U2t, (size_t)c->d_ff * HL * 2));
    }
    LIME_CUDA(need((void**)&c->sh_cQ, HL * 4));
    LIME_CUDA(need((void**)&c->sh_cK, HL * 4));
    if ((s = launch_ln_rows_bf16(c->links32, g.ell, g.d, g.ln, c->ln_eps, c->sh_That, st)) != LIME_OK) return s;
    if ((s = make_link_operands(c, 0, c->sh_That, g.ell, g.n_layers > 1, c->sh_Q2, c->sh_K2, c->sh_G2t, c->sh_U2t, c->sh_V2t,
                                c->sh_cQ, c->sh_cK, st)) != LIME_OK)
      return s;
  }
  c->have_weights = true;
  return LIME_OK;
}

size_t lime_workspace_bytes(const lime_ctx* ctx, int32_t B, int64_t total_tokens) {
  if (!ctx || B < 0 || total_tokens < 0 || total_tokens > 0x7fffffffLL) return 0;
  const Ctx* c = reinterpret_cast<const Ctx*>(ctx);
  return carve(c, nullptr, B, total_tokens).bytes + 256;
}

lime_status lime_lengths_to_offsets(lime_ctx* ctx, const int32_t* len, int32_t B, int32_t* off, void* stream) {
  if (!ctx || !off || B < 0 || (B > 0 && !len)) return LIME_INVALID_ARG;
  return launch_offsets(len, B, off, static_cast<cudaStream_t>(stream));
}

lime_status lime_gather_history(lime_ctx* ctx, const void* table, int64_t V, const int32_t* ids, int64_t total_tokens,
                                void* out, int32_t* dev_flag, void* stream) {
  if (!ctx || total_tokens < 0 || V < 0) return LIME_INVALID_ARG;
  if (total_tokens == 0) return LIME_OK;
  if (!table || !ids || !out || !aligned16(table) || !aligned16(out)) return LIME_INVALID_ARG;
  const Ctx* c = reinterpret_cast<const Ctx*>(ctx);
  return launch_gather(c->cfg.dtype, table, V, c->cfg.d, ids, total_tokens, out, dev_flag,
                       static_cast<cudaStream_t>(stream));
}

lime_status lime_gather_history_normalized(lime_ctx* ctx, const void* table, int64_t V, const int32_t* ids,
                                           int64_t total_tokens, void* out, int32_t* dev_flag, void* stream) {
  if (!ctx || total_tokens < 0 || V < 0) return LIME_INVALID_ARG;
  if (total_tokens == 0) return LIME_OK;
  if (!table || !ids || !out || !aligned16(table) || !aligned16(out)) return LIME_INVALID_ARG;
  const Ctx* c = reinterpret_cast<const Ctx*>(ctx);
  if (!c->cfg.ln)
    return launch_gather(c->cfg.dtype, table, V, c->cfg.d, ids, total_tokens, out, dev_flag, static_cast<cudaStream_t>(stream));
  return launch_gather_ln(c->cfg.dtype, table, V, c->cfg.d, c->ln_eps, ids, total_tokens, out, dev_flag,
                          static_cast<cudaStream_t>(stream));
}

lime_status lime_precompute_candidate_links(lime_ctx* ctx, const void* cand_emb, int64_t M, void* out_w, void* stream) {
  if (!ctx || M < 0) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  if (!c->have_weights) return LIME_NOT_READY;
  if (M == 0) return LIME_OK;
  if (!cand_emb || !out_w || !aligned16(cand_emb) || !aligned16(out_w)) return LIME_INVALID_ARG;
  if (precompute_tc_supported(c->cfg.dtype, c->cfg.d, c->ell_c, c->cfg.ell))
    return launch_precompute_tc(cand_emb, M, c->cfg.d, c->ell_c, c->cfg.ell, c->keff_hl, out_w, c->dev_err,
                                static_cast<cudaStream_t>(stream));
  if (precompute_rows_supported(c->cfg.dtype, c->cfg.d, c->ell_c, c->cfg.ell))
    return launch_precompute_rows(c->cfg.dtype, cand_emb, M, c->cfg.d, c->ell_c, c->keff, c->keff_hl, out_w, static_cast<cudaStream_t>(stream));
  return launch_precompute(c->cfg.dtype, cand_emb, M, c->cfg.d, c->ell_c, c->cfg.ell, c->keff, out_w,
                           static_cast<cudaStream_t>(stream));
}

lime_status lime_xor_layer(lime_ctx* ctx, int32_t layer, const void* hist_in, const int32_t* off, int32_t B,
                           int64_t total_tokens, const float* links_in, int32_t links_shared, void* hist_out,
                           float* links_out, void* ws, size_t ws_bytes, void* stream) {
  if (!ctx || B < 0 || total_tokens < 0 || total_tokens > 0x7fffffffLL) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  if (!c->have_weights) return LIME_NOT_READY;
  if (layer < 0 || layer >= c->cfg.n_layers) return LIME_INVALID_ARG;
  if (B == 0) return LIME_OK;
  if (!off || !links_in || !links_out || !ws || (total_tokens > 0 && !hist_in)) return LIME_INVALID_ARG;
  if (!aligned16(hist_in) || !aligned16(hist_out) || !aligned16(links_in) || !aligned16(links_out)) return LIME_INVALID_ARG;
  if (check_layer_weights(c, layer) != LIME_OK) return LIME_INVALID_ARG;
  char* base = reinterpret_cast<char*>(align_up(reinterpret_cast<uintptr_t>(ws)));
  const size_t pad = base - static_cast<char*>(ws);
  Workspace w = carve(c, base, B, total_tokens);
  if (w.bytes + pad > ws_bytes) return LIME_WORKSPACE_TOO_SMALL;
  return xor_layer_impl(c, layer, hist_in, off, B, total_tokens, links_in, links_shared, hist_out, links_out, w, false,
                        c->cfg.ln, static_cast<cudaStream_t>(stream));
}

static lime_status encode_user_impl(lime_ctx* ctx, const void* hist, bool hist_normalized, const int32_t* off, int32_t B,
                                    int64_t total_tokens, const float* link_ctx, void* link_states, void* ws, size_t ws_bytes,
                                    void* stream) {
  if (!ctx || B < 0 || total_tokens < 0 || total_tokens > 0x7fffffffLL) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  if (!c->have_weights) return LIME_NOT_READY;
  if (B == 0) return LIME_OK;
  if (!off || !link_states || !ws || (total_tokens > 0 && !hist)) return LIME_INVALID_ARG;
  if (!aligned16(hist) || !aligned16(link_ctx) || !aligned16(link_states)) return LIME_INVALID_ARG;
  const lime_config& g = c->cfg;
  for (int j = 0; j < g.n_layers; ++j)
    if (check_layer_weights(c, j) != LIME_OK) return LIME_INVALID_ARG;
  char* base = reinterpret_cast<char*>(align_up(reinterpret_cast<uintptr_t>(ws)));
  const size_t pad = base - static_cast<char*>(ws);
  Workspace w = carve(c, base, B, total_tokens);
  if (w.bytes + pad > ws_bytes) return LIME_WORKSPACE_TOO_SMALL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  lime_status s;
  const bool narrow = encode_small_wanted(c, B, total_tokens);
  if (!narrow && (s = launch_layer_schedules(off, B, w.chunk, w.chunk_dev, w.chunk_start, kHistTile, w.tile_start, w.chunk_user, w.merge_needed, w.groups, st)) != LIME_OK) return s;
  const int64_t BLd = (int64_t)B * g.ell * g.d;
  if (narrow) {
    EncodeSmallArgs a{};
    a.hist = hist; a.off = off; a.B = B; a.total = total_tokens; a.links = link_ctx ? link_ctx : c->links32; a.links_per_user = link_ctx != nullptr;
    a.w = &c->w; a.scale = c->attn_scale;
    a.H = g.H; a.ell = g.ell; a.n_layers = g.n_layers; a.ln = g.ln; a.hist_ln = g.ln && !hist_normalized; a.silu = g.phi == LIME_PHI_SILU;
    a.eps = c->ln_eps; a.scratch = w.S;
    const bool direct = !c->w.cand_Wv && c->cand_heads == 1;
    a.link_states = direct ? link_states : nullptr; a.lp = w.LP;
    if (g.dtype == LIME_F32) {
      if (direct) a.lp = static_cast<float*>(link_states);
      s = launch_encode_f32(a, c->dev_err, st);
    } else {
      s = launch_encode_small(a, st);
    }
    if (s != LIME_OK) return s;
    if (direct) return LIME_OK;
  } else if (layer_on_tensor_cores(c, 0)) {
    if ((s = encode_user_tc(c, hist, hist_normalized, off, B, total_tokens, link_ctx, link_states, w, st)) != LIME_OK) return s;
    if (!c->w.cand_Wv && c->cand_heads == 1) return LIME_OK;        // the last layer's kernel wrote the link states
  } else {
    for (int j = 0; j < g.n_layers; ++j) {
      const bool last = j == g.n_layers - 1;
      const float* lin = j == 0 ? (link_ctx ? link_ctx : c->links32) : w.T;
      const int shared = (j == 0 && !link_ctx) ? 1 : 0;
      s = xor_layer_impl(c, j, j == 0 ? hist : w.S, off, B, total_tokens, lin, shared, last ? nullptr : w.S, w.T, w, true,
                         (g.ln && !(j == 0 && hist_normalized)) ? 1 : 0, st);
      if (s != LIME_OK) return s;
      if ((s = launch_axpy(w.T, w.LP, BLd, j == 0, st)) != LIME_OK) return s;   // L^P = sum_j T^j  (Eq. 8)
    }
  }
  // link states = L^P W_V^c (Eq. 4's values), stored as the run's dtype
  const float* src = w.LP;
  if (c->w.cand_Wv) {
    LinearArgs lv{};
    lv.X = w.LP; lv.x_dtype = LIME_F32; lv.M = (int64_t)B * g.ell; lv.K = g.d; lv.N = g.d; lv.w_dtype = g.dtype;
    lv.W[0] = c->w.cand_Wv; lv.Y[0] = w.LS32; lv.y_dtype = LIME_F32; lv.n_out = 1;
    if ((s = launch_linear_simt(lv, st)) != LIME_OK) return s;
    src = w.LS32;
  }
  if (c->cand_heads > 1) return launch_expand_heads(src, (int64_t)B * g.ell, g.ell, g.d, c->cand_heads, link_states, g.dtype, st);
  return launch_cast_rows(src, BLd, link_states, g.dtype, st);
}

lime_status lime_encode_user(lime_ctx* ctx, const void* hist, const int32_t* off, int32_t B, int64_t total_tokens,
                             const float* link_ctx, void* link_states, void* ws, size_t ws_bytes, void* stream) {
  return encode_user_impl(ctx, hist, false, off, B, total_tokens, link_ctx, link_states, ws, ws_bytes, stream);
}

lime_status lime_encode_user_normalized(lime_ctx* ctx, const void* hist_normalized, const int32_t* off, int32_t B,
                                        int64_t total_tokens, const float* link_ctx, void* link_states, void* ws,
                                        size_t ws_bytes, void* stream) {
  return encode_user_impl(ctx, hist_normalized, true, off, B, total_tokens, link_ctx, link_states, ws, ws_bytes, stream);
}

lime_status lime_score_candidates(lime_ctx* ctx, const void* link_states, int32_t B, const void* cand_w,
                                  const void* cand_emb, const int32_t* cand_off, int32_t C, int64_t total_cands,
                                  const int32_t* cand_ids, int64_t corpus_rows, int32_t* dev_flag, float* logits,
                                  void* stream) {
  if (!ctx || B < 0 || C < 0 || total_cands < 0 || total_cands > 0x7fffffffLL) return LIME_INVALID_ARG;
  if (cand_ids && (corpus_rows <= 0 || corpus_rows > 0x7fffffffLL)) return LIME_INVALID_ARG;
  if (!cand_off && total_cands != (int64_t)B * C) return LIME_INVALID_ARG;
  if (B == 0 || total_cands == 0) return LIME_OK;
  if (!link_states || !cand_w || !cand_emb || !logits) return LIME_INVALID_ARG;
  if (!aligned16(link_states) || !aligned16(cand_w) || !aligned16(cand_emb)) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  ScoreArgs a{};
  a.LS = link_states; a.W = cand_w; a.T = cand_emb; a.dtype = c->cfg.dtype; a.B = B; a.ell = c->ell_c; a.d = c->cfg.d;
  a.cand_off = cand_off; a.C = C; a.total = total_cands; a.cand_ids = cand_ids; a.logits = logits;
  a.corpus_rows = cand_ids ? corpus_rows : 0; a.dev_flag = cand_ids ? dev_flag : nullptr;
  if (score_rows_preferred(a)) return launch_score_rows(a, static_cast<cudaStream_t>(stream));
  if (score_tc_supported(a)) return launch_score_tc(a, c->dev_err, static_cast<cudaStream_t>(stream));
  if (score_gather_tc_supported(a)) return launch_score_gather_tc(a, c->dev_err, static_cast<cudaStream_t>(stream));
  return launch_score_simt(a, static_cast<cudaStream_t>(stream));
}

// ---- feed-forward networks (Eq. 2; Sec. 3.3 interaction network) ----------------------------------------------------
static bool ffn_valid(const lime_ffn* f, int min_hidden) {
  if (!f || f->n_hidden < min_hidden || f->n_hidden > LIME_FFN_MAX_HIDDEN) return false;
  for (int i = 0; i < f->n_hidden; ++i)
    if (f->widths[i] < 1 || f->widths[i] > 1024) return false;
  for (int i = 0; i <= f->n_hidden; ++i)
    if (!f->W[i] || !aligned16(f->W[i])) return false;
  return true;
}
// layers after the first: layer i maps widths[i-1] to widths[i] (the last one to `out_last`)
static FfnArgs ffn_tail(const lime_ffn& f, int out_last) {
  FfnArgs a{};
  a.n_layers = f.n_hidden;
  for (int i = 1; i <= f.n_hidden; ++i) {
    a.in_w[i - 1] = f.widths[i - 1];
    a.out_w[i - 1] = i < f.n_hidden ? f.widths[i] : out_last;
    a.W[i - 1] = f.W[i];
    a.b[i - 1] = f.b[i];
  }
  return a;
}

lime_status lime_set_context_mlp(lime_ctx* ctx, int32_t d_c, const lime_ffn* mlp, void* stream) {
  if (!ctx || d_c < 1 || d_c > 4096 || !ffn_valid(mlp, 0)) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  if (!c->have_weights) return LIME_NOT_READY;
  const lime_config& g = c->cfg;
  const int w0 = mlp->n_hidden > 0 ? mlp->widths[0] : g.d;
  cudaFree(c->ctx_first);
  c->ctx_first = nullptr;
  c->have_ctx_mlp = false;
  LIME_CUDA(cudaMalloc(&c->ctx_first, sizeof(float) * (size_t)g.ell * w0));
  // weights-only part of the first layer: (L W_0[:d]) + b_0
  lime_status s = launch_rows_times_w(c->w.links, g.dtype, g.ell, g.d, mlp->W[0], g.dtype, w0, w0, mlp->b[0], c->ctx_first,
                                      "k_ctx_first", static_cast<cudaStream_t>(stream));
  if (s != LIME_OK) return s;
  c->ctx_mlp = *mlp;
  c->ctx_dc = d_c;
  c->have_ctx_mlp = true;
  return LIME_OK;
}

lime_status lime_contextualize_links(lime_ctx* ctx, const void* user_ctx, int32_t B, float* link_ctx, void* stream) {
  if (!ctx || B < 0) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  if (!c->have_ctx_mlp) return LIME_NOT_READY;
  if (B == 0) return LIME_OK;
  if (!user_ctx || !link_ctx || !aligned16(link_ctx)) return LIME_INVALID_ARG;
  const lime_config& g = c->cfg;
  const lime_ffn& f = c->ctx_mlp;
  const int w0 = f.n_hidden > 0 ? f.widths[0] : g.d;
  const char* W0c = static_cast<const char*>(f.W[0]) + (size_t)g.d * w0 * elem_size(g.dtype);     // rows d.. act on E^C
  if (link_ctx_mma_supported(g.dtype, c->ctx_dc, w0, g.ell, g.d, ffn_tail(f, g.d)))
    return launch_link_ctx_mma(c->ctx_first, user_ctx, c->ctx_dc, W0c, w0, B, g.ell, g.d, ffn_tail(f, g.d), link_ctx, static_cast<cudaStream_t>(stream));
  return launch_link_ctx_mlp(g.dtype, c->ctx_first, user_ctx, c->ctx_dc, W0c, w0, B, g.ell, ffn_tail(f, g.d), link_ctx,
                             static_cast<cudaStream_t>(stream));
}

lime_status lime_set_head(lime_ctx* ctx, const lime_ffn* head, void* stream) {
  if (!ctx || !ffn_valid(head, 1)) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  const lime_config& g = c->cfg;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int w0 = head->widths[0], w_last = head->widths[head->n_hidden - 1];
  cudaFree(c->head_W1bT); cudaFree(c->head_W1aT); cudaFree(c->head_w2);
  c->head_W1bT = nullptr; c->head_W1aT = nullptr; c->head_w2 = nullptr;
  c->have_head = false;
  LIME_CUDA(cudaMalloc(&c->head_w2, sizeof(float) * (size_t)w_last));
  lime_status s = launch_widen(head->W[head->n_hidden], g.dtype, c->head_w2, w_last, st);
  if (s != LIME_OK) return s;
  if (g.dtype == LIME_BF16) {
    // the T half of the first layer as a K-major B operand [w0 x d]
    LIME_CUDA(cudaMalloc(&c->head_W1bT, (size_t)w0 * g.d * 2));
    const char* W0t = static_cast<const char*>(head->W[0]) + (size_t)g.d * w0 * 2;
    if ((s = launch_transpose_bf16(W0t, g.d, w0, c->head_W1bT, st)) != LIME_OK) return s;
    LIME_CUDA(cudaMalloc(&c->head_W1aT, (size_t)w0 * g.d * 2));
    if ((s = launch_transpose_bf16(head->W[0], g.d, w0, c->head_W1aT, st)) != LIME_OK) return s;
  }
  c->head = *head;
  c->have_head = true;
  return LIME_OK;
}

size_t lime_head_workspace_bytes(const lime_ctx* ctx, int32_t B) {
  if (!ctx || B < 0) return 0;
  const Ctx* c = reinterpret_cast<const Ctx*>(ctx);
  if (!c->have_head) return 0;
  const size_t n = (size_t)B * c->ell_c * c->head.widths[0];
  return align_up(n * 4) + align_up(n * 2) + 256;
}

lime_status lime_score_candidates_head(lime_ctx* ctx, const void* link_states, int32_t B, const void* cand_w,
                                       const void* cand_emb, const int32_t* cand_off, int32_t C, int64_t total_cands,
                                       const int32_t* cand_ids, int64_t corpus_rows, int32_t* dev_flag, float* logits,
                                       void* ws, size_t ws_bytes, void* stream) {
  if (!ctx || B < 0 || C < 0 || total_cands < 0 || total_cands > 0x7fffffffLL) return LIME_INVALID_ARG;
  if (cand_ids && (corpus_rows <= 0 || corpus_rows > 0x7fffffffLL)) return LIME_INVALID_ARG;
  if (!cand_off && total_cands != (int64_t)B * C) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  if (!c->have_head) return LIME_NOT_READY;
  if (B == 0 || total_cands == 0) return LIME_OK;
  if (!link_states || !cand_w || !cand_emb || !logits || !ws) return LIME_INVALID_ARG;
  if (!aligned16(link_states) || !aligned16(cand_w) || !aligned16(cand_emb)) return LIME_INVALID_ARG;
  const lime_config& g = c->cfg;
  const lime_ffn& f = c->head;
  const int w0 = f.widths[0];
  char* base = reinterpret_cast<char*>(align_up(reinterpret_cast<uintptr_t>(ws)));
  const size_t n = (size_t)B * c->ell_c * w0;
  if ((size_t)(base - static_cast<char*>(ws)) + align_up(n * 4) + align_up(n * 2) > ws_bytes) return LIME_WORKSPACE_TOO_SMALL;
  float* LSW = reinterpret_cast<float*>(base);       // [B][ell][w0], or its bf16 pieces (three at most: the same 6 n bytes)
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  ScoreArgs a{};
  a.LS = link_states; a.W = cand_w; a.T = cand_emb; a.dtype = g.dtype; a.B = B; a.ell = c->ell_c; a.d = g.d;
  a.cand_off = cand_off; a.C = C; a.total = total_cands; a.cand_ids = cand_ids; a.logits = logits;
  a.corpus_rows = cand_ids ? corpus_rows : 0; a.dev_flag = cand_ids ? dev_flag : nullptr;
  if (score_mlp3_supported(a, f)) return launch_score_mlp3(a, f, st);
  // per user: LSW_b = LS_b W_0[:d]  (the O half of the first layer applied to the link states, so O is never formed)
  lime_status s;
  if (f.n_hidden == 1 && c->head_W1bT && score_head_tc_supported(a, w0)) {
    s = launch_gemm_rows_t(link_states, (int64_t)B * c->ell_c, g.d, c->head_W1aT, w0, c->ell_c, score_head_tc_terms(a, w0), base, c->dev_err,
                           "k_gemm_tc_lsw", st);
    if (s != LIME_OK) return s;
    ScoreHeadArgs h{base, c->head_W1bT, f.b[0], c->head_w2, f.b[1], w0};
    return launch_score_head_tc(a, h, c->dev_err, st);
  }
  s = launch_rows_times_w(link_states, g.dtype, (int64_t)B * c->ell_c, g.d, f.W[0], g.dtype, w0, w0, nullptr, LSW, "k_head_lsw", st);
  if (s != LIME_OK) return s;
  const char* W0t = static_cast<const char*>(f.W[0]) + (size_t)g.d * w0 * elem_size(g.dtype);
  return launch_score_head_simt(a, LSW, W0t, f.b[0], w0, ffn_tail(f, 1), st);
}

lime_status lime_pack_corpus_cache(lime_ctx* ctx, const void* cand_emb, const void* cand_w, int64_t corpus_rows, void* packed,
                                   void* stream) {
  if (!ctx || corpus_rows < 0 || corpus_rows > 0x7fffffffLL) return LIME_INVALID_ARG;
  if (corpus_rows == 0) return LIME_OK;
  if (!cand_emb || !cand_w || !packed || !aligned16(cand_emb) || !aligned16(cand_w) || !aligned16(packed)) return LIME_INVALID_ARG;
  const Ctx* c = reinterpret_cast<const Ctx*>(ctx);
  return launch_pack_corpus(c->cfg.dtype, cand_emb, cand_w, corpus_rows, c->cfg.d, c->ell_c, packed, static_cast<cudaStream_t>(stream));
}

lime_status lime_score_candidates_packed(lime_ctx* ctx, const void* link_states, int32_t B, const void* packed,
                                         int64_t corpus_rows, const int32_t* cand_ids, const int32_t* cand_off, int32_t C,
                                         int64_t total_cands, int32_t* dev_flag, float* logits, void* stream) {
  if (!ctx || B < 0 || C < 0 || total_cands < 0 || total_cands > 0x7fffffffLL) return LIME_INVALID_ARG;
  if (corpus_rows <= 0 || corpus_rows > 0x7fffffffLL) return LIME_INVALID_ARG;
  if (!cand_off && total_cands != (int64_t)B * C) return LIME_INVALID_ARG;
  if (B == 0 || total_cands == 0) return LIME_OK;
  if (!link_states || !packed || !cand_ids || !logits || !aligned16(link_states) || !aligned16(packed)) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  const int es = elem_size(c->cfg.dtype);
  ScoreArgs a{};
  a.LS = link_states; a.T = packed; a.W = static_cast<const char*>(packed) + (size_t)c->cfg.d * es;
  a.ldt = a.ldw = c->cfg.d + c->ell_c;
  a.dtype = c->cfg.dtype; a.B = B; a.ell = c->ell_c; a.d = c->cfg.d;
  a.cand_off = cand_off; a.C = C; a.total = total_cands; a.cand_ids = cand_ids; a.logits = logits;
  a.corpus_rows = corpus_rows; a.dev_flag = dev_flag;
  if (score_rows_preferred(a)) return launch_score_rows(a, static_cast<cudaStream_t>(stream));
  if (score_gather_tc_supported(a)) return launch_score_gather_tc(a, c->dev_err, static_cast<cudaStream_t>(stream));
  return launch_score_simt(a, static_cast<cudaStream_t>(stream));
}

lime_status lime_selftest_wait_expiry(lime_ctx* ctx, int32_t limit_us, void* stream) {
  if (!ctx || limit_us < 1 || limit_us > 1000000) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  return launch_wait_expiry(c->dev_err, (uint64_t)limit_us * 1000ull, LIME_SELFTEST_WAIT_CODE, static_cast<cudaStream_t>(stream));
}

lime_status lime_device_status(lime_ctx* ctx, int32_t* code) {
  if (!ctx || !code) return LIME_INVALID_ARG;
  Ctx* c = reinterpret_cast<Ctx*>(ctx);
  int v = 0;
  LIME_CUDA(cudaMemcpy(&v, c->dev_err, sizeof(int), cudaMemcpyDeviceToHost));
  *code = v;
  if (v != 0) {
    LIME_CUDA(cudaMemset(c->dev_err, 0, sizeof(int)));
    return LIME_DEVICE_TIMEOUT;
  }
  return LIME_OK;
}

}  // extern "C"
