// Ragged bookkeeping, the history-embedding gather and small elementwise helpers.
#include "lime_common.cuh"

namespace lime {

// ----------------------------------------------------------------------------- block-wide exclusive scan
// What the threads before this one hold, of two values at once, and the block's totals.  One barrier: every warp adds up the warp sums
// itself.  `sums`: shared memory for up to 32 warps; consecutive scans alternate between two of them.
__device__ __forceinline__ int2 block_scan2(int2 v, int2* sums, int2& total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int2 incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, incl.x, o), y = __shfl_up_sync(0xffffffffu, incl.y, o);
    if (lane >= o) { incl.x += x; incl.y += y; }
  }
  if (lane == 31) sums[wid] = incl;
  __syncthreads();
  const int2 w = lane < (int)(blockDim.x >> 5) ? sums[lane] : make_int2(0, 0);
  total = make_int2(__reduce_add_sync(0xffffffffu, w.x), __reduce_add_sync(0xffffffffu, w.y));
  return make_int2(__reduce_add_sync(0xffffffffu, lane < wid ? w.x : 0) + incl.x - v.x,
                   __reduce_add_sync(0xffffffffu, lane < wid ? w.y : 0) + incl.y - v.y);
}

__global__ void __launch_bounds__(1024) k_offsets(const int32_t* __restrict__ len, int B, int32_t* __restrict__ off) {
  __shared__ int2 sums[2][32];
  pdl_launch_dependents();     // simple kernel: the next one may set itself up beside it
  pdl_wait();                  // nothing is read or written before the previous kernel is complete
  int carry = 0;
  for (int b0 = 0, k = 0; b0 < B; b0 += blockDim.x, k ^= 1) {
    const int b = b0 + threadIdx.x;
    int2 total;
    const int2 before = block_scan2(make_int2(b < B ? max(len[b], 0) : 0, 0), sums[k], total);
    if (b < B) off[b] = carry + before.x;
    carry += total.x;
  }
  if (threadIdx.x == 0) off[B] = carry;
}

// The work lists of the XOR layers in one launch: chunks of the links<-history attention, tiles of the history update, and (group_start
// given) the chunk items dealt to `G` groups of CTAs so that the groups' token tiles come out even.  One block, a thread per user (the
// users of 1024 threads at a time).  Every layer waits for this kernel, so it is kept a short chain: a user's length is read once and stays
// in a register (of the first 1024), both prefix sums are one scan, and the dealing works in shared memory up to SCAP items.  (The lengths
// read again for each list, two scans of five barriers, the item's user looked up in global memory and two loops of one thread: 3.1 us
// after the lookup for 256 users of 512 tokens at d = 128, 9 us for 64 users at d = 256 with 32 links; this way one request of one user
// takes 38.0 us, 40.75 before, the 256 users 133.9, 135.7, the 64 at d = 256 225.8, 229.)
// The dealing: items are sorted by size (a counting sort over their tile counts, largest first) and handed out in
// rounds of G: within a round the group with the least work so far takes the largest item, the next group the next
// one, and so on.  Ragged histories dealt round-robin leave the busiest group 16 % above the mean (1024 users of
// 1024..4096 tokens over 37 groups); this order leaves it under 1 %.  A round is one rank computation over
// the G loads in shared memory and one barrier.
// group_start[G+1], group_items[items]: the items of group j in the order it takes them.  scratch: 4 x items ints.
// WALK (with the dealing): a user's items are listed by its warp's lanes together and counted in two steps.  One thread walks them
// otherwise, 0.15 us an item: nothing for the few items that users have, 176 us for a single user of 4M tokens (977 items; 23 with WALK)
// and 49 us of 1M (13).  An instance of its own, like FIT: where it is not needed it costs 0.5 to 1.2 us (16 users of 100..1024 tokens
// 108.4 -> 109, 64 users 202.5 -> 203.7), so the host asks for it where the total makes more than 32 items of the ordinary length
// (short ones, of which there are 64 at most, are left to the thread).
// FIT: the lengths of the items are fitted where some history is longer than one (rule.fit_groups); an instance of its own, because the
// code alone, never reached, cost the batch of 256 users x 512 4.5 us.
template <bool FIT, bool WALK>
__global__ void __launch_bounds__(1024)
k_layer_schedules(const int32_t* __restrict__ off, int B, const ChunkRule rule, int32_t* __restrict__ chunk_out,
                  int32_t* __restrict__ chunk_start, int tile,
                  int32_t* __restrict__ tile_start, int32_t* __restrict__ chunk_user, int32_t* __restrict__ merge_needed,
                  int G, int att_tile, int32_t* __restrict__ group_start, int32_t* __restrict__ group_items,
                  int32_t* __restrict__ scratch) {
  constexpr int KEYS = 256, GMAX = 160, KCAP = 16384, SCAP = 2048;
  __shared__ int2 sums[2][32];
  __shared__ int32_t hist[KEYS];
  __shared__ __align__(16) int32_t load[GMAX];
  __shared__ int32_t cnt[GMAX], first[GMAX];
  __shared__ uint8_t skey[KCAP];                   // sizes in sorted order (the first KCAP items; the rest are read from global)
  __shared__ int32_t small[3 * SCAP];
  pdl_launch_dependents();     // simple kernel: the next one may set itself up beside it
  const bool deal = group_start != nullptr && chunk_user != nullptr;
  if (deal) {
    for (int i = threadIdx.x; i < KEYS; i += blockDim.x) hist[i] = 0;
    for (int i = threadIdx.x; i < GMAX; i += blockDim.x) { load[i] = i < G ? 0 : 0x7fffffff; cnt[i] = 0; }
  }
  pdl_wait();                  // nothing is read or written before the previous kernel is complete
  const int n_first = (int)threadIdx.x < B ? off[threadIdx.x + 1] - off[threadIdx.x] : 0;
  auto length = [&](int b) { return b < (int)blockDim.x ? n_first : off[b + 1] - off[b]; };      // b: one of this thread's
  int longest = 0, short_items = 0;
  if (rule.short_tokens > 0 || FIT) {
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
      const int n = length(b);
      longest = max(longest, n);
      if ((!FIT || rule.short_tokens > 0) && n > rule.short_tokens) short_items += (n + rule.short_tokens - 1) / rule.short_tokens;
    }
    longest = __reduce_max_sync(0xffffffffu, longest);
    short_items = __reduce_add_sync(0xffffffffu, short_items);
    const int lane = threadIdx.x & 31;
    if (lane == 0) sums[0][threadIdx.x >> 5] = make_int2(longest, short_items);
    __syncthreads();
    const int2 w = lane < (int)(blockDim.x >> 5) ? sums[0][lane] : make_int2(0, 0);
    longest = __reduce_max_sync(0xffffffffu, w.x);
    short_items = __reduce_add_sync(0xffffffffu, w.y);
  }
  const bool take_short = longest > 2 * rule.short_tokens && short_items <= rule.short_items && (!FIT || rule.short_tokens > 0);
  int chunk = take_short ? rule.short_tokens : rule.tokens;
  if constexpr (FIT) if (!take_short && longest > chunk && B <= 3 * SCAP) {
    // Rounds of the groups over the items, each with its tiles and what an item costs besides (draining the pipeline, the way out of its
    // accumulator, filling it again: 8800 cycles with partials to write, 3100 without, a tile of 128 tokens takes 1490): the length for
    // which that comes out least.  A warp per length.  64 links, us with 2048 tokens (or the power of two that the total asks for) / fitted:
    // 32 users of 32768, four layers 1670 / 1626; three layers, 10 of 30000 383 / 354, 16 of 4000..8000 188 / 168, 4 of 32768 203 / 185.
    constexpr float OVER_PART = 5.9f, OVER_ONE = 2.1f;
    __shared__ float best_cost[32];
    __shared__ int best_tiles[32];
    int tiles_all = 0;
    for (int b = threadIdx.x; b < B; b += blockDim.x) small[b] = max(length(b), 0);
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    for (int b = lane; b < B; b += 32) tiles_all += (small[b] + 127) / 128;
    tiles_all = __reduce_add_sync(0xffffffffu, tiles_all);
    float cost = INFINITY;
    int at = 0;
    for (int t = (rule.tokens * 3 / 4 + 127) / 128 + wid; t <= 64; t += n_warps) {
      int items = 0, ones = 0;
      for (int b = lane; b < B; b += 32) {
        const int k = (small[b] + t * 128 - 1) / (t * 128);
        items += k;
        ones += k == 1;
      }
      items = __reduce_add_sync(0xffffffffu, items);
      ones = __reduce_add_sync(0xffffffffu, ones);
      const float c = (float)((items + rule.fit_groups - 1) / rule.fit_groups) *
                      ((float)tiles_all + OVER_PART * (float)(items - ones) + OVER_ONE * (float)ones) / (float)items;
      if (items <= rule.fit_items && c < cost) { cost = c; at = t; }
    }
    if (lane == 0) { best_cost[wid] = cost; best_tiles[wid] = at; }
    __syncthreads();
    cost = INFINITY;
    at = 0;
    for (int w = 0; w < n_warps; ++w)
      if (best_cost[w] < cost || (best_cost[w] == cost && best_tiles[w] < at)) { cost = best_cost[w]; at = best_tiles[w]; }
    if (at > 0) chunk = at * 128;
    __syncthreads();
  }
  // does any user's attention output need the merge step (several chunks to combine, or no history: a zero row)?
  int merge = 0;
  for (int b = threadIdx.x; b < B; b += blockDim.x)
    if (length(b) <= 0 || length(b) > chunk) merge = 1;
  merge = __syncthreads_or(merge);
  if (threadIdx.x == 0) {
    *chunk_out = chunk;
    if (merge_needed != nullptr) *merge_needed = merge;
  }
  // bucket 0 holds the largest items
  auto bucket = [&](int tokens) { return KEYS - 1 - min(KEYS - 1, (tokens + att_tile - 1) / att_tile); };
  // WALK: f(what, i, first) for the k consecutive items from `first` of every thread's user, by that thread up to OWN, else by the lanes of
  // its warp together.  Every thread of the warp calls it.
  constexpr int OWN = 8;
  auto each_item = [&](int k, int first, auto f, int what) {
    if (k <= OWN)
      for (int i = 0; i < k; ++i) f(what, first + i, first);
    for (unsigned many = __ballot_sync(0xffffffffu, k > OWN); many != 0; many &= many - 1) {
      const int src = __ffs(many) - 1;
      const int all = __shfl_sync(0xffffffffu, k, src), from = __shfl_sync(0xffffffffu, first, src), w = __shfl_sync(0xffffffffu, what, src);
      for (int i = threadIdx.x & 31; i < all; i += 32) f(w, from + i, from);
    }
  };
  int2 carry = make_int2(0, 0);
  int item_first = 0;                              // this thread's first item, of its first user
  for (int b0 = 0, k = 1; b0 < B; b0 += blockDim.x, k ^= 1) {
    const int b = b0 + threadIdx.x;
    const int n = b < B ? max(length(b), 0) : 0;
    const int n_chunks = (n + chunk - 1) / chunk;
    int2 total;
    const int2 before = block_scan2(make_int2(n_chunks, (n + tile - 1) / tile), sums[k], total);
    const int item = carry.x + before.x;
    if (b0 == 0) item_first = item;
    if (b < B) { chunk_start[b] = item; tile_start[b] = carry.y + before.y; }
    // inverse map (chunk item -> user): the attention kernel strides through the items, and one read of this table
    // replaces a search over chunk_start per item
    if constexpr (WALK) {
      each_item(n_chunks, item, [&](int user, int i, int) { chunk_user[i] = user; }, b);
      if (n_chunks > 1) atomicAdd(&hist[bucket(chunk)], n_chunks - 1);       // full items, and the last one, which may be shorter
      if (n_chunks > 0) atomicAdd(&hist[bucket(n - (n_chunks - 1) * chunk)], 1);
    } else if (chunk_user != nullptr) {
      for (int i = 0; i < n_chunks; ++i) {
        chunk_user[item + i] = b;
        if (deal) atomicAdd(&hist[KEYS - 1 - min(KEYS - 1, (min(chunk, n - i * chunk) + att_tile - 1) / att_tile)], 1);
      }
    }
    carry.x += total.x;
    carry.y += total.y;
  }
  if (threadIdx.x == 0) { chunk_start[B] = carry.x; tile_start[B] = carry.y; }
  if (!deal) return;
  const int n_items = carry.x;
  int32_t* const sorted = n_items <= SCAP ? small : scratch;
  int32_t* const key_of = n_items <= SCAP ? nullptr : scratch + n_items;                 // by sorted position, from KCAP on
  int32_t* const group_of = n_items <= SCAP ? small + SCAP : scratch + 2 * (size_t)n_items;
  int32_t* const slot_of = n_items <= SCAP ? small + 2 * SCAP : scratch + 3 * (size_t)n_items;
  __syncthreads();
  {                                                // (at least KEYS threads)
    int2 total;
    const int mine = threadIdx.x < KEYS ? hist[threadIdx.x] : 0;
    const int2 before = block_scan2(make_int2(mine, 0), sums[0], total);
    if (threadIdx.x < KEYS) hist[threadIdx.x] = before.x;
  }
  __syncthreads();
  auto place = [&](int at, int item, int key) {
    sorted[at] = item;
    if (at < KCAP) skey[at] = (uint8_t)key;
    else key_of[at] = key;
  };
  if constexpr (WALK) {
    for (int b0 = 0; b0 < B; b0 += blockDim.x) {
      const int b = b0 + threadIdx.x;
      const int n = b < B ? max(length(b), 0) : 0, k = (n + chunk - 1) / chunk, item = n == 0 ? 0 : b0 == 0 ? item_first : chunk_start[b];
      const int full = k > 1 ? atomicAdd(&hist[bucket(chunk)], k - 1) : 0;
      each_item(k - 1, item, [&](int at, int i, int first) { place(at + i - first, i, KEYS - 1 - bucket(chunk)); }, full);
      if (k > 0) {
        const int in = bucket(n - (k - 1) * chunk);
        place(atomicAdd(&hist[in], 1), item + k - 1, KEYS - 1 - in);
      }
    }
  } else {
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
      const int n = max(length(b), 0), item = b < (int)blockDim.x ? item_first : chunk_start[b];
      for (int i = 0; i * chunk < n; ++i) {
        const int key = min(KEYS - 1, (min(chunk, n - i * chunk) + att_tile - 1) / att_tile);
        place(atomicAdd(&hist[KEYS - 1 - key], 1), item + i, key);
      }
    }
  }
  __syncthreads();
  for (int r0 = 0; r0 < n_items; r0 += G) {
    const int j = threadIdx.x;
    int rank = 0, mine = 0;
    if (j < G) {
      mine = load[j];
#pragma unroll 4
      for (int o = 0; o < G; o += 4) {             // (loads past G are the largest there is)
        const int4 l = *reinterpret_cast<const int4*>(load + o);
        rank += (l.x < mine || (l.x == mine && o < j)) + (l.y < mine || (l.y == mine && o + 1 < j)) +
                (l.z < mine || (l.z == mine && o + 2 < j)) + (l.w < mine || (l.w == mine && o + 3 < j));
      }
    }
    __syncthreads();                               // every rank is taken before a load changes
    if (j < G && r0 + rank < n_items) {
      const int at = r0 + rank;
      const int key = at < KCAP ? (int)skey[at] : key_of[at];
      group_of[at] = j;                             // by sorted position: no dependent read inside a round
      slot_of[at] = cnt[j]++;
      load[j] = mine + key;
    }
    __syncthreads();
  }
  {                                                // (at least GMAX threads)
    int2 total;
    const int2 before = block_scan2(make_int2((int)threadIdx.x < G ? cnt[threadIdx.x] : 0, 0), sums[1], total);
    if ((int)threadIdx.x < G) first[threadIdx.x] = group_start[threadIdx.x] = before.x;
    if (threadIdx.x == 0) group_start[G] = total.x;
  }
  __syncthreads();
  for (int at = threadIdx.x; at < n_items; at += blockDim.x) group_items[first[group_of[at]] + slot_of[at]] = sorted[at];
}

// a thread per user, 256 at least (the dealing scans its 256 buckets in one go), 1024 at most
static int schedule_threads(int B) { return B <= 256 ? 256 : B >= 1024 ? 1024 : (B + 31) / 32 * 32; }

lime_status launch_layer_schedules(const int32_t* off, int B, const ChunkRule& chunk, int32_t* chunk_out, int32_t* chunk_start, int tile, int32_t* tile_start,
                                   int32_t* chunk_user, int32_t* merge_needed, const GroupSchedule& gs, cudaStream_t st) {
  if (gs.group_start != nullptr && (gs.n_groups < 1 || gs.n_groups > 160 || gs.att_tile < 1)) return LIME_INVALID_ARG;
  ProfScope _p("k_layer_schedules", st);
  const auto kernel = chunk.fit_groups > 0 ? k_layer_schedules<true, false> : gs.walk ? k_layer_schedules<false, true> : k_layer_schedules<false, false>;
  launch_pdl(kernel, dim3(1), dim3(schedule_threads(B)), 0, st, off, B, chunk, chunk_out, chunk_start, tile, tile_start, chunk_user, merge_needed,
             gs.n_groups, gs.att_tile, gs.group_start, gs.group_items, gs.scratch);
  LIME_LAUNCH_CHECK("k_layer_schedules");
  return LIME_OK;
}

lime_status launch_offsets(const int32_t* len, int B, int32_t* off, cudaStream_t st) {
  ProfScope _p("k_offsets", st);
  launch_pdl(k_offsets, dim3(1), dim3(schedule_threads(B)), 0, st, len, B, off);
  LIME_LAUNCH_CHECK("k_offsets");
  return LIME_OK;
}

// ----------------------------------------------------------------------------- gather
// out[t, :] = table[ids[t], :].  Rows are 16-byte multiples (d % 8 == 0 for both dtypes), so a row moves as
// uint4 words: `LANES` consecutive threads own one row and each moves row_vec / LANES words, giving fully
// coalesced 128-bit loads and stores.  Reads of hot (Zipf head) rows hit L2; the stream is write-dominated.
template <int LANES>
__global__ void __launch_bounds__(256)
k_gather(const uint4* __restrict__ table, int64_t V, int row_vec, const int32_t* __restrict__ ids, int64_t total,
         uint4* __restrict__ out, int32_t* __restrict__ dev_flag) {
  pdl_launch_dependents();     // simple kernel: the next one may set itself up beside it
  pdl_wait();                  // nothing is read or written before the previous kernel is complete
  const int rows_per_block = blockDim.x / LANES;
  const int sub = threadIdx.x % LANES;
  const int64_t stride = (int64_t)gridDim.x * rows_per_block;
  for (int64_t t = (int64_t)blockIdx.x * rows_per_block + threadIdx.x / LANES; t < total; t += stride) {
    const int32_t id = __ldg(ids + t);
    const bool ok = id >= 0 && (int64_t)id < V;
    uint4* dst = out + t * row_vec;
    if (ok) {
      const uint4* src = table + (int64_t)id * row_vec;
      for (int v = sub; v < row_vec; v += LANES) dst[v] = __ldg(src + v);
    } else {
      for (int v = sub; v < row_vec; v += LANES) dst[v] = make_uint4(0, 0, 0, 0);
      if (sub == 0 && dev_flag != nullptr) atomicMin(dev_flag, (int32_t)min(t, (int64_t)INT32_MAX));
    }
  }
}

// out[t, :] = LayerNorm(table[ids[t], :]) (non-affine), in the storage type (ids == NULL: the rows of `table` in order,
// i.e. a plain LayerNorm pass over V = total rows).  Same row-per-LANES mapping; a lane keeps
// its WORDS 16-byte words of the row in registers, the lanes of a row reduce the sum and then the squared
// deviations with shuffles (two passes: exact mean first), and the normalised row is written once.  The loop runs
// per warp-wide group of rows so that every lane takes part in the shuffles.
// a 16-byte word of the storage type <-> floats (bf16: two elements per 32-bit lane, widened with a shift / a mask
// and narrowed pairwise with one round-to-nearest conversion)
template <typename T> struct Word16;
template <> struct Word16<float> {
  static __device__ __forceinline__ void unpack(const uint4& w, float (&x)[4]) {
    x[0] = __uint_as_float(w.x); x[1] = __uint_as_float(w.y); x[2] = __uint_as_float(w.z); x[3] = __uint_as_float(w.w);
  }
  static __device__ __forceinline__ uint4 pack(const float (&x)[4]) {
    return make_uint4(__float_as_uint(x[0]), __float_as_uint(x[1]), __float_as_uint(x[2]), __float_as_uint(x[3]));
  }
};
template <> struct Word16<__nv_bfloat16> {
  static __device__ __forceinline__ void unpack(const uint4& w, float (&x)[8]) {
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) { x[2 * k] = __uint_as_float(u[k] << 16); x[2 * k + 1] = __uint_as_float(u[k] & 0xffff0000u); }
  }
  static __device__ __forceinline__ uint4 pack(const float (&x)[8]) {
    uint32_t u[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const __nv_bfloat162 p2 = __floats2bfloat162_rn(x[2 * k], x[2 * k + 1]);
      u[k] = *reinterpret_cast<const uint32_t*>(&p2);
    }
    return make_uint4(u[0], u[1], u[2], u[3]);
  }
};

template <typename T, int LANES, int WORDS>
__global__ void __launch_bounds__(256)
k_gather_ln(const uint4* __restrict__ table, int64_t V, int row_vec, int d, float eps, const int32_t* __restrict__ ids,
            int64_t total, uint4* __restrict__ out, int32_t* __restrict__ dev_flag) {
  pdl_launch_dependents();     // simple kernel: the next one may set itself up beside it
  pdl_wait();                  // nothing is read or written before the previous kernel is complete
  constexpr int PER = 16 / (int)sizeof(T);                 // elements per 16-byte word
  constexpr int ROWS = 1;   // rows per lane group and pass (more in flight measured slower: the grid already covers the latency)
  const int rows_per_block = blockDim.x / LANES;
  const int sub = threadIdx.x % LANES;
  const int64_t stride = (int64_t)gridDim.x * rows_per_block * ROWS;
  for (int64_t base = (int64_t)blockIdx.x * rows_per_block * ROWS; base < total; base += stride) {
    int64_t t[ROWS];
    bool live[ROWS], ok[ROWS];
    int32_t id[ROWS];
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
      t[k] = base + (int64_t)k * rows_per_block + threadIdx.x / LANES;
      live[k] = t[k] < total;
      id[k] = live[k] ? (ids != nullptr ? __ldg(ids + t[k]) : (int32_t)t[k]) : 0;   // no ids: row t of `table` itself
      ok[k] = live[k] && id[k] >= 0 && (int64_t)id[k] < V;
    }
    uint4 w[ROWS][WORDS];
#pragma unroll
    for (int k = 0; k < ROWS; ++k)
#pragma unroll
      for (int i = 0; i < WORDS; ++i) {
        const int v = sub + i * LANES;
        w[k][i] = (ok[k] && v < row_vec) ? __ldg(table + (int64_t)id[k] * row_vec + v) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
      float x[WORDS][PER];
      float sum = 0.f;
#pragma unroll
      for (int i = 0; i < WORDS; ++i) {
        Word16<T>::unpack(w[k][i], x[i]);
#pragma unroll
        for (int j = 0; j < PER; ++j) sum += x[i][j];
      }
#pragma unroll
      for (int o = LANES / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const float mu = sum / (float)d;
      float var = 0.f;
#pragma unroll
      for (int i = 0; i < WORDS; ++i) {
        if (sub + i * LANES < row_vec) {
#pragma unroll
          for (int j = 0; j < PER; ++j) { x[i][j] -= mu; var = fmaf(x[i][j], x[i][j], var); }
        }
      }
#pragma unroll
      for (int o = LANES / 2; o > 0; o >>= 1) var += __shfl_xor_sync(0xffffffffu, var, o);
      const float rstd = rsqrtf(var / (float)d + eps);
      if (live[k]) {
#pragma unroll
        for (int i = 0; i < WORDS; ++i) {
          const int v = sub + i * LANES;
          if (v < row_vec) {
            uint4 o4 = make_uint4(0, 0, 0, 0);              // an id outside [0, V) gives a zero row, as in k_gather
            if (ok[k]) {
#pragma unroll
              for (int j = 0; j < PER; ++j) x[i][j] *= rstd;
              o4 = Word16<T>::pack(x[i]);
            }
            out[t[k] * row_vec + v] = o4;
          }
        }
        if (!ok[k] && sub == 0 && dev_flag != nullptr) atomicMin(dev_flag, (int32_t)min(t[k], (int64_t)INT32_MAX));
      }
    }
  }
}

template <typename T, int WORDS>
static void launch_gather_ln_w(int lanes, int blocks, const uint4* tb, int64_t V, int row_vec, int d, float eps,
                               const int32_t* ids, int64_t total, uint4* o, int32_t* dev_flag, cudaStream_t st) {
  switch (lanes) {
    case 32: launch_pdl(k_gather_ln<T, 32, WORDS>, dim3((unsigned)blocks), dim3(256), 0, st, tb, V, row_vec, d, eps, ids, total, o, dev_flag); break;
    case 16: launch_pdl(k_gather_ln<T, 16, WORDS>, dim3((unsigned)blocks), dim3(256), 0, st, tb, V, row_vec, d, eps, ids, total, o, dev_flag); break;
    case 8:  launch_pdl(k_gather_ln<T, 8, WORDS>, dim3((unsigned)blocks), dim3(256), 0, st, tb, V, row_vec, d, eps, ids, total, o, dev_flag); break;
    default: launch_pdl(k_gather_ln<T, 4, WORDS>, dim3((unsigned)blocks), dim3(256), 0, st, tb, V, row_vec, d, eps, ids, total, o, dev_flag); break;
  }
}
template <typename T>
static lime_status launch_gather_ln_t(int lanes, int words, int blocks, const uint4* tb, int64_t V, int row_vec, int d, float eps,
                                      const int32_t* ids, int64_t total, uint4* o, int32_t* dev_flag, cudaStream_t st) {
  if (words <= 1) launch_gather_ln_w<T, 1>(lanes, blocks, tb, V, row_vec, d, eps, ids, total, o, dev_flag, st);
  else if (words <= 2) launch_gather_ln_w<T, 2>(lanes, blocks, tb, V, row_vec, d, eps, ids, total, o, dev_flag, st);
  else if (words <= 4) launch_gather_ln_w<T, 4>(lanes, blocks, tb, V, row_vec, d, eps, ids, total, o, dev_flag, st);
  else if (words <= 8) launch_gather_ln_w<T, 8>(lanes, blocks, tb, V, row_vec, d, eps, ids, total, o, dev_flag, st);
  else return LIME_UNSUPPORTED_SHAPE;                                  // d <= 1024 keeps a row within 32 lanes x 8 words
  return LIME_OK;
}

lime_status launch_gather_ln(int dtype, const void* table, int64_t V, int d, float eps, const int32_t* ids, int64_t total,
                             void* out, int32_t* dev_flag, cudaStream_t st) {
  if (total == 0) return LIME_OK;
  const int es = dtype == LIME_F32 ? 4 : 2;
  const int row_vec = d * es / 16;
  // two words per lane where the row allows: half the shuffle steps and two independent loads per thread
  int lanes = row_vec >= 64 ? 32 : (row_vec >= 32 ? 16 : (row_vec >= 16 ? 8 : 4));
  const int words = (row_vec + lanes - 1) / lanes;
  const int rows_per_block = 256 / lanes;
  int64_t blocks = (total + rows_per_block - 1) / rows_per_block;
  const int64_t cap = (int64_t)kSMs * 16;
  if (blocks > cap) blocks = cap;
  ProfScope _p("k_gather_ln", st);
  const lime_status s =
      dtype == LIME_F32
          ? launch_gather_ln_t<float>(lanes, words, (int)blocks, (const uint4*)table, V, row_vec, d, eps, ids, total, (uint4*)out, dev_flag, st)
          : launch_gather_ln_t<__nv_bfloat16>(lanes, words, (int)blocks, (const uint4*)table, V, row_vec, d, eps, ids, total, (uint4*)out,
                                              dev_flag, st);
  if (s != LIME_OK) return s;
  LIME_LAUNCH_CHECK("k_gather_ln");
  return LIME_OK;
}

lime_status launch_gather(int dtype, const void* table, int64_t V, int d, const int32_t* ids, int64_t total,
                          void* out, int32_t* dev_flag, cudaStream_t st) {
  if (total == 0) return LIME_OK;
  const int es = dtype == LIME_F32 ? 4 : 2;
  const int row_vec = d * es / 16;
  const int threads = 256;
  // enough lanes per row that each thread moves 1-2 words
  int lanes = row_vec >= 32 ? 32 : (row_vec >= 16 ? 16 : (row_vec >= 8 ? 8 : 4));
  const int rows_per_block = threads / lanes;
  int64_t blocks = (total + rows_per_block - 1) / rows_per_block;
  const int64_t cap = (int64_t)kSMs * 16;
  if (blocks > cap) blocks = cap;
  ProfScope _p("k_gather", st);
  const uint4* tb = (const uint4*)table;
  uint4* o = (uint4*)out;
  switch (lanes) {
    case 32: launch_pdl(k_gather<32>, dim3((unsigned)blocks), dim3(threads), 0, st, tb, V, row_vec, ids, total, o, dev_flag); break;
    case 16: launch_pdl(k_gather<16>, dim3((unsigned)blocks), dim3(threads), 0, st, tb, V, row_vec, ids, total, o, dev_flag); break;
    case 8:  launch_pdl(k_gather<8>, dim3((unsigned)blocks), dim3(threads), 0, st, tb, V, row_vec, ids, total, o, dev_flag); break;
    default: launch_pdl(k_gather<4>, dim3((unsigned)blocks), dim3(threads), 0, st, tb, V, row_vec, ids, total, o, dev_flag); break;
  }
  LIME_LAUNCH_CHECK("k_gather");
  return LIME_OK;
}

// ----------------------------------------------------------------------------- elementwise helpers
template <typename T>
__global__ void k_cast_rows(const float* __restrict__ in, int64_t n, T* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    Store<T>::st(out + i, in[i]);
}
template <typename T>
__global__ void k_widen(const T* __restrict__ in, int64_t n, float* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = Store<T>::ld(in + i);
}
__global__ void k_axpy(const float* __restrict__ x, float* __restrict__ y, int64_t n, int zero_first) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = (zero_first ? 0.0f : y[i]) + x[i];
}

// Link states of the per-head candidate side (Eq. 1 applied to Eq. 4): row (h, l) of a user is L^P row l on head h's
// columns and zero elsewhere, so that the full-width dot <T_c, row (h, l)> is head h's dot product.
template <typename T>
__global__ void k_expand_heads(const float* __restrict__ src, int64_t n_out, int ell, int d, int heads, T* __restrict__ out) {
  const int dh = d / heads;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_out; i += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(i % d);
    const int64_t row = i / d;                       // (user, head, link)
    const int l = (int)(row % ell), h = (int)((row / ell) % heads);
    const int64_t b = row / ((int64_t)ell * heads);
    Store<T>::st(out + i, j / dh == h ? src[(b * ell + l) * d + j] : 0.f);
  }
}

static inline int ew_blocks(int64_t n) {
  int64_t b = (n + 255) / 256;
  const int64_t cap = (int64_t)kSMs * 8;
  return (int)(b > cap ? cap : (b < 1 ? 1 : b));
}

lime_status launch_expand_heads(const float* src, int64_t rows_in, int ell, int d, int heads, void* out, int dtype,
                                cudaStream_t st) {
  const int64_t n_out = rows_in * heads * d;
  if (n_out == 0) return LIME_OK;
  ProfScope _p("k_expand_heads", st);
  if (dtype == LIME_F32) k_expand_heads<float><<<ew_blocks(n_out), 256, 0, st>>>(src, n_out, ell, d, heads, (float*)out);
  else k_expand_heads<__nv_bfloat16><<<ew_blocks(n_out), 256, 0, st>>>(src, n_out, ell, d, heads, (__nv_bfloat16*)out);
  LIME_LAUNCH_CHECK("k_expand_heads");
  return LIME_OK;
}

lime_status launch_cast_rows(const float* in, int64_t n, void* out, int dtype, cudaStream_t st) {
  if (n == 0) return LIME_OK;
  ProfScope _p("k_cast_rows", st);
  if (dtype == LIME_F32) k_cast_rows<float><<<ew_blocks(n), 256, 0, st>>>(in, n, (float*)out);
  else k_cast_rows<__nv_bfloat16><<<ew_blocks(n), 256, 0, st>>>(in, n, (__nv_bfloat16*)out);
  LIME_LAUNCH_CHECK("k_cast_rows");
  return LIME_OK;
}
lime_status launch_widen(const void* in, int dtype, float* out, int64_t n, cudaStream_t st) {
  if (n == 0) return LIME_OK;
  ProfScope _p("k_widen", st);
  if (dtype == LIME_F32) k_widen<float><<<ew_blocks(n), 256, 0, st>>>((const float*)in, n, out);
  else k_widen<__nv_bfloat16><<<ew_blocks(n), 256, 0, st>>>((const __nv_bfloat16*)in, n, out);
  LIME_LAUNCH_CHECK("k_widen");
  return LIME_OK;
}
lime_status launch_axpy(const float* x, float* y, int64_t n, int zero_first, cudaStream_t st) {
  if (n == 0) return LIME_OK;
  ProfScope _p("k_axpy", st);
  k_axpy<<<ew_blocks(n), 256, 0, st>>>(x, y, n, zero_first);
  LIME_LAUNCH_CHECK("k_axpy");
  return LIME_OK;
}

}  // namespace lime
