/* The planner of libpard: kernels and their orchestration.
 *
 * Steps (paper passages in pard.h):
 *   prepass   per-ctx deadline range, input checks, whether deadlines come in order; with few queues
 *             also their constants
 *   segconst  per-segment constants of Eq. 3: d_k(B_k), base, L_sub (max over
 *             downstream paths), folded into A = base + d + L_sub
 *   pack      request -> one 64-bit sort element (segment | deadline | index), digit counts of the
 *             passes; with few queues also the counts behind the window tables
 *   sort      LSD radix sort, 8 bits per pass, one read and one write of the
 *             elements per pass (tile prefixes by decoupled look-back); in arrival order with up to 256
 *             queues one pass straight from the requests, counted by the prepass (nothing is packed)
 *   windows   queue boundaries, batch-window tables, kept counts and output offsets (with few queues
 *             from the counts, beside the sort)
 *   decide    every request on its own from its queue's table: admitted position c, estimate, keep
 *             flag, survivors to their final place; too many windows: the same by a segmented
 *             prefix-min scan (k_scan_path)
 * Calls grouped by ctx in small contexts are planned by a block per ctx (pard_local.cu), in large ones that come in
 * order without a sort (pard_direct.cuh), the comparison rules by a walk of every queue behind the sort (pard_policy.cu).
 */
#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>

#include "pard_plan_internal.cuh"

using namespace pard_plan_detail;

namespace {

struct Layout {
  /* [hdr, zero_end) must be zero when the first kernel starts: cleared by k_clear (of the two
   * look-back arrays only the first: every sort pass clears the array of the pass after it) */
  uint64_t hdr, ctx_dmin, ctx_dmax, seg_off, seg_kept, hist, whist, hist_ctx, lookback, zero_end, tile_first,
      ctx_start, pipes, ktab, kept_base, chunk_base, tile_agg, tile_carry, win_off, win_cnt, wtab, kept_tmp,
      buf_a, buf_b, total;
  uint32_t n_seg, sort_tiles, dec_tiles, max_passes, win_capacity;
  uint32_t lb_rows;           /* rows of 256 words of a look-back array: tiles, and groups of tiles */
  uint32_t ctx_tiles;         /* most tiles of passes inside the contexts' ranges */
  uint32_t small_tiles, tile_size, geometry;   /* see make_layout, k_sort_rest */
  uint32_t ctx_passes;        /* 1: the call may sort inside the contexts' ranges (contexts of more than a tile on average) */
};

__host__ __device__ inline uint32_t bit_width64(unsigned long long x) {
  uint32_t b = 0;
  while (x) { ++b; x >>= 1; }
  return b;
}

inline uint32_t ceil_log2(uint64_t x) {          /* smallest b with 2^b >= x */
  uint32_t b = 0;
  while (((uint64_t)1 << b) < x) ++b;
  return b;
}

/* Passes of the sort of a large call that get a launch of their own: the 24 bits that a queue id and
 * the deadlines of about a second take. */
constexpr uint32_t kOwnPasses = 3;

bool local_sort_candidate(uint64_t n, uint32_t n_ctx) {
  if (n_ctx == 1) return n > 0 && n <= (uint64_t)kSortTile;         /* certain: one ctx inside one tile */
  return n >= (uint64_t)n_ctx * (kSortTile / 4) && n <= (uint64_t)n_ctx * kSortTile;
}

Layout make_layout(uint64_t n, uint32_t n_ctx, int32_t stage_stride) {
  Layout L;
  auto al = [](uint64_t x) { return (x + 255) & ~(uint64_t)255; };
  L.n_seg = n_ctx * (uint32_t)stage_stride;
  /* the sort's tiles: kSortTile elements, or, where one or two rounds of smaller ones do, as many as the
   * device holds at a time (see k_sort_rest; three rounds of smaller ones lose to two of kSortTile) */
  L.small_tiles = n <= 2ull * kResidentTiles * kSmallTile ? 1u : 0u;
  L.tile_size = kSortTile;
  L.geometry = 0;
  if (L.small_tiles) {
    const uint64_t rounds = std::max<uint64_t>(1, (n + (uint64_t)kResidentTiles * kSmallTile - 1) / ((uint64_t)kResidentTiles * kSmallTile));
    const uint64_t size = (n + kResidentTiles * rounds - 1) / (kResidentTiles * rounds);
    const uint32_t both = (uint32_t)std::min<uint64_t>(kSmallLo + kSmallHi, std::max<uint64_t>(kSmallLeast, (size + 255) / 256));
    const uint32_t lo = std::max(1u, (both * kSmallLo + (kSmallLo + kSmallHi) / 2) / (kSmallLo + kSmallHi));
    L.geometry = lo | (both - lo) << 8;
    L.tile_size = 256 * both;
  }
  L.sort_tiles = (uint32_t)((n + L.tile_size - 1) / L.tile_size);
  L.dec_tiles = (uint32_t)((n + kDecTile - 1) / kDecTile);
  uint32_t ibits = std::max(1u, ceil_log2(n));
  uint32_t sbits = ceil_log2(L.n_seg);
  L.max_passes = std::min<uint32_t>(kMaxPasses, (std::min(64u - ibits, sbits + 60u) + 7) / 8);
  uint64_t o = 0;
  L.hdr = o;       o = al(o + sizeof(PlanHeader));
  L.ctx_dmin = o;  o = al(o + 8ull * n_ctx);          /* complement of the minimum: starts at 0 */
  L.ctx_dmax = o;  o = al(o + 8ull * n_ctx);
  L.seg_off = o;   o = al(o + 4ull * (L.n_seg + 1));
  L.seg_kept = o;  o = al(o + 4ull * L.n_seg);
  L.hist = o;      o = al(o + 4ull * kMaxPasses * kBins);
  L.whist = o;     o = al(o + (L.n_seg <= kHistSegs ? 4ull * kHistCap : 0ull));   /* window counts of calls with few queues */
  /* passes kept inside the contexts' ranges cut the tiles at ctx boundaries: at most one more
   * tile per ctx; they keep digit counts per ctx */
  L.ctx_passes = (n_ctx > 1 && (uint64_t)n_ctx * kSortTile < n) ? 1u : 0u;
  L.ctx_tiles = (uint32_t)((n + kSortTile - 1) / kSortTile) + (L.ctx_passes ? n_ctx : 0u);
  L.lb_rows = std::max(L.ctx_passes ? L.ctx_tiles : 0u, L.sort_tiles + L.sort_tiles / kLookGroup + 1);
  L.hist_ctx = o;  o = al(o + (L.ctx_passes ? 4ull * kMaxPasses * kBins * (uint64_t)n_ctx : 0ull));
  L.lookback = o;  L.zero_end = al(o + 4ull * kBins * (uint64_t)L.lb_rows);
  o = al(o + 2 * 4ull * kBins * (uint64_t)L.lb_rows);                      /* two arrays, used in turn */
  L.tile_first = o; o = al(o + (L.ctx_passes ? 4ull * ((uint64_t)n_ctx + 1) : 0ull));
  L.ctx_start = o; o = al(o + 4ull * ((uint64_t)n_ctx + 1));
  L.pipes = o;     o = al(o + 8ull * kMaxPipelinesPerCall);
  L.ktab = o;      o = al(o + sizeof(PardSegConst) * (uint64_t)L.n_seg);
  L.kept_base = o; o = al(o + 4ull * (L.n_seg + 1));
  L.chunk_base = o; o = al(o + 4ull * (L.n_seg + 1));
  L.tile_agg = o;  o = al(o + 8ull * L.dec_tiles);
  L.tile_carry = o; o = al(o + 4ull * L.dec_tiles);
  L.win_capacity = (uint32_t)(n / 32 + 4ull * L.n_seg + 1024);
  if (L.n_seg <= kHistSegs) L.win_capacity = std::max(L.win_capacity, kHistCap);   /* counted tables: see k_seg_const */
  L.win_off = o;   o = al(o + 4ull * (L.n_seg + 1));
  L.win_cnt = o;   o = al(o + 4ull * (L.n_seg + 1));
  L.wtab = o;      o = al(o + 16ull * L.win_capacity);
  L.kept_tmp = o;  o = al(o + 4ull * n);
  L.buf_a = o;     o = al(o + 8ull * n);
  L.buf_b = o;     o = al(o + 8ull * n);
  L.total = o;
  return L;
}

/* See k_sort_local: the call's requests come grouped by ctx and no ctx exceeds a tile. */
__device__ __forceinline__ bool sort_is_local(const PlanHeader* hdr, uint32_t candidate) {
  return candidate && !hdr->unsorted && !hdr->ctx_too_big && !hdr->wide;
}

/* Words of the header that blocks of the running kernel may set (a wait has run out, a ctx is not grouped)
 * are read by one thread for its whole block: threads that read for themselves could see it change, and a
 * block whose first warp has left would go on with what that warp was to fetch. */
__device__ __forceinline__ bool gave_up(const PlanHeader* hdr) {
  return __syncthreads_or(threadIdx.x == 0 && ld_relaxed(&hdr->aborted)) != 0;
}

/* True in every thread of exactly one block: the one whose `mine` arrivals at `counter` complete `all`.
 * Every thread's earlier global writes are visible to that block afterwards. */
__device__ __forceinline__ bool last_arrival(uint32_t* counter, uint32_t mine, uint32_t all) {
  __shared__ uint32_t s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = mine && atomicAdd(counter, mine) + mine == all ? 1u : 0u;
  __syncthreads();
  const bool last = s_last != 0;
  if (last) __threadfence();
  return last;
}
__device__ __forceinline__ bool last_block_done(uint32_t* counter) { return last_arrival(counter, 1u, gridDim.x); }

/* Clears the part of the scratch that must start at zero.  A kernel rather than a memset: it is
 * launched like every other kernel of the call, so its blocks are placed while the previous
 * work of the stream drains. */
__global__ void __launch_bounds__(256)
k_clear(uint4* __restrict__ p, unsigned long long n16) {
  pdl_wait();
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += step)
    p[i] = make_uint4(0u, 0u, 0u, 0u);
}

/* Width of the sort key, once the widest deadline span is known, and the part of it that the
 * passes have to sort.  key_sbits: the queue-id bits to sort (all of them, or the stage bits only
 * when the passes stay inside the contexts' ranges).  The deadline field below them needs no pass
 * when every queue's requests stand in the order it asks for: in arrival order the index alone
 * orders a queue, and in budget order (low budget first everywhere) requests whose deadlines never
 * step back along the array, or along every ctx of an array grouped by ctx, are ordered as they
 * come.  (2^24 such requests in 256 contexts: one pass instead of four, 696 -> 408 us for the call.) */
__device__ __forceinline__ void set_key_width(PlanHeader* hdr, unsigned long long span, uint32_t sbits, uint32_t ibits,
                                              uint32_t key_sbits, uint32_t arrival_order, bool priority) {
  uint32_t dbits = bit_width64(span);
  if (arrival_order && sbits + dbits + ibits > 64) {    /* no room: the rule reads the deadlines from the requests */
    dbits = 0;
    hdr->lookup = 1;
  }
  const bool in_order = arrival_order || (!priority && !(hdr->time_steps_back && hdr->pair_steps_back));
  const uint32_t skip = in_order ? dbits : 0u;
  hdr->span_max = span;
  hdr->dbits = dbits;
  hdr->pshift = skip;
  hdr->keybits = key_sbits + dbits - skip;
  hdr->npass = (key_sbits + dbits - skip + 7) / 8;
  if (sbits + dbits + ibits > 64) {
    hdr->npass = 0;
    hdr->wide = 1;
    set_status(hdr, PARD_ERANGE);
  }
}

/* What the constants of a call's queues are made from, and what follows from them and the deadline
 * ranges before any request is packed. */
struct ConstArgs {
  PipeTable pipes;
  pard_queue_state_t st;
  uint32_t n_pipelines, n_ctx;
  PardSegConst* ktab;
  uint32_t sbits, ibits, key_sbits;
  uint32_t with_key_width;         /* the block that finishes last also finds the key width (no launches for it) */
  uint32_t arrival_order, win_hist, force_scan;
  uint32_t* win_off;
  uint32_t* win_cnt;
  long long* path_sums;            /* see PolicyArgs; or null */
};

__device__ __forceinline__ long long* sums_of(const ConstArgs& a, uint32_t c) {
  return a.path_sums ? a.path_sums + (size_t)c * a.st.stage_stride * kMaskPaths : nullptr;
}

/* What the constants of a queue take from the deadline range [lo, hi] of its ctx, as in ctx_constants; the new `narrow`. */
__device__ __forceinline__ uint32_t range_constants(PardSegConst* K, long long A, long long d, uint32_t narrow, unsigned long long lo, unsigned long long hi) {
  const long long A_rel = (narrow & kSegHighFirst) ? (long long)hi - A : A - (long long)lo;
  const bool fits = fits_narrow(__ldcg(&K->d_magic), d, A_rel, (narrow & kSegHighFirst) != 0) && !(narrow & kSegNoStage);
  narrow = (narrow & ~kSegNarrow) | (fits ? kSegNarrow : 0u);
  K->A_rel = A_rel;
  K->narrow = narrow;
  return narrow;
}

/* By one whole block, once every ctx's deadline range and every queue's constants are there: what
 * hangs on both.  RANGES: the constants do not know the ranges yet. */
template <bool RANGES>
__device__ void finish_constants(const ConstArgs& a, const unsigned long long* ctx_dmin_inv, const unsigned long long* ctx_dmax,
                                 PlanHeader* hdr) {
  __shared__ unsigned long long s_span[32];
  __shared__ uint32_t s_w[kHistSegs];
  __shared__ uint32_t s_scan;
  const uint32_t tid = threadIdx.x, lane = tid & 31, S = (uint32_t)a.st.stage_stride, n_seg = a.n_ctx * S;
  unsigned long long span = 0;
  for (uint32_t c = tid; c < a.n_ctx; c += blockDim.x) {
    const unsigned long long lo = ~__ldcg(&ctx_dmin_inv[c]), hi = __ldcg(&ctx_dmax[c]);
    if (lo <= hi && hi - lo > span) span = hi - lo;
  }
  for (int o = 16; o; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, span, o);
    span = x > span ? x : span;
  }
  if (lane == 0) s_span[tid >> 5] = span;
  if (tid == 0) s_scan = a.force_scan;
  __syncthreads();
  if (tid == 0) {
    for (uint32_t w = 1; w < blockDim.x / 32; ++w) span = s_span[w] > span ? s_span[w] : span;
    set_key_width(hdr, span, a.sbits, a.ibits, a.key_sbits, a.arrival_order, a.st.d_priority != nullptr);
  }
  /* Few queues: their batch-window tables are COUNTED while the requests are packed (k_pack)
   * instead of being searched for in the sorted elements afterwards.  That needs the tables'
   * extents before any request has been looked at: a queue can have no window beyond that of its
   * ctx's latest deadline.  Entry 0 of a queue counts its requests with deadline < A, entry b + 1
   * those of window b; every queue has at least entry 0, so that the counts also give the queues'
   * lengths. */
  if (!RANGES && !a.win_hist) return;
  for (uint32_t q = tid; q < n_seg; q += blockDim.x) {   /* all queues side by side */
    const uint32_t c = q / S;
    const unsigned long long lo = ~__ldcg(&ctx_dmin_inv[c]), hi = __ldcg(&ctx_dmax[c]);
    PardSegConst* K = a.ktab + q;
    const long long A = __ldcg(&K->A), d = __ldcg(&K->d);
    uint32_t narrow = __ldcg(&K->narrow);
    if (RANGES) narrow = range_constants(K, A, d, narrow, lo, hi);
    if (a.win_hist) {
      uint32_t w = 1;
      if (!(narrow & kSegNoStage) && lo <= hi) {
        const long long X = (long long)hi - A;
        const unsigned long long nb = X < 0 ? 0ull : (unsigned long long)X / (unsigned long long)d + 1;
        if (nb >= 4096) s_scan = 1;                      /* kWinMaxPerSeg: too many windows for a table */
        else w = (uint32_t)nb + 1;
      }
      s_w[q] = w;
    }
  }
  if (!a.win_hist) return;
  __syncthreads();
  if (tid == 0) {
    uint32_t total = 0;
    bool scan = s_scan != 0;
    for (uint32_t q = 0; q < n_seg; ++q) {
      uint32_t w = s_w[q];
      if (total + w > kHistCap) { scan = true; w = 1; }
      a.win_off[q] = total;
      a.win_cnt[q] = w;
      total += w;
    }
    hdr->win_total = total;
    if (scan) hdr->use_scan = 1;
  }
}

/* Kept requests per queue -> first output slot of every queue, the number of
 * kCompactChunk-sized copy jobs before every queue, and the total.  One block,
 * eight queues per thread and round. */
template <int THREADS>
__device__ void kept_scan_block(const uint32_t* seg_kept, uint32_t n_seg, uint32_t* kept_base,
                                uint32_t* chunk_base, uint32_t* out_seg_kept, unsigned long long* out_n_kept) {
  constexpr int PER = 8, WARPS = THREADS / 32;
  __shared__ uint32_t s_a[32], s_b[32];
  __shared__ uint32_t s_ca, s_cb;
  if (threadIdx.x == 0) { s_ca = 0; s_cb = 0; }
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  /* a thread's eight entries as two 16-byte accesses where the arrays allow it */
  const bool vec_in = ((uintptr_t)seg_kept & 15) == 0;
  const bool vec_out = (((uintptr_t)kept_base | (uintptr_t)chunk_base) & 15) == 0;
  const bool vec_user = out_seg_kept && ((uintptr_t)out_seg_kept & 15) == 0;
  for (uint32_t base = 0; base < n_seg + 1; base += THREADS * PER) {
    const uint32_t i0 = base + threadIdx.x * PER;
    uint32_t v[PER], c[PER], x = 0, y = 0;
    if (vec_in && i0 + PER <= n_seg) {
      /* (L2 loads here and in kept_move_jobs: inside k_scan_path other blocks of the same kernel wrote these) */
      const uint4 a = __ldcg(reinterpret_cast<const uint4*>(seg_kept + i0)), b = __ldcg(reinterpret_cast<const uint4*>(seg_kept + i0 + 4));
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
      for (int k = 0; k < PER; ++k) v[k] = i0 + k < n_seg ? __ldcg(&seg_kept[i0 + k]) : 0;
    }
    if (vec_user && i0 + PER <= n_seg) {
      *reinterpret_cast<uint4*>(out_seg_kept + i0) = make_uint4(v[0], v[1], v[2], v[3]);
      *reinterpret_cast<uint4*>(out_seg_kept + i0 + 4) = make_uint4(v[4], v[5], v[6], v[7]);
    } else if (out_seg_kept) {
#pragma unroll
      for (int k = 0; k < PER; ++k) if (i0 + k < n_seg) out_seg_kept[i0 + k] = v[k];
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      c[k] = (v[k] + kCompactChunk - 1) / kCompactChunk;
      x += v[k];
      y += c[k];
    }
    const uint32_t tx = x, ty = y;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t p = __shfl_up_sync(0xffffffffu, x, o), q = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= (uint32_t)o) { x += p; y += q; }
    }
    if (lane == 31) { s_a[warp] = x; s_b[warp] = y; }
    __syncthreads();
    if (warp == 0) {
      const uint32_t a = lane < WARPS ? s_a[lane] : 0u, b = lane < WARPS ? s_b[lane] : 0u;
      uint32_t ta = a, tb = b;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t p = __shfl_up_sync(0xffffffffu, ta, o), q = __shfl_up_sync(0xffffffffu, tb, o);
        if (lane >= (uint32_t)o) { ta += p; tb += q; }
      }
      s_a[lane] = ta - a;
      s_b[lane] = tb - b;
    }
    __syncthreads();
    uint32_t ea = s_ca + s_a[warp] + x - tx, eb = s_cb + s_b[warp] + y - ty;   /* exclusive, before this thread's queues */
    uint32_t oa[PER], ob[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      oa[k] = ea; ob[k] = eb;
      ea += v[k];
      eb += c[k];
    }
    if (vec_out && i0 + PER <= n_seg + 1) {
      *reinterpret_cast<uint4*>(kept_base + i0) = make_uint4(oa[0], oa[1], oa[2], oa[3]);
      *reinterpret_cast<uint4*>(kept_base + i0 + 4) = make_uint4(oa[4], oa[5], oa[6], oa[7]);
      *reinterpret_cast<uint4*>(chunk_base + i0) = make_uint4(ob[0], ob[1], ob[2], ob[3]);
      *reinterpret_cast<uint4*>(chunk_base + i0 + 4) = make_uint4(ob[4], ob[5], ob[6], ob[7]);
    } else {
#pragma unroll
      for (int k = 0; k < PER; ++k) if (i0 + k <= n_seg) { kept_base[i0 + k] = oa[k]; chunk_base[i0 + k] = ob[k]; }
    }
    __syncthreads();
    if (threadIdx.x == THREADS - 1) { s_ca = ea; s_cb = eb; }
    __syncthreads();
  }
  if (threadIdx.x == 0 && out_n_kept) *out_n_kept = s_ca;
}

/* the lanes whose digit is d, from one ballot per digit bit */
template <int BITS>
__device__ __forceinline__ uint32_t digit_peers(uint32_t d, const uint32_t (&bal)[BITS]) {
  uint32_t m = 0xffffffffu;
#pragma unroll
  for (int k = 0; k < BITS; ++k) m &= ((d >> k) & 1u) ? bal[k] : ~bal[k];
  return m;
}

#include "pard_direct.cuh"

/* Constants of all queues, a block per ctx, with a launch of their own: calls with many queues, whose
 * blocks would hold up the prepass, and calls without requests. */
__global__ void __launch_bounds__(kConstThreads)
k_seg_const(const __grid_constant__ ConstArgs a, const unsigned long long* __restrict__ ctx_dmin_inv,
            const unsigned long long* __restrict__ ctx_dmax, PlanHeader* hdr) {
  pdl_wait();
  __shared__ CtxScratch scratch;
  if (ctx_constants<true>(a.pipes, a.n_pipelines, a.st, blockIdx.x, ~ctx_dmin_inv[blockIdx.x], ctx_dmax[blockIdx.x],
                    a.ktab + (size_t)blockIdx.x * a.st.stage_stride, scratch, sums_of(a, blockIdx.x)))
    set_status(hdr, PARD_EDATA);
  if (a.with_key_width && last_block_done(&hdr->seg_done)) finish_constants<false>(a, ctx_dmin_inv, ctx_dmax, hdr);
}

/* First tile of every ctx when the tiles are cut at ctx boundaries: the running sum of
 * ceil(requests of the ctx / kSortTile).  One block of 1,024 threads. */
__device__ __forceinline__ void tile_table(const uint32_t* __restrict__ ctx_start, uint32_t n_ctx, uint32_t* __restrict__ tile_first) {
  __shared__ uint32_t s_w[32];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t per = (n_ctx + 1023) / 1024;          /* contexts per thread, consecutive */
  const uint32_t c0 = tid * per, c1 = min(n_ctx, c0 + per);
  uint32_t sum = 0;
  for (uint32_t c = c0; c < c1; ++c) sum += (ctx_start[c + 1] - ctx_start[c] + kSortTile - 1) / kSortTile;
  uint32_t incl = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (uint32_t)o) incl += y;
  }
  if (lane == 31) s_w[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = s_w[lane];
    uint32_t x = w;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    s_w[lane] = x - w;
  }
  __syncthreads();
  uint32_t run = s_w[warp] + incl - sum;
  for (uint32_t c = c0; c < c1; ++c) {
    tile_first[c] = run;
    run += (ctx_start[c + 1] - ctx_start[c] + kSortTile - 1) / kSortTile;
  }
  if (c1 == n_ctx && c0 < n_ctx) tile_first[n_ctx] = run;
  if (n_ctx == 0 && tid == 0) tile_first[0] = 0;
}

/* The constants are there but for what they take from the deadline ranges (k_dir_count worked them out): a thread per
 * queue; the block that finishes last finds the key width.  (k_seg_const, which would do it all again, takes 13 us for 8,192 queues.)
 * The grid's last block lays out the tiles of the passes behind (k_tile_table). */
__global__ void __launch_bounds__(1024)
k_seg_finish(const __grid_constant__ ConstArgs a, const unsigned long long* __restrict__ ctx_dmin_inv,
             const unsigned long long* __restrict__ ctx_dmax, PlanHeader* hdr, const uint32_t* __restrict__ ctx_start, uint32_t* __restrict__ tile_first) {
  pdl_wait();
  if (hdr->direct) return;
  const uint32_t S = (uint32_t)a.st.stage_stride, q = blockIdx.x * 1024 + threadIdx.x;
  if (blockIdx.x == gridDim.x - 1) {
    tile_table(ctx_start, a.n_ctx, tile_first);
  } else if (q < a.n_ctx * S) {
    PardSegConst* K = a.ktab + q;
    range_constants(K, K->A, K->d, K->narrow, ~ctx_dmin_inv[q / S], ctx_dmax[q / S]);
  }
  if (a.with_key_width && last_block_done(&hdr->seg_done)) finish_constants<false>(a, ctx_dmin_inv, ctx_dmax, hdr);
}

/* ------------------------------------------------------------------------ */
/* prepass: one coalesced 16-byte read per request                           */
/* ------------------------------------------------------------------------ */
/* Range checks, the smallest / largest deadline of every ctx, and whether the requests stand in
 * deadline order.  A thread follows the ctx of the requests it reads and only hands its range over
 * when that ctx changes.  (ctx_dmin_inv holds the complement of the minimum, so that both arrays
 * start from zero and grow by atomicMax.)
 * TABLE: the ranges of all contexts are gathered in shared memory and handed to global memory once
 * per block, for requests of many contexts in mixed order: 2.5 M requests of 512 contexts cost
 * 203 us with two global atomics per request.  The table holds 32-bit offsets
 * from the first request's deadline; a deadline further than 2^31 us from it goes to global memory
 * directly.  Bound by the read of the requests: four in flight per thread at 48 registers keep
 * five blocks on a multiprocessor. */
constexpr int kPreUn = 4;
constexpr uint32_t kCountSegs = 256;             /* COUNT: most queues, one digit */

__device__ __noinline__ void const_block(const ConstArgs& a, uint32_t c, PlanHeader* hdr) {
  __shared__ CtxScratch scratch;
  if (ctx_constants<true>(a.pipes, a.n_pipelines, a.st, c, 0, 0, a.ktab + (size_t)c * a.st.stage_stride, scratch, sums_of(a, c)))
    set_status(hdr, PARD_EDATA);
}
__device__ __noinline__ void const_tail(const ConstArgs& a, const unsigned long long* ctx_dmin_inv, const unsigned long long* ctx_dmax,
                                        PlanHeader* hdr) {
  if (last_block_done(&hdr->seg_done)) finish_constants<true>(a, ctx_dmin_inv, ctx_dmax, hdr);
}

/* const_blocks: so many further blocks, the first ones of the grid, work out the queues' constants
 * meanwhile -- a chain of dependent loads that needs no deadline --, and the block that finishes last
 * completes them (one launch and its 8 us less for every call of up to 1,024 queues).
 * COUNT: calls in arrival order, sorted by the queue id alone.  Their order needs no look at the deadlines, and the
 * queues' lengths are all that the one pass wants, so they are counted here and k_pack is left out (k_sort_requests). */
template <bool TABLE, bool COUNT>
__global__ void __launch_bounds__(256, 5)
k_prepass(const uint4* __restrict__ req, uint32_t n, uint32_t n_ctx, uint32_t S,
          unsigned long long* __restrict__ ctx_dmin_inv, unsigned long long* __restrict__ ctx_dmax,
          PlanHeader* hdr, uint32_t const_blocks, const __grid_constant__ ConstArgs ca, uint32_t* __restrict__ hist) {
  pdl_wait();
  if (blockIdx.x < const_blocks) {
    const_block(ca, blockIdx.x, hdr);
    const_tail(ca, ctx_dmin_inv, ctx_dmax, hdr);
    return;
  }
  const uint32_t my_block = blockIdx.x - const_blocks, blocks = gridDim.x - const_blocks;
  extern __shared__ uint32_t s_range[];          /* TABLE: [n_ctx] complement of the smallest offset, [n_ctx] largest + 1, 0 = none */
  constexpr uint32_t kNone = 0xffffffffu;
  const uint32_t lane = threadIdx.x & 31;
  unsigned long long origin = 0;
  if (TABLE) {
    const uint4 f = __ldg(&req[0]);
    origin = (((unsigned long long)f.y << 32) | f.x) - (1ull << 31);
    for (uint32_t i = threadIdx.x; i < 2 * n_ctx; i += blockDim.x) s_range[i] = 0;
    __syncthreads();
  }
  __shared__ uint32_t s_count[COUNT ? 8 : 1][COUNT ? kCountSegs : 1];
  uint32_t* const count = s_count[COUNT ? threadIdx.x >> 5 : 0];
  if (COUNT) {
    for (uint32_t q = lane; q < kCountSegs; q += 32) count[q] = 0;
    __syncwarp();
  }
  bool time_back = COUNT, pair_back = COUNT;     /* see PlanHeader; looked for until both have been met */
  uint32_t run_ctx = kNone;
  unsigned long long lmin = ~0ull, lmax = 0;
  bool bad_seen = false;
  auto flush = [&]() {
    if (run_ctx == kNone) return;
    if (TABLE) {
      const unsigned long long a = lmin - origin, b = lmax - origin;
      if ((a >> 32) == 0 && b < 0xffffffffull) {
        atomicMax(&s_range[run_ctx], ~(uint32_t)a);
        atomicMax(&s_range[n_ctx + run_ctx], (uint32_t)b + 1u);
        return;
      }
    }
    atomicMax(&ctx_dmin_inv[run_ctx], ~lmin);
    atomicMax(&ctx_dmax[run_ctx], lmax);
  };
  /* whole warp (converged): one hand-over if all lanes follow the same ctx, else one per lane */
  auto warp_flush = [&]() {
    const uint32_t c0 = __shfl_sync(0xffffffffu, run_ctx, 0);
    if (__all_sync(0xffffffffu, run_ctx == c0)) {
      for (int o = 16; o; o >>= 1) {
        const unsigned long long a = __shfl_xor_sync(0xffffffffu, lmin, o);
        const unsigned long long b = __shfl_xor_sync(0xffffffffu, lmax, o);
        lmin = a < lmin ? a : lmin;
        lmax = b > lmax ? b : lmax;
      }
      if (lane == 0) flush();
    } else {
      flush();
    }
    run_ctx = kNone;
    lmin = ~0ull;
    lmax = 0;
  };
  const uint64_t chunk = (uint64_t)blockDim.x * kPreUn;
  for (uint64_t base = (uint64_t)my_block * chunk; base < n; base += (uint64_t)blocks * chunk) {
    uint4 r[kPreUn];
    const uint64_t first = base + (threadIdx.x >> 5) * (32 * kPreUn);   /* a warp's requests lie side by side */
#pragma unroll
    for (int i = 0; i < kPreUn; ++i) {
      const uint64_t j = first + i * 32 + lane;
      r[i] = j < n ? __ldg(&req[j]) : make_uint4(0u, 0u, kNone, 0u);
    }
    /* Are the requests in deadline order already?  Queues filled in arrival order with one
     * objective are; then the key's deadline field needs no radix pass.  Mostly a warp's 128 requests are
     * of one ctx and share the deadlines' high word: then low words are compared, one shuffle per row. */
    bool ordered = false;                        /* all 128 there, in range, of one ctx and in order: their range is that of the ends */
    if (!(time_back && pair_back)) {
      uint4 p = make_uint4(0u, 0u, 0u, 0u);      /* the request before the warp's first one */
      if (first > 0 && first < n) p = __ldg(&req[first - 1]);
      const uint32_t c0 = __shfl_sync(0xffffffffu, r[0].z, 0), h0 = __shfl_sync(0xffffffffu, r[0].y, 0);
      uint32_t other = first + 32 * kPreUn <= n && c0 < n_ctx && h0 < (uint32_t)(PARD_TIME_LIMIT_US >> 32) ? 0u : 1u, top = 0;
      uint32_t last = 0;                         /* lane 31: the row before */
      bool back = false;
#pragma unroll
      for (int i = 0; i < kPreUn; ++i) {
        const uint32_t px = __shfl_sync(0xffffffffu, lane == 31 ? last : r[i].x, (lane - 1) & 31);
        last = r[i].x;
        back |= r[i].x < px;                     /* (lane 0 of the first row compares with 0) */
        other |= (r[i].z ^ c0) | (r[i].y ^ h0);
        top = max(top, r[i].w & 0xffffu);
      }
      if (__all_sync(0xffffffffu, other == 0)) { /* what is left: the warp's first request against the one before */
        ordered = __all_sync(0xffffffffu, !back && top < S);
        const unsigned long long D = ((unsigned long long)r[0].y << 32) | r[0].x, pD = ((unsigned long long)p.y << 32) | p.x;
        const bool tb = back || (lane == 0 && D < pD), pb = back || (lane == 0 && (r[0].z < p.z || (r[0].z == p.z && D < pD)));
        time_back = time_back || __any_sync(0xffffffffu, tb);
        pair_back = pair_back || __any_sync(0xffffffffu, pb);
      } else {
        /* one shuffle per row and word: lane 31 hands out the row before, whose last request precedes
         * lane 0's (rows beyond the array compare as in order) */
        bool time_seen = false, pair_seen = false;
#pragma unroll
        for (int i = 0; i < kPreUn; ++i) {
          const uint4 q = i == 0 ? p : r[i > 0 ? i - 1 : 0];
          const bool give = lane == 31;
          const unsigned long long D = ((unsigned long long)r[i].y << 32) | r[i].x, qD = ((unsigned long long)q.y << 32) | q.x;
          const unsigned long long pD = __shfl_sync(0xffffffffu, give ? qD : D, (lane - 1) & 31);
          const uint32_t pc = __shfl_sync(0xffffffffu, give ? q.z : r[i].z, (lane - 1) & 31);
          const bool in = first + i * 32 + lane < n;
          time_seen |= in && D < pD;
          pair_seen |= in && (r[i].z < pc || (r[i].z == pc && D < pD));
        }
        time_back = time_back || __any_sync(0xffffffffu, time_seen);
        pair_back = pair_back || __any_sync(0xffffffffu, pair_seen);
      }
    }
    /* a new chunk usually lies in another ctx than the last one: hand the old one over together */
    if (__any_sync(0xffffffffu, run_ctx != kNone && r[0].z != run_ctx)) warp_flush();
    if (ordered) {
      if (r[0].z != run_ctx) {                   /* (uniform) */
        flush();
        run_ctx = r[0].z;
        lmin = ~0ull;
        lmax = 0;
      }
      const unsigned long long D0 = ((unsigned long long)r[0].y << 32) | r[0].x, D1 = ((unsigned long long)r[kPreUn - 1].y << 32) | r[kPreUn - 1].x;
      lmin = D0 < lmin ? D0 : lmin;
      lmax = D1 > lmax ? D1 : lmax;
      continue;
    }
#pragma unroll
    for (int i = 0; i < kPreUn; ++i) {
      if (first + i * 32 + lane >= n) continue;
      const unsigned long long D = ((unsigned long long)r[i].y << 32) | r[i].x;
      const uint32_t ctx = r[i].z, stage = r[i].w & 0xffffu;
      if (D >= (unsigned long long)PARD_TIME_LIMIT_US || ctx >= n_ctx || stage >= S) {
        bad_seen = true;
        if (COUNT) atomicAdd(&count[ctx < n_ctx && stage < S ? ctx * S + stage : 0u], 1u);   /* (request_element sorts it there) */
        continue;
      }
      if (COUNT) atomicAdd(&count[ctx * S + stage], 1u);
      if (ctx != run_ctx) {
        flush();
        run_ctx = ctx;
        lmin = ~0ull;
        lmax = 0;
      }
      lmin = D < lmin ? D : lmin;
      lmax = D > lmax ? D : lmax;
    }
  }
  /* One hand-over per block when the whole block stayed in one ctx (the usual case), and one store
   * of each flag per block until some block has made it: a pair of atomics per warp on the two
   * words of a single ctx cost 10 us at 1 M requests, a store per warp to the flags 16 us. */
  __shared__ uint32_t s_c[8], s_back[8];
  __shared__ unsigned long long s_min[8], s_max[8];
  const uint32_t warp = threadIdx.x >> 5;
  {
    const uint32_t c0 = __shfl_sync(0xffffffffu, run_ctx, 0);
    const bool whole = __all_sync(0xffffffffu, run_ctx == c0 || run_ctx == kNone);
    if (TABLE || !whole) warp_flush();
    for (int o = 16; o; o >>= 1) {
      const unsigned long long a = __shfl_xor_sync(0xffffffffu, lmin, o);
      const unsigned long long b = __shfl_xor_sync(0xffffffffu, lmax, o);
      lmin = a < lmin ? a : lmin;
      lmax = b > lmax ? b : lmax;
    }
    if (lane == 0) {
      s_c[warp] = TABLE || !whole ? kNone : c0;
      s_min[warp] = lmin;
      s_max[warp] = lmax;
      s_back[warp] = (time_back ? 1u : 0u) | (pair_back ? 2u : 0u);
    }
  }
  if (bad_seen) set_status(hdr, PARD_EDATA);
  __syncthreads();
  if (warp == 0) {
    const uint32_t back = __reduce_or_sync(0xffffffffu, lane < 8 ? s_back[lane] : 0u);
    uint32_t c = lane < 8 ? s_c[lane] : kNone;
    unsigned long long a = lane < 8 ? s_min[lane] : ~0ull, b = lane < 8 ? s_max[lane] : 0ull;
    const uint32_t c0 = __reduce_min_sync(0xffffffffu, c);
    if (__all_sync(0xffffffffu, c == c0 || c == kNone)) {
      for (int o = 4; o; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, a, o), y = __shfl_xor_sync(0xffffffffu, b, o);
        a = x < a ? x : a;
        b = y > b ? y : b;
      }
      c = lane == 0 ? c0 : kNone;
    }
    if (c != kNone) {                              /* (most blocks of a ctx find its range as wide as theirs already) */
      const unsigned long long x = __ldcg(&ctx_dmin_inv[c]), y = __ldcg(&ctx_dmax[c]);
      if (x < ~a) atomicMax(&ctx_dmin_inv[c], ~a);
      if (y < b) atomicMax(&ctx_dmax[c], b);
    }
    if (!COUNT && lane == 30 && (back & 1u) && __ldcg(&hdr->time_steps_back) == 0) hdr->time_steps_back = 1;
    if (!COUNT && lane == 31 && (back & 2u) && __ldcg(&hdr->pair_steps_back) == 0) hdr->pair_steps_back = 1;
  }
  if (TABLE) {
    __syncthreads();
    for (uint32_t c = threadIdx.x; c < n_ctx; c += blockDim.x) {
      if (s_range[n_ctx + c] == 0) continue;     /* none of the ctx's requests in this block's share */
      const unsigned long long lo = origin + (uint32_t)~s_range[c], hi = origin + (s_range[n_ctx + c] - 1u);
      if (__ldcg(&ctx_dmin_inv[c]) < ~lo) atomicMax(&ctx_dmin_inv[c], ~lo);
      if (__ldcg(&ctx_dmax[c]) < hi) atomicMax(&ctx_dmax[c], hi);
    }
  }
  if (COUNT)
    for (uint32_t q = threadIdx.x; q < n_ctx * S; q += 256) {
      uint32_t sum = 0;
#pragma unroll
      for (int w = 0; w < 8; ++w) sum += s_count[COUNT ? w : 0][q];
      if (sum) atomicAdd(&hist[q], sum);
    }
  if (const_blocks) const_tail(ca, ctx_dmin_inv, ctx_dmax, hdr);
}

constexpr uint32_t kPreTableCtx = 4096;          /* 32 KB of table: five blocks still fit a multiprocessor */
void launch_prepass(const uint4* req, uint32_t n, uint32_t n_ctx, uint32_t S, unsigned long long* ctx_dmin_inv,
                    unsigned long long* ctx_dmax, PlanHeader* hdr, uint32_t const_blocks, const ConstArgs& ca, int sms,
                    cudaStream_t stream, uint32_t* count = nullptr) {
  const uint32_t grid = std::min<uint32_t>((n + 256 * kPreUn - 1) / (256 * kPreUn), (uint32_t)sms * 5);
  /* the table pays once a block has more requests than the table has entries to clear and hand over */
  const bool table = n_ctx > 1 && n_ctx <= kPreTableCtx && n / grid >= 2 * n_ctx;
  launch_pdl(table ? (count ? k_prepass<true, true> : k_prepass<true, false>) : (count ? k_prepass<false, true> : k_prepass<false, false>),
             const_blocks + grid, 256, table ? 8ull * n_ctx : 0ull, stream, req, n, n_ctx, S, ctx_dmin_inv, ctx_dmax, hdr, const_blocks, ca, count);
}

__global__ void k_ctx_span(const unsigned long long* __restrict__ ctx_dmin_inv,
                           const unsigned long long* __restrict__ ctx_dmax, uint32_t n_ctx,
                           PlanHeader* hdr) {
  pdl_wait();
  if (hdr->direct) return;
  uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long span = 0;
  if (c < n_ctx && ~ctx_dmin_inv[c] <= ctx_dmax[c]) span = ctx_dmax[c] - ~ctx_dmin_inv[c];
  for (int o = 16; o; o >>= 1) {
    unsigned long long a = __shfl_xor_sync(0xffffffffu, span, o);
    span = a > span ? a : span;
  }
  if ((threadIdx.x & 31) == 0 && span) atomicMax(&hdr->span_max, span);
}

__global__ void k_key_width(uint32_t sbits, uint32_t ibits, PlanHeader* hdr, uint32_t arrival_order, uint32_t key_sbits,
                            uint32_t priority) {
  pdl_wait();
  if (hdr->direct) return;
  set_key_width(hdr, hdr->span_max, sbits, ibits, key_sbits, arrival_order, priority != 0);
}

/* one request's digits, of a key of one word */
__device__ __forceinline__ void count_digits(uint32_t* hist, uint32_t key, uint32_t npass) {
  if (npass > 0) atomicAdd(hist + (key & 255u), 1u);
  if (npass > 1) atomicAdd(hist + kBins + ((key >> 8) & 255u), 1u);
  if (npass > 2) atomicAdd(hist + 2 * kBins + ((key >> 16) & 255u), 1u);
  if (npass > 3) atomicAdd(hist + 3 * kBins + (key >> 24), 1u);
}

/* Request -> sort element; digit histograms of every pass.  Bound by instructions, so the usual call --
 * every request in range, low budget first, keys of one word, window tables within the shared counters
 * -- has a loop of its own that tests none of it per request (2^24 requests with window counts:
 * 98 -> 77 us). */
constexpr uint32_t kPackCtx = 64;
template <bool WIN>
__global__ void __launch_bounds__(256)
k_pack(const uint4* __restrict__ req, uint32_t n, uint32_t n_ctx, uint32_t S,
       const unsigned long long* __restrict__ ctx_dmin_inv, const unsigned long long* __restrict__ ctx_dmax,
       const uint8_t* __restrict__ priority, uint32_t ibits,
       PlanHeader* __restrict__ hdr, unsigned long long* __restrict__ dst,
       uint32_t* __restrict__ hist, uint32_t local_candidate,
       const PardSegConst* __restrict__ ktab, const uint32_t* __restrict__ win_off,
       const uint32_t* __restrict__ win_cnt, uint32_t* __restrict__ whist) {
  pdl_wait();
  __shared__ uint32_t s_hist[kMaxPasses * kBins];
  /* WIN: the batch-window tables are counted here (few queues); per-queue constants in shared memory */
  constexpr uint32_t kWinWords = 2048;                      /* more would cost the kernel its occupancy */
  __shared__ uint32_t s_win[WIN ? kWinWords : 1];
  __shared__ long long s_A[WIN ? kHistSegs : 1], s_d[WIN ? kHistSegs : 1];
  __shared__ unsigned long long s_magic[WIN ? kHistSegs : 1];
  __shared__ uint4 s_wcon[WIN ? kHistSegs : 1];            /* per queue: A_rel, first table entry, entries, A_rel and d fit 32 bits */
  /* Few contexts: the low words of their smallest deadlines in shared memory (a replay's epochs, 16 contexts, 451.6 -> 449.7 us.
   * 512 contexts with priorities, all in such tables: the kernel 20.7 -> 24.9). */
  __shared__ uint32_t s_low[kPackCtx];
  const bool table = n_ctx > 1 && n_ctx <= kPackCtx;
  if (hdr->wide || sort_is_local(hdr, local_candidate)) return;   /* sorted block by block: k_sort_local read the requests itself */
  const uint32_t npass = hdr->npass, dbits = hdr->dbits, pshift = hdr->pshift;
  for (uint32_t i = threadIdx.x; i < npass * kBins; i += blockDim.x) s_hist[i] = 0;
  /* The counters are kept in as many copies as fit (a power of two, at most one per lane), lane l
   * counting in copy l mod copies: requests of one warp that fall into the same entry -- the
   * usual case when most of a queue is expired, or lies in few windows -- then hit different words. */
  uint32_t win_total = 0, copies = 1, my_copy = 0;
  bool win_shared = false;                                  /* tables beyond kWinWords entries are counted in global memory */
  bool win_derive = false, all_narrow = true;
  if (WIN) {
    win_total = (uint32_t)hdr->win_total;
    win_shared = win_total <= kWinWords;
    while (copies < 32 && 2 * copies * win_total <= kWinWords) copies *= 2;
    my_copy = (threadIdx.x & (copies - 1)) * win_total;
    if (win_shared) for (uint32_t i = threadIdx.x; i < win_total * copies; i += blockDim.x) s_win[i] = 0;
    /* When the queue id lies inside the last pass's digit the queues' lengths can be read off that
     * pass's digit counts (see k_windows), and entry 0 of a queue -- its requests with deadline < A,
     * often most of an overloaded queue -- is its length minus its other entries: such requests
     * are then not counted here at all. */
    win_derive = npass > 0 && hdr->keybits - (dbits - pshift) <= hdr->keybits - 8 * (npass - 1);
    for (uint32_t q = threadIdx.x; q < n_ctx * S; q += blockDim.x) {
      const PardSegConst K = ktab[q];
      s_A[q] = K.A; s_d[q] = K.d; s_magic[q] = K.d_magic;
      all_narrow = all_narrow && (K.narrow & (kSegNarrow | kSegNoStage)) == kSegNarrow;
      s_wcon[q] = make_uint4((uint32_t)narrow_A(K), win_off[q], win_cnt[q], (K.narrow & (kSegNarrow | kSegNoStage)) == kSegNarrow ? 1u : 0u);
    }
  }
  if (table && threadIdx.x < n_ctx) s_low[threadIdx.x] = (uint32_t)~ctx_dmin_inv[threadIdx.x];
  bool plain = !hdr->bad_input && !priority && hdr->keybits + pshift <= 32 && dbits <= 29;
  if (WIN) plain = __syncthreads_and(plain && win_shared && all_narrow);
  else __syncthreads();
  const unsigned long long dmask = dbits >= 64 ? ~0ull : ((1ull << dbits) - 1);
  /* n < 2^30: positions and strides in 32 bits (the grid has at most n threads) */
  const uint32_t stride = gridDim.x * blockDim.x;
  const bool key32 = hdr->keybits + pshift <= 32;   /* the key fits one word: its digits are peeled off that word */
  const bool off32 = dbits <= 29;              /* deadline offsets fit signed 32-bit arithmetic */
  uint32_t cur_ctx = 0xffffffffu;              /* the ctx whose deadline range is at hand (requests of a ctx mostly sit together) */
  unsigned long long cmin = 0, cmax = 0;
  constexpr int kUn = 4;                       /* requests in flight per thread (measured against 1: 74 vs 78.5 us at 2^24) */
  if (plain) {
    const uint32_t up = 1u << ibits;
    uint32_t low = 0;                          /* low word of the ctx's smallest deadline */
    for (uint32_t j0 = blockIdx.x * blockDim.x + threadIdx.x; j0 < n; j0 += stride * kUn) {
      if (threadIdx.x < kUn)                   /* the next round's requests, 256 in a row each (2^24: 5 us less) */
        l2_ahead(reinterpret_cast<const unsigned long long*>(req), 2ull * (j0 - threadIdx.x), 2ull * stride * (kUn + threadIdx.x), 512, 2ull * n);
      uint4 rr[kUn];
#pragma unroll
      for (int u = 0; u < kUn; ++u) {
        const uint32_t j = j0 + (uint32_t)u * stride;
        if (j < n) rr[u] = __ldg(&req[j]);
      }
#pragma unroll
      for (int u = 0; u < kUn; ++u) {
        const uint32_t j = j0 + (uint32_t)u * stride;
        if (j >= n) break;
        const uint4 r = rr[u];
        if (table) {
          low = s_low[r.z];
        } else if (r.z != cur_ctx) {
          cur_ctx = r.z;
          low = (uint32_t)~ctx_dmin_inv[cur_ctx];
        }
        const uint32_t seg = r.z * S + (r.w & 0xffffu), off = (r.x - low) & (uint32_t)dmask, key = (seg << dbits) | off;
        dst[j] = (unsigned long long)key * up + j;
        count_digits(s_hist, key >> pshift, npass);
        if (WIN) {
          const uint4 c = s_wcon[seg];
          const int32_t X = (int32_t)off - (int32_t)c.x;
          const uint32_t h = X < 0 ? 0u : min(div_magic32((uint32_t)X, s_magic[seg]) + 1, c.z - 1);   /* never beyond the queue's entries */
          if (h || !win_derive) atomicAdd(&s_win[my_copy + c.y + h], 1u);
        }
      }
    }
  } else
  for (uint32_t j0 = blockIdx.x * blockDim.x + threadIdx.x; j0 < n; j0 += stride * kUn) {
    uint4 rr[kUn];
#pragma unroll
    for (int u = 0; u < kUn; ++u) {
      const uint32_t j = j0 + (uint32_t)u * stride;
      if (j < n) rr[u] = __ldg(&req[j]);
    }
#pragma unroll
    for (int u = 0; u < kUn; ++u) {
      const uint32_t j = j0 + (uint32_t)u * stride;
      if (j >= n) break;
      const uint4 r = rr[u];
      const uint32_t ctx = r.z, stage = r.w & 0xffffu;
      const bool ok = ctx < n_ctx && stage < S;
      const uint32_t seg = ok ? ctx * S + stage : 0u;
      if (ok && ctx != cur_ctx) {
        cur_ctx = ctx;
        cmin = ~ctx_dmin_inv[ctx];
        cmax = ctx_dmax[ctx];
      }
      /* ascending offsets give the queue's decision order: deadlines counted up from the ctx's
       * smallest, or down from its largest when the queue is served high budget first */
      const bool high_first = ok && priority && __ldg(&priority[seg]) != 0;
      uint32_t h = 0;                            /* the request's entry in its queue's window table: 0 for deadline < A, else window + 1 */
      bool count = false;
      uint4 c = make_uint4(0u, 0u, 1u, 0u);      /* A - ctx's smallest deadline (if it fits 32 bits), first entry, entries, fits? */
      if (key32 && off32) {
        /* everything in single words: the offset is below 2^29, so the low words of the 64-bit
         * difference are the difference */
        const uint32_t off = ok ? ((high_first ? (uint32_t)cmax - r.x : r.x - (uint32_t)cmin) & (uint32_t)dmask) : 0u;
        uint32_t key = (seg << dbits) | off;
        if (WIN && ok) {
          c = s_wcon[seg];
          count = true;
          if (c.w) {
            const int32_t X = (int32_t)off - (int32_t)c.x;
            if (X >= 0) {
              const uint32_t b = div_magic32((uint32_t)X, s_magic[seg]);
              h = b + 1 < c.z ? b + 1 : c.z - 1;   /* never beyond the queue's entries (a queue decided by scanning has one) */
            }
          } else {
            const long long X = (long long)(((unsigned long long)r.y << 32) | r.x) - s_A[seg];
            if (X >= 0) {
              const unsigned long long M = s_magic[seg];
              const unsigned long long b = (((unsigned long long)X >> 32) == 0 && M) ? div_magic32((uint32_t)X, M)
                                                                                    : (unsigned long long)X / (unsigned long long)s_d[seg];
              h = b + 1 < c.z ? (uint32_t)b + 1 : c.z - 1;
            }
          }
        }
        *reinterpret_cast<uint2*>(dst + j) = make_uint2((key << ibits) | j, __funnelshift_l(key, 0u, ibits));
        uint32_t* hp = s_hist;
        key >>= pshift;                          /* <= 29 here */
        for (uint32_t p = 0; p < npass; ++p, hp += kBins, key >>= 8) atomicAdd(hp + (key & 255u), 1u);
      } else {
        const unsigned long long D = ((unsigned long long)r.y << 32) | r.x;
        const unsigned long long off = ok ? ((high_first ? cmax - D : D - cmin) & dmask) : 0ull;
        unsigned long long key = ((unsigned long long)seg << dbits) | off;
        if (WIN && ok) {
          c = s_wcon[seg];
          count = true;
          const long long X = (long long)D - s_A[seg];
          if (X >= 0) {
            const unsigned long long M = s_magic[seg];
            const unsigned long long b = (((unsigned long long)X >> 32) == 0 && M) ? div_magic32((uint32_t)X, M)
                                                                                  : (unsigned long long)X / (unsigned long long)s_d[seg];
            h = b + 1 < c.z ? (uint32_t)b + 1 : c.z - 1;
          }
        }
        dst[j] = (key << ibits) | j;
        uint32_t* hp = s_hist;
        key >>= pshift;
        for (uint32_t p = 0; p < npass; ++p, hp += kBins, key >>= 8) atomicAdd(hp + ((uint32_t)key & 255u), 1u);
      }
      if (WIN) {
        /* a request flagged by the prepass (its element is its index alone) sorts into queue 0 and is
         * counted there, entry 0: the counts stay the queues' lengths */
        if (!ok) { c.y = 0; h = 0; count = true; }
        if (count && (h != 0 || !win_derive)) {
          if (win_shared) atomicAdd(&s_win[my_copy + c.y + h], 1u);
          else atomicAdd(&whist[c.y + h], 1u);
        }
      }
    }
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < npass * kBins; i += blockDim.x)
    if (s_hist[i]) atomicAdd(&hist[i], s_hist[i]);
  if (WIN && win_shared)
    for (uint32_t i = threadIdx.x; i < win_total; i += blockDim.x) {
      uint32_t sum = 0;
      for (uint32_t r = 0; r < copies; ++r) sum += s_win[r * win_total + i];
      if (sum) atomicAdd(&whist[i], sum);
    }
}

/* ------------------------------------------------------------------------ */
/* window tables: the decision pass without a scan                           */
/* ------------------------------------------------------------------------ */
/* Inside one queue the threshold u is a step function of the deadline: every
 * request whose deadline falls into the same batch window
 *     b = floor((D - A) / d)
 * has u = cap * (b + 1) (requests with D < A have u = 0).  The running minimum
 * of u_t - t that fixes the admitted position therefore only changes at the
 * window boundaries: with P[b] = number of requests of the queue whose window
 * is below b, the minimum over a complete window b is u(b) - (P[b+1] - 1), and
 *     E[b] = minimum over all complete runs before window b
 * is a prefix minimum over at most a few thousand windows per queue.  A request
 * at queue position r in window b then has
 *     min_{t<r}(u_t - t) = min(E[b], u(b) - (r - 1) if r > P[b])
 * with no reference to any other request.  P comes from a search in the sorted
 * elements (k_windows) or a count while they are packed, E and the raw-mode kept counts Kp from a
 * per-queue prefix pass over the windows.  Queues with more than kWinMaxPerSeg
 * windows, or more windows in total than the table holds, make the call fall
 * back to the scan kernels (same results). */
struct __align__(16) WinEntry {
  uint32_t P;      /* requests of the queue in earlier windows (or expired)       */
  int32_t E;       /* min of u_t - t over those requests, kWinInf if there is none */
  uint32_t Kp;     /* raw mode: kept requests among them                          */
  uint32_t pad;
};
constexpr uint32_t kWinMaxPerSeg = 4096;
/* window of a non-negative X = D - A */
__device__ __forceinline__ unsigned long long win_of(unsigned long long X, const PardSegConst& K) {
  if ((X >> 32) == 0 && K.d_magic) return div_magic32((uint32_t)X, K.d_magic);
  return X / (unsigned long long)K.d;
}

/* E and Kp of the table of one queue (cnt >= 1 entries): the warp runs over the queue's windows, 32 at a
 * time.  SHARED: the P are in shared memory, s_P, and go out with the rest of their entries. */
template <bool SHARED = false>
__device__ __forceinline__ uint32_t win_prefix_warp(uint32_t cap, WinEntry* __restrict__ tab, uint32_t cnt, uint32_t lane, uint32_t raw,
                                                    const uint32_t* s_P = nullptr) {
  auto P_of = [&](uint32_t b) { return SHARED ? s_P[b] : __ldcg(&tab[b].P); };
  auto put = [&](uint32_t b, uint32_t P, int32_t E, uint32_t Kp) {
    if (SHARED) *reinterpret_cast<uint4*>(&tab[b]) = make_uint4(P, (uint32_t)E, Kp, 0u);
    else { tab[b].E = E; tab[b].Kp = Kp; }
  };
  const uint32_t P0 = P_of(0);
  int32_t e_carry = P0 > 0 ? -(int32_t)(P0 - 1) : kWinInf;     /* the expired run: u = 0 */
  uint32_t k_carry = 0;
  if (lane == 0) put(0, P0, e_carry, 0);
  for (uint32_t b0 = 0; b0 + 1 < cnt; b0 += 32) {              /* windows b0..b0+31 -> entries b0+1.. */
    const uint32_t b = b0 + lane;
    int32_t val = kWinInf;
    uint32_t kept = 0, q = 0;
    if (b + 1 < cnt) {
      const uint32_t p = P_of(b);
      q = P_of(b + 1);
      if (q > p) {
        const uint32_t u = win_u(b, cap);
        val = (int32_t)u - (int32_t)(q - 1);
        const uint32_t top = u < q ? u : q;
        kept = top > p ? top - p : 0;
      }
    }
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t v2 = __shfl_up_sync(0xffffffffu, val, o);
      const uint32_t k2 = __shfl_up_sync(0xffffffffu, kept, o);
      if (lane >= (uint32_t)o) { val = min(val, v2); kept += k2; }
    }
    const int32_t e_inc = min(e_carry, val);
    const uint32_t k_inc = k_carry + kept;
    if (b + 1 < cnt) put(b + 1, q, e_inc, k_inc);
    e_carry = __shfl_sync(0xffffffffu, e_inc, 31);
    k_carry = __shfl_sync(0xffffffffu, k_inc, 31);
  }
  /* With the table complete the queue's number of kept requests is known before any request has
   * been decided: the last entry closes the queue (P = its length n), the running Kp counts the
   * kept requests under raw positions, and the running E is the minimum of u_t - t over the whole
   * queue, so that the admitted count behind the last request is n - 1 + min(E, 1). */
  const uint32_t n_q = P_of(cnt - 1);
  return n_q == 0 ? 0u : (raw ? k_carry : (uint32_t)((int32_t)n_q - 1 + min(e_carry, 1)));
}

/* The window tables of a call with few queues, from the counts k_pack took: P is the running sum
 * of a queue's counts, E and Kp follow as in the searched tables, and the queues' first positions
 * are the running sum of their lengths.  By one block, a warp per queue: a block of the first sort
 * kernel's launch, beside the sort (the counts do not depend on the order of the elements; as a launch
 * of its own it held the sort up by 6 us). */
struct WinCountArgs {
  uint32_t on, n_seg, raw, sbits;
  const PardSegConst* ktab;
  const uint32_t* whist;
  const uint32_t* win_off;
  const uint32_t* win_cnt;
  WinEntry* wtab;
  uint32_t* seg_off;
  uint32_t* out_seg_off;
  uint32_t* seg_kept;
  uint32_t* out_seg_kept;
  uint32_t* kept_base;
  unsigned long long* out_n_kept;
  const uint32_t* hist;
};
__device__ __noinline__ void win_from_counts(PlanHeader* hdr, const WinCountArgs& a) {
  if (hdr->wide) return;
  const uint32_t n_seg = a.n_seg;
  __shared__ uint32_t s_len[kHistSegs], s_kept[kHistSegs];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  /* entry 0 left uncounted by k_pack (same condition there): the queue's length, from the last
   * pass's digit counts, minus its other entries */
  const uint32_t npass = hdr->npass;
  const uint32_t top_bits = npass ? hdr->keybits - 8 * (npass - 1) : 0;
  const bool derive = npass > 0 && a.sbits <= top_bits;
  for (uint32_t q = warp; q < n_seg; q += blockDim.x / 32) {
    const uint32_t off = a.win_off[q], cnt = a.win_cnt[q];
    uint32_t entry0 = 0;
    if (derive) {
      const uint32_t* h = a.hist + (npass - 1) * kBins;
      const uint32_t d0 = min(q << (top_bits - a.sbits), (uint32_t)kBins), d1 = min((q + 1) << (top_bits - a.sbits), (uint32_t)kBins);
      uint32_t len = 0, others = 0;
      for (uint32_t d = d0 + lane; d < d1; d += 32) len += h[d];
      for (uint32_t b = 1 + lane; b < cnt; b += 32) others += a.whist[off + b];
      for (int o = 16; o; o >>= 1) {
        len += __shfl_xor_sync(0xffffffffu, len, o);
        others += __shfl_xor_sync(0xffffffffu, others, o);
      }
      entry0 = len - others;
    }
    uint32_t run = 0;
    for (uint32_t b0 = 0; b0 < cnt; b0 += 32) {
      const uint32_t b = b0 + lane;
      uint32_t x = b < cnt ? a.whist[off + b] : 0u;
      if (derive && b == 0) x = entry0;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x += y;
      }
      if (b < cnt) a.wtab[off + b].P = run + x;        /* requests of the queue up to and including entry b's */
      run += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) s_len[q] = run;
    __threadfence_block();
    __syncwarp();
    /* P as the decision reads it: entry b = requests in windows below b, i.e. the sum up to entry b */
    const uint32_t kept = cnt ? win_prefix_warp(a.ktab[q].cap, a.wtab + off, cnt, lane, a.raw) : 0u;
    if (lane == 0) s_kept[q] = kept;      /* the queue's kept count, known before the sort */
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const bool scan = hdr->use_scan != 0;                /* then the scan path counts and packs */
    uint32_t first = 0, kept = 0;
    for (uint32_t q = 0; q < n_seg; ++q) {
      a.seg_off[q] = first;
      if (a.out_seg_off) a.out_seg_off[q] = first;
      first += s_len[q];
      if (!scan) {
        a.kept_base[q] = kept;
        a.seg_kept[q] = s_kept[q];
        if (a.out_seg_kept) a.out_seg_kept[q] = s_kept[q];
        kept += s_kept[q];
      }
    }
    a.seg_off[n_seg] = first;
    if (a.out_seg_off) a.out_seg_off[n_seg] = first;
    if (!scan && a.out_n_kept) *a.out_n_kept = kept;
  }
}

/* ------------------------------------------------------------------------ */
/* one LSD radix pass (8 bits), stable, tile prefixes by decoupled look-back */
/* ------------------------------------------------------------------------ */
/* Tile = kSortTile elements; every warp owns a run of consecutive elements
 * (kItemsLo rounds of 32 for the warps that also do the look-back, kItemsHi
 * rounds for the others) and visits it 32 at a time, so the tile order is
 * (warp, round, lane).
 *   1. every warp counts its digits (shared atomics, order irrelevant);
 *   2. thread d turns the counts of digit d into the first tile-local slot of
 *      every (warp, digit) and publishes the tile's count for the look-back;
 *   3. the lower part of the block adds up the counts of all earlier tiles
 *      (look-back, kLookBatch tiles per memory round trip) while the other
 *      warps already rank;
 *   4. ranking: the lanes that hold the same digit find each other through a
 *      shared word (atomic OR), take consecutive slots in lane order and drop
 *      their elements into the shared tile buffer, now sorted by digit;
 *   5. the buffer is written out, run by run, to the digit's global range.
 * Large tiles keep the number of tiles in flight, and with it the depth of the
 * look-back, small. */
/* Hands in the `mine` pieces of work that this block has finished and waits until all `target` of them have
 * been handed in to `word` (from zero; k_scan_path: until a flag is set); what their blocks wrote before is
 * visible to this block afterwards.  A block comes here when it has found nothing left to take, so the pieces outstanding are with blocks that
 * run already: the wait needs no block that has yet to be placed.  Bounded all the same: about half a
 * second, then PARD_ETIMEOUT and false in every block. */
__device__ bool finish_pieces(PlanHeader* hdr, uint32_t* word, uint32_t mine, uint32_t target) {
  __shared__ uint32_t s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    if (mine) {
      __threadfence();
      atomicAdd(word, mine);
    }
    uint32_t spins = 0;
    bool ok = true;
    while (ld_relaxed(word) < target) {     /* up to about half a second: other work may hold multiprocessors for a while */
      if (++spins > 8 * kSpinLimit || ((spins & 15) == 0 && ld_relaxed(&hdr->aborted))) { ok = false; break; }
      __nanosleep(200);
    }
    if (!ok) set_aborted(hdr);
    __threadfence();
    s_ok = ok ? 1u : 0u;
  }
  __syncthreads();
  return s_ok != 0;
}

constexpr int kItemsReq = (kItemsLo + kItemsHi) / 2;     /* k_sort_requests: its loads take the registers of the longer shares (10 and 22: 200 bytes spilled) */

struct SortSmem {
  unsigned long long keys[kSortTile];
  uint32_t slot[kSortThreads / 32][kBins];    /* counts, then next free tile-local slot per (warp, digit) */
  uint32_t match[kSortThreads / 32][kBins];   /* lanes currently holding the digit */
  uint32_t dstart[kBins];
  uint32_t gofs[kBins];
  uint32_t scan[2][kSortThreads / 32];
  uint32_t tile;
  uint32_t abort;
  uint32_t done;                              /* tiles of the pass at hand that this block has finished */
  uint32_t ctx, lo_tile, base, limit, first;   /* the tile's ctx and range when passes stay inside the contexts */
};

/* A pass that takes the requests themselves instead of elements (k_sort_requests), and, for the rules that look no
 * further than the deadline, what k_policy_terms would write beside them. */
struct RequestPass {
  const uint4* req;
  const unsigned long long* ctx_dmin_inv;
  uint32_t n_ctx, S, nexus;
  const PardSegConst* ktab;
  uint32_t* rounds;                                    /* [n] rounds that a request still fits, or null */
};
/* k_pack's element of a request, low budget first; cmin: its ctx's smallest deadline */
__device__ __forceinline__ unsigned long long request_element(const RequestPass& rp, const uint4& r, uint32_t j, uint32_t dbits, uint32_t ibits,
                                                              unsigned long long cmin, bool plain) {
  const uint32_t ctx = r.z, stage = r.w & 0xffffu;
  if (plain) {                                         /* the key fits one word, deadline offsets 31 bits */
    const uint32_t key = (ctx * rp.S + stage) << dbits | ((r.x - (uint32_t)cmin) & ((1u << dbits) - 1));
    return (unsigned long long)(ctx < rp.n_ctx && stage < rp.S ? key : 0u) * (1u << ibits) + j;
  }
  const unsigned long long off = ((((unsigned long long)r.y << 32) | r.x) - cmin) & ((1ull << dbits) - 1);   /* dbits < 64: see set_key_width */
  const unsigned long long e = ((unsigned long long)(ctx * rp.S + stage) << dbits | off) << ibits;
  return (ctx < rp.n_ctx && stage < rp.S ? e : 0ull) | j;
}

/* one warp's share of step 1: ITEMS rounds of 32 consecutive elements */
template <int ITEMS, bool L2, int CAP>
__device__ __forceinline__ void sort_load_count(unsigned long long (&key)[CAP], const unsigned long long* src,
                                                uint64_t first, uint32_t n, uint32_t shift, uint32_t* slot_row,
                                                uint32_t lane, uint32_t dig_mask, int items) {
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    if (i >= items) break;                             /* the same for the whole warp */
    const uint64_t j = first + i * 32 + lane;
    key[i] = j < n ? (L2 ? __ldcg(src + j) : src[j]) : ~0ull;
  }
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    if (i >= items) break;
    atomicAdd(&slot_row[(uint32_t)(key[i] >> shift) & dig_mask], 1u);
  }
}
/* the same in two steps, from the requests */
template <int ITEMS, int CAP>
__device__ __forceinline__ void sort_load_requests(unsigned long long (&key)[CAP], const RequestPass& rp, uint64_t first, uint32_t n,
                                                   uint32_t dbits, uint32_t ibits, uint32_t lane, int items, bool plain) {
  constexpr int kUn = 4;                               /* requests under way together */
  const bool one = rp.n_ctx == 1;
  const unsigned long long only = ~__ldg(&rp.ctx_dmin_inv[0]);
#pragma unroll
  for (int i0 = 0; i0 < ITEMS; i0 += kUn) {
    if (i0 >= items) break;                            /* the same for the whole warp */
    uint4 r[kUn];
    unsigned long long cmin[kUn];
#pragma unroll
    for (int u = 0; u < kUn; ++u) r[u] = __ldg(&rp.req[min(first + (i0 + u) * 32 + lane, (uint64_t)n - 1)]);
#pragma unroll
    for (int u = 0; u < kUn; ++u) cmin[u] = one ? only : ~__ldg(&rp.ctx_dmin_inv[min(r[u].z, rp.n_ctx - 1)]);
#pragma unroll
    for (int u = 0; u < kUn; ++u) {
      if (i0 + u >= ITEMS) break;
      const uint64_t j = first + (i0 + u) * 32 + lane;
      key[i0 + u] = j < n ? request_element(rp, r[u], (uint32_t)j, dbits, ibits, cmin[u], plain) : ~0ull;
    }
  }
}
template <int ITEMS, int CAP>
__device__ __forceinline__ void sort_count(const unsigned long long (&key)[CAP], uint32_t shift, uint32_t* slot_row, uint32_t dig_mask, int items) {
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    if (i >= items) break;
    atomicAdd(&slot_row[(uint32_t)(key[i] >> shift) & dig_mask], 1u);
  }
}

/* one warp's share of step 4 */
template <int ITEMS, int CAP>
__device__ __forceinline__ void sort_rank_drop(const unsigned long long (&key)[CAP], uint32_t shift,
                                               uint32_t* slot_row, uint32_t* match_row, unsigned long long* keys,
                                               uint32_t lanebit, int items = ITEMS, uint32_t dig_mask = 255u) {
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    if (i >= items) break;                             /* the same for the whole block */
    const uint32_t d = (uint32_t)(key[i] >> shift) & dig_mask;
    atomicOr(&match_row[d], lanebit);
    __syncwarp();
    const uint32_t grp = match_row[d];
    const uint32_t below = grp & (lanebit - 1);
    const uint32_t first = slot_row[d];                /* same word for the whole group */
    __syncwarp();
    if (below == 0) {                                  /* lowest lane of the group */
      slot_row[d] = first + __popc(grp);
      match_row[d] = 0;
    }
    keys[first + __popc(below)] = key[i];
    __syncwarp();
  }
}

/* The same two steps for a pass whose digit has one or two bits (the top pass of a key of 8k + 1
 * or 8k + 2 bits): the lanes that hold the same digit find each other by one ballot per digit
 * bit, lane j keeps the warp's running count of digit j in a register, and neither the counting
 * nor the ranking touches shared memory apart from the key's own store.  Measured at 2^24
 * elements: a 1-bit pass 89 us against 120 us through the generic code (where 32 lanes hammer two
 * counters); with four ballots (a 4-bit digit) the instructions outweigh the saved shared-memory
 * traffic (16.2 us against 14.5 us at 2^20 elements), so wider digits stay on the generic code.
 * The 89 us are what a pass costs with ranking almost free: tile load, write-out, scans and
 * barriers.  Full tiles only (no padding keys). */
template <int ITEMS, int BITS, bool L2, int CAP>
__device__ __forceinline__ void sort_load_count_few(unsigned long long (&key)[CAP], const unsigned long long* src,
                                                    uint64_t first, uint32_t shift, uint32_t* slot_row, uint32_t lane, int items) {
#pragma unroll
  for (int i = 0; i < ITEMS; ++i)
    if (i < items) key[i] = L2 ? __ldcg(src + first + i * 32 + lane) : src[first + i * 32 + lane];
  uint32_t mine = 0;                                     /* lane j: keys of this warp with digit j */
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    if (i >= items) break;
    const uint32_t d = (uint32_t)(key[i] >> shift);
    uint32_t bal[BITS];
#pragma unroll
    for (int k = 0; k < BITS; ++k) bal[k] = __ballot_sync(0xffffffffu, (d >> k) & 1u);
    mine += __popc(digit_peers<BITS>(lane, bal));
  }
  if (lane < (1u << BITS)) slot_row[lane] = mine;
}

template <int ITEMS, int BITS, int CAP>
__device__ __forceinline__ void sort_count_few(const unsigned long long (&key)[CAP], uint32_t shift, uint32_t* slot_row, uint32_t lane, int items) {
  uint32_t mine = 0;                                     /* lane j: keys of this warp with digit j */
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    if (i >= items) break;
    const uint32_t d = (uint32_t)(key[i] >> shift);
    uint32_t bal[BITS];
#pragma unroll
    for (int k = 0; k < BITS; ++k) bal[k] = __ballot_sync(0xffffffffu, (d >> k) & 1u);
    mine += __popc(digit_peers<BITS>(lane, bal));
  }
  if (lane < (1u << BITS)) slot_row[lane] = mine;
}

template <int ITEMS, int CAP, int BITS>
__device__ __forceinline__ void sort_rank_drop_few(const unsigned long long (&key)[CAP], uint32_t shift,
                                                   const uint32_t* slot_row, unsigned long long* keys, uint32_t lane, int items) {
  uint32_t next = lane < (1u << BITS) ? slot_row[lane] : 0u;   /* lane j: next free slot of digit j for this warp */
  const uint32_t below = (1u << lane) - 1;
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    if (i >= items) break;
    const uint32_t d = (uint32_t)(key[i] >> shift) & ((1u << BITS) - 1);
    uint32_t bal[BITS];
#pragma unroll
    for (int k = 0; k < BITS; ++k) bal[k] = __ballot_sync(0xffffffffu, (d >> k) & 1u);
    const uint32_t grp = digit_peers<BITS>(d, bal);
    const uint32_t first = __shfl_sync(0xffffffffu, next, d);
    keys[first + __popc(grp & below)] = key[i];
    next += __popc(digit_peers<BITS>(lane, bal));
  }
}

/* digit width known at run time only: one instantiation per width */
template <int ITEMS, bool L2, int CAP>
__device__ __forceinline__ void sort_load_count_few_n(unsigned long long (&key)[CAP], const unsigned long long* src,
                                                      uint64_t first, uint32_t shift, uint32_t bits, uint32_t* slot_row,
                                                      uint32_t lane, int items) {
  if (bits == 1) sort_load_count_few<ITEMS, 1, L2>(key, src, first, shift, slot_row, lane, items);
  else sort_load_count_few<ITEMS, 2, L2>(key, src, first, shift, slot_row, lane, items);
}
template <int ITEMS, int CAP>
__device__ __forceinline__ void sort_count_few_n(const unsigned long long (&key)[CAP], uint32_t shift, uint32_t bits, uint32_t* slot_row,
                                                 uint32_t lane, int items) {
  if (bits == 1) sort_count_few<ITEMS, 1>(key, shift, slot_row, lane, items);
  else sort_count_few<ITEMS, 2>(key, shift, slot_row, lane, items);
}
template <int ITEMS, int CAP>
__device__ __forceinline__ void sort_rank_drop_few_n(const unsigned long long (&key)[CAP], uint32_t shift, uint32_t bits,
                                                     const uint32_t* slot_row, unsigned long long* keys, uint32_t lane, int items) {
  if (bits == 1) sort_rank_drop_few<ITEMS, CAP, 1>(key, shift, slot_row, keys, lane, items);
  else sort_rank_drop_few<ITEMS, CAP, 2>(key, shift, slot_row, keys, lane, items);
}

/* CTX: the pass stays inside every ctx's range of the array (requests grouped by ctx, contexts of
 * more than a tile): tiles are cut at ctx boundaries (tile_first[c] = first tile of ctx c), the
 * digit counts are per ctx, a digit's range starts at the ctx's first position, and the look-back
 * stops at the ctx's first tile -- so the ctx bits of the key need no pass at all. */
struct CtxTiles {
  const uint32_t* ctx_start;     /* [n_ctx + 1] */
  const uint32_t* tile_first;    /* [n_ctx + 1] */
  const uint32_t* hist;          /* [n_ctx][kMaxPasses][kBins] */
  uint32_t n_ctx;
};

/* PERSIST: the block takes tile after tile, and the elements may have been written by other blocks
 * of the same kernel (they are read from L2).  False: given up, a bounded wait ran out. */
template <bool PERSIST, bool CTX, bool SMALL, bool REQ = false>
__device__ __forceinline__ bool sort_tiles(SortSmem& S, uint32_t pass, PlanHeader* hdr, unsigned long long* __restrict__ buf_a,
            unsigned long long* __restrict__ buf_b, const uint32_t* __restrict__ hist,
            uint32_t* __restrict__ lookback, uint32_t* __restrict__ lookback_next, uint32_t n,
            uint32_t ibits, uint32_t stall, const CtxTiles& ct, uint32_t geometry, const RequestPass& rp = RequestPass{}) {
  constexpr int WARPS = kSortThreads / 32;
  constexpr int kLo = SMALL ? kSmallLo : REQ ? kItemsReq : kItemsLo, kHi = SMALL ? kSmallHi : REQ ? kItemsReq : kItemsHi;     /* at most so many rounds per warp */
  const int items_lo = SMALL ? (int)(geometry & 255u) : kLo, items_hi = SMALL ? (int)(geometry >> 8) : kHi;
  const uint32_t tile_size = 256u * (uint32_t)(items_lo + items_hi);
  static_assert(kLoWarps * 32 == kBins, "one look-back thread per digit");
  const unsigned long long* src = (pass & 1) ? buf_b : buf_a;
  unsigned long long* dst = (pass & 1) ? buf_a : buf_b;
  hist += pass * kBins;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lanebit = 1u << lane;
  const uint32_t n_tiles = (uint32_t)(((uint64_t)n + tile_size - 1) / tile_size);
  for (;;) {
  if (tid == 0) {
    const uint32_t given_up = PERSIST ? 0u : __ldcg(&hdr->aborted);     /* (see gave_up; in flight beside the ticket) */
    uint32_t t = atomicAdd(&hdr->ticket[pass], 1u);
    if (given_up) t = 0xffffffffu;                       /* behind all tiles */
    S.tile = t;
    S.abort = 0;
    if (CTX) {                                           /* the ctx of the tile: last c with tile_first[c] <= t */
      uint32_t lo = 0, hi = ct.n_ctx;
      while (hi - lo > 1) {
        const uint32_t mid = lo + (hi - lo) / 2;
        if (ct.tile_first[mid] <= t) lo = mid; else hi = mid;
      }
      S.ctx = t < ct.tile_first[ct.n_ctx] ? lo : 0xffffffffu;     /* the grid may hold more blocks than there are tiles */
      S.lo_tile = ct.tile_first[lo];
      S.base = ct.ctx_start[lo] + (t - ct.tile_first[lo]) * (uint32_t)kSortTile;
      S.limit = ct.ctx_start[lo + 1];
      S.first = ct.ctx_start[lo];
      /* (tiles of one ctx after the other: about that far on, from a 16-byte boundary) */
      if (!PERSIST) l2_ahead(src, S.base & ~1u, (uint64_t)kSortAhead * kSortTile, kSortTile, n);
    }
  }
  for (uint32_t i = tid; i < WARPS * kBins; i += kSortThreads) {
    (&S.slot[0][0])[i] = 0;
    (&S.match[0][0])[i] = 0;
  }
  uint32_t gh = (!CTX && tid < kBins) ? hist[tid] : 0; /* count of digit tid in the whole array (in the ctx), needed in step 2 */
  __syncthreads();
  const uint32_t tile = S.tile;
  if (!CTX && tile >= n_tiles) return true;
  if (CTX && S.ctx == 0xffffffffu) return true;
  if (CTX && tid < kBins) gh = ct.hist[((size_t)S.ctx * kMaxPasses + pass) * kBins + tid];
  const uint64_t base = CTX ? (uint64_t)S.base : (uint64_t)tile * tile_size;
  if (REQ && !PERSIST && tid == 0)
    l2_ahead(reinterpret_cast<const unsigned long long*>(rp.req), 2 * base, 2ull * kSortAhead * tile_size, 2 * tile_size, 2ull * n);
  if (!REQ && !PERSIST && !CTX && tid == 0) l2_ahead(src, base, (uint64_t)kSortAhead * tile_size, tile_size, n);
  const uint32_t limit = CTX ? S.limit : n;            /* end of the range the tile belongs to */
  const int64_t lo_tile = CTX ? (int64_t)S.lo_tile : 0;
  const uint32_t shift = ibits + hdr->pshift + 8 * pass;

  /* 1. load and count.  The warps that will do the look-back own fewer
   * elements than the others, so that both groups finish at about the same
   * time and the look-back has registers for a wide batch. */
  unsigned long long key[kHi];
  const bool lo_warp = warp < kLoWarps;
  const uint32_t wfirst = lo_warp ? warp * (32 * items_lo) : kLoWarps * 32 * items_lo + (warp - kLoWarps) * (32 * items_hi);
  /* a digit of one or two bits on a full tile: counted and ranked by ballots */
  const uint32_t dig_bits = min(8u, hdr->keybits - 8 * pass);
  /* inside a ctx the bits above the key (the ctx's part of the queue id) are the same everywhere
   * and take no part in the digit */
  const uint32_t dig_mask = CTX ? (1u << dig_bits) - 1 : 255u;
  const bool few = dig_bits <= 2 && base + tile_size <= (uint64_t)limit;
  if constexpr (REQ) {
    const uint32_t dbits = hdr->dbits;
    const bool plain = dbits < 32 && hdr->keybits + hdr->pshift <= 32;
    if (lo_warp) sort_load_requests<kLo>(key, rp, base + wfirst, limit, dbits, ibits, lane, items_lo, plain);
    else sort_load_requests<kHi>(key, rp, base + wfirst, limit, dbits, ibits, lane, items_hi, plain);
    if (few) {
      if (lo_warp) sort_count_few_n<kLo>(key, shift, dig_bits, S.slot[warp], lane, items_lo);
      else sort_count_few_n<kHi>(key, shift, dig_bits, S.slot[warp], lane, items_hi);
    } else if (lo_warp) sort_count<kLo>(key, shift, S.slot[warp], dig_mask, items_lo);
    else sort_count<kHi>(key, shift, S.slot[warp], dig_mask, items_hi);
  } else if (few) {
    if (lo_warp) sort_load_count_few_n<kLo, PERSIST>(key, src, base + wfirst, shift, dig_bits, S.slot[warp], lane, items_lo);
    else sort_load_count_few_n<kHi, PERSIST>(key, src, base + wfirst, shift, dig_bits, S.slot[warp], lane, items_hi);
  } else if (lo_warp) sort_load_count<kLo, PERSIST>(key, src, base + wfirst, limit, shift, S.slot[warp], lane, dig_mask, items_lo);
  else sort_load_count<kHi, PERSIST>(key, src, base + wfirst, limit, shift, S.slot[warp], lane, dig_mask, items_hi);
  __syncthreads();

  /* 2. thread d owns digit d */
  uint32_t cnt = 0, x = 0, g = 0;
  if (tid < kBins) {
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
      const uint32_t t = S.slot[w][tid];
      S.slot[w][tid] = cnt;                            /* exclusive over the warps */
      cnt += t;
    }
    x = cnt;
    g = gh;
    for (int o = 1; o < 32; o <<= 1) {                 /* scans over the 256 digits */
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      const uint32_t z = __shfl_up_sync(0xffffffffu, g, o);
      if (lane >= (uint32_t)o) { x += y; g += z; }
    }
    if (lane == 31) { S.scan[0][warp] = x; S.scan[1][warp] = g; }
    /* the tile's count is all that later tiles need from this one for now */
    if (!(stall && tile == 0)) st_relaxed(lookback + (size_t)tile * kBins + tid, cnt | kLbAgg);
    lookback_next[(size_t)tile * kBins + tid] = 0;     /* the array of the pass after this one */
    if (SMALL && (tile % kLookGroup) == 0) lookback_next[((size_t)n_tiles + tile / kLookGroup) * kBins + tid] = 0;
  }
  __syncthreads();
  uint32_t dstart = 0, gstart = 0;
  if (tid < kBins) {
    uint32_t wx = 0, wg = 0;
#pragma unroll
    for (int w = 0; w < kBins / 32; ++w)
      if (w < (int)warp) { wx += S.scan[0][w]; wg += S.scan[1][w]; }
    dstart = wx + x - cnt;                             /* first tile-local slot of digit tid  */
    gstart = wg + g - gh + (CTX ? S.first : 0u);       /* first global position of digit tid  */
    S.dstart[tid] = dstart;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) S.slot[w][tid] += dstart;
  }
  __syncthreads();

  /* 3. look-back by the lower part of the block; the other warps go on.  When all tiles
   * start together (SMALL) no running sum is there to be found, and the walk back over single tiles took
   * a round trip for every eight of them.  There the tiles form groups of kLookGroup: a tile adds up the
   * counts of its own group's earlier tiles, the group's last tile publishes the group's, and the walk
   * back goes over groups.  (At 2,048 wide tiles groups make it slower, 554 -> 573 us for a plan of
   * 2^24: there a running sum is mostly one round trip away.) */
  if (tid < kBins) {
    uint32_t excl = 0, spins = 0;
    const uint32_t* lb = lookback;                       /* rows to walk back over, from row t down to row lowest */
    uint32_t* own = lookback + (size_t)tile * kBins + tid;
    int64_t t = (int64_t)tile - 1, lowest = lo_tile;
    bool publish = true;
    uint32_t mine = cnt;
    if (SMALL) {
      const uint32_t in_group = tile % kLookGroup;
      uint32_t missing = in_group;                       /* earlier tiles of the group whose counts are still to come */
      while (missing) {
        uint32_t v[kLookGroup - 1];
#pragma unroll
        for (int k = 0; k < kLookGroup - 1; ++k) v[k] = k < (int)missing ? ld_relaxed(lb + (size_t)(tile - in_group + k) * kBins + tid) : 0u;
        bool all = true;
#pragma unroll
        for (int k = kLookGroup - 2; k >= 0; --k) {      /* from the latest down: the row that is not there yet is usually a late one */
          if (k < (int)missing && all) {
            if (v[k] >> 30) { excl += v[k] & kLbMask; missing = (uint32_t)k; }
            else all = false;
          }
        }
        if (missing) {
          if (++spins > kSpinLimit) { S.abort = 1; break; }
          __nanosleep(40);
        }
      }
      mine = excl + cnt;                                 /* the group up to this tile */
      publish = in_group == kLookGroup - 1;
      lb = lookback + (size_t)n_tiles * kBins;
      own = lookback + ((size_t)n_tiles + tile / kLookGroup) * kBins + tid;
      t = (int64_t)(tile / kLookGroup) - 1;
      lowest = 0;
      if (publish && !S.abort) st_relaxed(own, mine | kLbAgg);
    }
    bool done = t < lowest;
    while (!done) {
      uint32_t v[kLookBatch];
#pragma unroll
      for (int k = 0; k < kLookBatch; ++k)
        v[k] = (t - k >= lowest) ? ld_relaxed(lb + (size_t)(t - k) * kBins + tid) : +kLbIncl;   /* before the first row: nothing */
      int used = 0;
#pragma unroll
      for (int k = 0; k < kLookBatch; ++k) {
        if (!done && used == k && (v[k] >> 30) != 0) {
          excl += v[k] & kLbMask;
          used = k + 1;
          if (v[k] & kLbIncl) done = true;
        }
      }
      t -= used;
      if (!done && used < kLookBatch) {                /* met a row that has not been published yet */
        if (++spins > kSpinLimit) { S.abort = 1; break; }
        __nanosleep(40);
      }
    }
    if (publish && !S.abort && !(stall && tile == 0)) st_relaxed(own, ((excl + cnt) & kLbMask) | kLbIncl);
    S.gofs[tid] = gstart + excl - dstart;
  }

  /* 4. rank and drop into the tile buffer */
  if (few) {
    if (lo_warp) sort_rank_drop_few_n<kLo, kHi>(key, shift, dig_bits, S.slot[warp], S.keys, lane, items_lo);
    else sort_rank_drop_few_n<kHi, kHi>(key, shift, dig_bits, S.slot[warp], S.keys, lane, items_hi);
  } else if (lo_warp) sort_rank_drop<kLo, kHi>(key, shift, S.slot[warp], S.match[warp], S.keys, lanebit, items_lo, dig_mask);
  else sort_rank_drop<kHi, kHi>(key, shift, S.slot[warp], S.match[warp], S.keys, lanebit, items_hi, dig_mask);
  __syncthreads();
  if (S.abort) {
    if (tid == 0) set_aborted(hdr);
    return false;
  }

  /* 5. write out */
  const uint32_t nvalid = (uint32_t)min((uint64_t)tile_size, (uint64_t)limit - base);
  if (REQ && rp.rounds) {
    const uint32_t dbits = hdr->dbits, imask = (1u << ibits) - 1;
    const unsigned long long dmask = (1ull << dbits) - 1;
    const bool lookup = hdr->lookup != 0;
    uint32_t* const out = reinterpret_cast<uint32_t*>(dst);
    longlong2* con = reinterpret_cast<longlong2*>(&S.match[0][0]);   /* per queue, which is the digit: what its deadlines are compared with, 1 / d */
    bool easy = dbits <= 29 && !lookup;                /* 32-bit arithmetic will do */
    for (uint32_t q = tid; q < rp.n_ctx * rp.S; q += kSortThreads) {
      const PardSegConst& K = rp.ktab[q];
      const bool none = K.narrow & kSegNoStage;
      const long long from = none ? 1ll << 62 : (lookup ? K.A : K.A_rel) - (rp.nexus ? K.lsub : 0ll);   /* Nexus: the current module only, base + d */
      if (none && (q + 1 < kBins ? S.dstart[q + 1] : nvalid) > S.dstart[q]) set_status(hdr, PARD_EDATA);   /* (the tile has requests of the queue) */
      con[q] = make_longlong2(from, (long long)K.d_magic);
      easy = easy && (none || (K.d_magic != 0 && from > -(1ll << 30)));
    }
    if (__syncthreads_and(easy)) {
#pragma unroll 4
      for (uint32_t pos = tid; pos < nvalid; pos += kSortThreads) {
        const unsigned long long k = S.keys[pos];
        const uint32_t d = (uint32_t)(k >> shift) & 255u, at = S.gofs[d] + pos;
        const longlong2 c = con[d];
        const int32_t X = (int32_t)(__funnelshift_r((uint32_t)k, (uint32_t)(k >> 32), ibits) & (uint32_t)dmask) - (int32_t)min(c.x, 1ll << 30);
        out[at] = (uint32_t)k & imask;
        rp.rounds[at] = X < 0 ? 0u : div_magic32((uint32_t)X, (unsigned long long)c.y) + 1;   /* < 2^30: d >= 2 */
      }
    } else {
      for (uint32_t pos = tid; pos < nvalid; pos += kSortThreads) {
        const unsigned long long k = S.keys[pos];
        const uint32_t d = (uint32_t)(k >> shift) & 255u, at = S.gofs[d] + pos, idx = (uint32_t)k & imask;
        const longlong2 c = con[d];
        const long long X = (long long)(lookup ? __ldg(reinterpret_cast<const unsigned long long*>(&rp.req[idx])) : (k >> ibits) & dmask) - c.x;
        out[at] = idx;
        rp.rounds[at] = rounds_fit(X, (unsigned long long)c.y, (unsigned long long)rp.ktab[d].d);
      }
    }
    return true;
  }
#pragma unroll 4
  for (uint32_t pos = tid; pos < nvalid; pos += kSortThreads) {
    const unsigned long long k = S.keys[pos];
    const uint32_t d = (uint32_t)(k >> shift) & dig_mask;
    dst[S.gofs[d] + pos] = k;
  }
  if (!PERSIST) return true;
  __syncthreads();                                     /* the tile buffer and the tables are reused */
  if (tid == 0 && !(stall && tile == 0)) ++S.done;
  }
}

/* (a call: inlined into the loop over the passes the wide tiles would spill more) */
template <bool CTX>
__device__ __noinline__ bool sort_tiles_resident(SortSmem& S, uint32_t pass, PlanHeader* hdr, unsigned long long* buf_a,
            unsigned long long* buf_b, const uint32_t* hist, uint32_t* lookback, uint32_t* lookback_next, uint32_t n,
            uint32_t ibits, uint32_t stall, const CtxTiles& ct) {
  return sort_tiles<true, CTX, false>(S, pass, hdr, buf_a, buf_b, hist, lookback, lookback_next, n, ibits, stall, ct, 0u);
}

/* One pass, one tile per block. */
template <bool CTX>
__global__ void __launch_bounds__(kSortThreads, 2)
k_sort_pass(uint32_t pass, PlanHeader* hdr, unsigned long long* __restrict__ buf_a,
            unsigned long long* __restrict__ buf_b, const uint32_t* __restrict__ hist,
            uint32_t* __restrict__ lookback, uint32_t* __restrict__ lookback_next, uint32_t n,
            uint32_t ibits, uint32_t stall, uint32_t local_candidate, const CtxTiles ct, const __grid_constant__ WinCountArgs wc) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (wc.on && blockIdx.x == gridDim.x - 1) { win_from_counts(hdr, wc); return; }
  if ((CTX && hdr->direct) || pass >= hdr->npass || sort_is_local(hdr, local_candidate)) return;
  sort_tiles<false, CTX, false>(*reinterpret_cast<SortSmem*>(smem_raw), pass, hdr, buf_a, buf_b, hist, lookback, lookback_next, n, ibits,
                                stall, ct, 0u);
}

/* The one pass of a call in arrival order with up to 256 queues, from the requests: their elements need not be written
 * and read back first, and for the rules that compare the deadline alone (rp.rounds) the pass leaves what the walk and
 * the outputs want, the index and the rounds, 8 bytes per request.  2^24 requests of 16 queues under the window scan:
 * k_pack, the pass and k_policy_terms took 57 + 81 + 57 us, this takes 122 (403 MB: 62 by bytes), the call 402 -> 309.
 * Bound by instructions (half of the issue slots, 140 per 32 requests) and by the pass's shared-memory atomics.
 * Requests are loaded four at a time, ahead of any use: one by one 201 us. */
template <bool SMALL>
__global__ void __launch_bounds__(kSortThreads, 2)
k_sort_requests(PlanHeader* hdr, unsigned long long* __restrict__ buf_a, unsigned long long* __restrict__ buf_b, const uint32_t* __restrict__ hist,
                uint32_t* __restrict__ lookback, uint32_t* __restrict__ lookback_next, uint32_t n, uint32_t ibits, uint32_t stall,
                uint32_t geometry, const __grid_constant__ RequestPass rp) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  sort_tiles<false, false, SMALL, true>(*reinterpret_cast<SortSmem*>(smem_raw), 0u, hdr, buf_a, buf_b, hist, lookback, lookback_next, n, ibits,
                                        stall, CtxTiles{}, geometry, rp);
}

/* All passes from `pass` on, by one grid.  How many passes a key needs is only known on the device, and a
 * pass that finds nothing to do still costs a launch: 2.5 to 4.5 us each, up to seven per call.  A block
 * takes tiles by ticket until the pass has none left, hands in how many it has finished, and begins the
 * next pass when all tiles have been handed in.  It never waits for a block
 * that has not been placed: however few of the grid's blocks run at a time -- other streams may hold the
 * multiprocessors, another call's grid of this kind among them -- those that run finish the pass.  (Every
 * tile handed in by itself: 214.0 against 211.2 us for 2.5 M requests of 512 contexts; a block's tiles
 * together: 212.4, as when the grid's blocks were counted.)
 * At 2^24 elements such a grid takes 9 us more per pass than one block per tile (the blocks' loads
 * no longer start under the write-out of others), so the passes that large calls usually need keep
 * launches of their own.  Calls of one or two rounds of small tiles (SMALL) do all passes here,
 * with tiles sized so that every block takes the same number of them. */
template <bool CTX, bool SMALL>
__global__ void __launch_bounds__(kSortThreads, 2)
k_sort_rest(uint32_t pass, PlanHeader* hdr, unsigned long long* buf_a, unsigned long long* buf_b,
            const uint32_t* __restrict__ hist, uint32_t* lookback, size_t lb_words, uint32_t n,
            uint32_t ibits, uint32_t stall, uint32_t local_candidate, const CtxTiles ct, const __grid_constant__ WinCountArgs wc,
            uint32_t geometry) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (wc.on && blockIdx.x == gridDim.x - 1) { win_from_counts(hdr, wc); return; }
  if ((CTX && hdr->direct) || sort_is_local(hdr, local_candidate) || gave_up(hdr)) return;
  const uint32_t npass = hdr->npass;
  const uint32_t tile_size = SMALL ? 256u * ((geometry & 255u) + (geometry >> 8)) : (uint32_t)kSortTile;
  const uint32_t tiles = CTX ? ct.tile_first[ct.n_ctx] : (uint32_t)(((uint64_t)n + tile_size - 1) / tile_size);
  for (uint32_t p = pass; p < npass; ++p) {
    SortSmem& S = *reinterpret_cast<SortSmem*>(smem_raw);
    if (threadIdx.x == 0) S.done = 0;
    uint32_t* now = lookback + (p & 1) * lb_words;
    uint32_t* next = lookback + ((p + 1) & 1) * lb_words;
    bool go;
    if constexpr (SMALL) go = sort_tiles<true, CTX, true>(S, p, hdr, buf_a, buf_b, hist, now, next, n, ibits, p == 0 ? stall : 0u, ct, geometry);
    else go = sort_tiles_resident<CTX>(S, p, hdr, buf_a, buf_b, hist, now, next, n, ibits, p == 0 ? stall : 0u, ct);
    if (!go) return;
    if (p + 1 < npass && !finish_pieces(hdr, &hdr->sort_bar[p], S.done, tiles)) return;
  }
}


__global__ void __launch_bounds__(1024)
k_tile_table(const uint32_t* __restrict__ ctx_start, uint32_t n_ctx, uint32_t* __restrict__ tile_first, const PlanHeader* hdr) {
  pdl_wait();
  if (!hdr->direct) tile_table(ctx_start, n_ctx, tile_first);
}

/* k_pack for passes that stay inside the contexts: a block packs one tile (all of one ctx) and
 * adds its digit counts to the ctx's.  The digits cover the stage and deadline bits only; a
 * request of another ctx inside the tile breaks the caller's promise. */
__global__ void __launch_bounds__(256)
k_pack_ctx(const uint4* __restrict__ req, uint32_t S, const unsigned long long* __restrict__ ctx_dmin_inv,
           const unsigned long long* __restrict__ ctx_dmax, const uint8_t* __restrict__ priority, uint32_t ibits,
           PlanHeader* __restrict__ hdr, unsigned long long* __restrict__ dst, uint32_t* __restrict__ hist_ctx,
           const CtxTiles ct) {
  pdl_wait();
  __shared__ uint32_t s_hist[kMaxPasses * kBins];
  __shared__ uint32_t s_c, s_base, s_limit, s_skip;
  const uint32_t tile = blockIdx.x;
  if (threadIdx.x == 0) {
    const bool unsorted = ld_relaxed(&hdr->unsorted) != 0;       /* found out of ctx order, by k_ctx_ranges or a block of this kernel (see gave_up) */
    if (unsorted && tile == 0) { hdr->aborted = 1; set_status(hdr, PARD_EDATA); }
    s_skip = unsorted || hdr->direct || hdr->wide || ld_relaxed(&hdr->aborted) ? 1u : 0u;
  }
  __syncthreads();
  if (s_skip) return;
  if (threadIdx.x == 0) {
    uint32_t lo = 0, hi = ct.n_ctx;
    while (hi - lo > 1) {
      const uint32_t mid = lo + (hi - lo) / 2;
      if (ct.tile_first[mid] <= tile) lo = mid; else hi = mid;
    }
    s_c = tile < ct.tile_first[ct.n_ctx] ? lo : 0xffffffffu;
    s_base = ct.ctx_start[lo] + (tile - ct.tile_first[lo]) * (uint32_t)kSortTile;
    s_limit = ct.ctx_start[lo + 1];
  }
  const uint32_t npass = hdr->npass, dbits = hdr->dbits, pshift = hdr->pshift;
  for (uint32_t i = threadIdx.x; i < npass * kBins; i += blockDim.x) s_hist[i] = 0;
  __syncthreads();
  const uint32_t c = s_c;
  if (c == 0xffffffffu) return;
  const uint32_t end = min(s_limit, s_base + (uint32_t)kSortTile);
  const unsigned long long dmask = dbits >= 64 ? ~0ull : ((1ull << dbits) - 1);
  const unsigned long long cmin = ~ctx_dmin_inv[c], cmax = ctx_dmax[c];
  const unsigned long long keymask = hdr->keybits >= 64 ? ~0ull : ((1ull << hdr->keybits) - 1);
  bool foreign = false;
  if (!hdr->bad_input && !priority && hdr->keybits + pshift <= 32 && dbits <= 29) {
    /* the usual call, as in k_pack: single words, and four requests in flight (2^24 requests in 256 contexts: 76 -> 60 us) */
    const unsigned long long part = ((unsigned long long)(c * S) << dbits) << ibits;     /* the ctx's part of every element */
    const uint32_t up = 1u << ibits, low = (uint32_t)cmin;
    constexpr uint32_t kUn = 4;
    for (uint32_t j0 = s_base + threadIdx.x; j0 < end; j0 += kUn * blockDim.x) {
      uint4 rr[kUn];
#pragma unroll
      for (uint32_t u = 0; u < kUn; ++u) {
        const uint32_t j = j0 + u * blockDim.x;
        if (j < end) rr[u] = __ldg(&req[j]);
      }
#pragma unroll
      for (uint32_t u = 0; u < kUn; ++u) {
        const uint32_t j = j0 + u * blockDim.x;
        if (j >= end) break;
        const uint4 r = rr[u];
        foreign = foreign || r.z != c;
        const uint32_t key = ((r.w & 0xffffu) << dbits) | (r.z == c ? r.x - low : 0u);
        dst[j] = part + (unsigned long long)key * up + j;
        count_digits(s_hist, key >> pshift, npass);
      }
    }
  } else
  for (uint32_t j = s_base + threadIdx.x; j < end; j += blockDim.x) {
    const uint4 r = __ldg(&req[j]);
    const unsigned long long D = ((unsigned long long)r.y << 32) | r.x;
    const uint32_t stage = r.w & 0xffffu;
    unsigned long long key = 0;
    if (r.z != c) foreign = true;
    else if (stage < S) {
      const uint32_t seg = c * S + stage;
      const bool high_first = priority && __ldg(&priority[seg]) != 0;
      key = ((unsigned long long)seg << dbits) | ((high_first ? cmax - D : D - cmin) & dmask);
    }
    dst[j] = (key << ibits) | j;                         /* a flagged request keeps its index alone, as in k_pack */
    key = (key >> pshift) & keymask;                     /* the ctx's part of the queue id takes no part in the digits */
    uint32_t* hp = s_hist;
    for (uint32_t p = 0; p < npass; ++p, hp += kBins, key >>= 8) atomicAdd(hp + ((uint32_t)key & 255u), 1u);
  }
  if (__syncthreads_or(foreign)) {
    if (threadIdx.x == 0) { hdr->unsorted = 1; hdr->aborted = 1; set_status(hdr, PARD_EDATA); }
    return;
  }
  uint32_t* h = hist_ctx + (size_t)c * kMaxPasses * kBins;
  for (uint32_t i = threadIdx.x; i < npass * kBins; i += blockDim.x)
    if (s_hist[i]) atomicAdd(&h[i], s_hist[i]);
}

/* ------------------------------------------------------------------------ */
/* calls whose requests come grouped by ctx, every ctx within one tile       */
/* ------------------------------------------------------------------------ */
/* Batched decision epochs and small what-if instances arrive as one array with the requests of
 * a ctx side by side.  If no ctx holds more than a tile, nothing has to move between ctxs: a
 * block sorts "its" ctx in shared memory -- radix passes over the stage and deadline bits only,
 * no global scatter, no look-back -- and the global passes do not run.  `candidate` is the
 * host's part of the test (between kSortTile / 4 and kSortTile requests per ctx on average);
 * the device adds what only it can see.  A call with a single ctx of at most kSortTile requests
 * needs no test at all: its one block is certain, and neither the range search nor the global
 * passes are launched -- the case of one module's queue planned every few milliseconds. */
/* Where every ctx would begin if the requests came in ascending ctx order, one warp per ctx.  Whether
 * they do is settled by k_sort_local (k_pack_ctx), where every block checks that its range holds
 * requests of its ctx only. */
__global__ void __launch_bounds__(256)
k_ctx_ranges(const uint4* __restrict__ req, uint32_t n, uint32_t n_ctx, uint32_t* __restrict__ ctx_start,
             PlanHeader* hdr) {
  pdl_wait();
  const uint32_t c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (c <= n_ctx) ctx_range_search(req, n, n_ctx, c, ctx_start, hdr, (uint32_t)kSortTile);   /* whole warps stay together */
}

/* One block per ctx: the ctx's requests, read from the caller's array, turned into the sort
 * elements k_pack would have made, sorted in shared memory and written to the buffer the global
 * passes would have ended in (k_pack does not run then).  Inside a ctx only the stage and the
 * deadline offset differ; the ctx's own contribution to the segment field is left out of the
 * element while it is sorted and added on the way out, so that the passes see a plain bit field. */
__global__ void __launch_bounds__(kSortThreads, 2)
k_sort_local(PlanHeader* __restrict__ hdr, uint32_t candidate, const uint4* __restrict__ req,
             const unsigned long long* __restrict__ ctx_dmin_inv, const unsigned long long* __restrict__ ctx_dmax,
             const uint8_t* __restrict__ priority, unsigned long long* __restrict__ buf_a,
             unsigned long long* __restrict__ buf_b, const uint32_t* __restrict__ ctx_start, uint32_t n,
             uint32_t S, uint32_t stage_bits, uint32_t ibits) {
  pdl_wait();
  constexpr int WARPS = kSortThreads / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SortSmem& Sm = *reinterpret_cast<SortSmem*>(smem_raw);
  if (!__syncthreads_or(threadIdx.x == 0 && sort_is_local(hdr, candidate))) return;     /* (see gave_up: `unsorted` is set below) */
  const uint32_t c = blockIdx.x;
  const uint32_t first = ctx_start ? ctx_start[c] : 0u;              /* no table: the call has one ctx */
  const uint32_t cnt = ctx_start ? ctx_start[c + 1] - first : n;
  if (cnt == 0) return;
  unsigned long long* dst = (hdr->npass & 1) ? buf_b : buf_a;
  const uint32_t dbits = hdr->dbits;
  const unsigned long long dmask = dbits >= 64 ? ~0ull : ((1ull << dbits) - 1);
  const unsigned long long dmin = ~ctx_dmin_inv[c], dmax = ctx_dmax[c];
  const uint32_t pshift = hdr->pshift;
  const uint32_t local_bits = dbits - pshift + stage_bits;
  const uint32_t passes = (local_bits + 7) / 8;
  const unsigned long long ctx_part = (unsigned long long)c * S << (dbits + ibits);   /* < 2^64: the key fits */
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lanebit = 1u << lane;
  constexpr int kItems = kSortTile / kSortThreads;       /* every warp owns the same share here: nothing else to do meanwhile */
  static_assert(kItems * kSortThreads == kSortTile, "the tile divides evenly");
  const uint32_t wfirst = warp * (32 * kItems);

  /* the ctx's requests, straight from the caller's array, turned into sort elements without the
   * ctx's share of the segment field (k_pack's element minus ctx_part); a request of another
   * ctx inside the range means the requests are not grouped after all */
  unsigned long long key[kItems];
  bool foreign = false;
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t pos = wfirst + i * 32 + lane;
    key[i] = ~0ull;                                       /* padding sorts last */
    if (pos < cnt) {
      const uint32_t j = first + pos;
      const uint4 r = __ldg(&req[j]);
      const unsigned long long D = ((unsigned long long)r.y << 32) | r.x;
      const uint32_t stage = r.w & 0xffffu;
      foreign |= ctx_start != nullptr && r.z != c;       /* with one ctx there is no other: an input error */
      if (r.z == c && stage < S) {
        const bool high_first = priority && __ldg(&priority[c * S + stage]) != 0;
        const unsigned long long off = (high_first ? dmax - D : D - dmin) & dmask;
        key[i] = ((((unsigned long long)stage << dbits) | off) << ibits) | j;
      } else {
        key[i] = (unsigned long long)j - ctx_part;        /* flagged by the prepass; k_pack's element is j */
      }
    }
  }
  if (__syncthreads_or(foreign)) {                        /* the global passes take over (k_pack, then k_sort_pass) */
    if (tid == 0) hdr->unsorted = 1;
    return;
  }
  for (uint32_t i = tid; i < WARPS * kBins; i += kSortThreads) (&Sm.match[0][0])[i] = 0;   /* ranking leaves it clear */
  for (uint32_t p = 0; p < passes; ++p) {
    const uint32_t shift = ibits + pshift + 8 * p;
    for (uint32_t i = tid; i < WARPS * kBins; i += kSortThreads) (&Sm.slot[0][0])[i] = 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kItems; ++i) atomicAdd(&Sm.slot[warp][(uint32_t)(key[i] >> shift) & 255u], 1u);
    __syncthreads();
    uint32_t count = 0, x = 0;
    if (tid < kBins) {                                  /* thread d owns digit d */
#pragma unroll
      for (int w = 0; w < WARPS; ++w) {
        const uint32_t t = Sm.slot[w][tid];
        Sm.slot[w][tid] = count;                        /* exclusive over the warps */
        count += t;
      }
      x = count;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x += y;
      }
      if (lane == 31) Sm.scan[0][warp] = x;
    }
    __syncthreads();
    if (tid < kBins) {
      uint32_t wx = 0;
#pragma unroll
      for (int w = 0; w < kBins / 32; ++w)
        if (w < (int)warp) wx += Sm.scan[0][w];
      const uint32_t dstart = wx + x - count;           /* first slot of digit tid */
#pragma unroll
      for (int w = 0; w < WARPS; ++w) Sm.slot[w][tid] += dstart;
    }
    __syncthreads();
    sort_rank_drop<kItems, kItems>(key, shift, Sm.slot[warp], Sm.match[warp], Sm.keys, lanebit);
    __syncthreads();
    if (p + 1 < passes) {
#pragma unroll
      for (int i = 0; i < kItems; ++i) key[i] = Sm.keys[wfirst + i * 32 + lane];
      __syncthreads();
    }
  }
  if (passes == 0) {                                    /* nothing differs inside a ctx: index order stands */
#pragma unroll
    for (int i = 0; i < kItems; ++i) Sm.keys[wfirst + i * 32 + lane] = key[i];
    __syncthreads();
  }
  for (uint32_t pos = tid; pos < cnt; pos += kSortThreads) dst[first + pos] = Sm.keys[pos] + ctx_part;
}

/* ------------------------------------------------------------------------ */
/* decision pass over the sorted elements                                    */
/* ------------------------------------------------------------------------ */
__device__ __forceinline__ unsigned long long pack_val(SegVal a, unsigned long long state) {
  return state | ((unsigned long long)a.head << 32) | (uint32_t)a.m;
}
__device__ __forceinline__ SegVal unpack_val(unsigned long long w) {
  SegVal a;
  a.m = (int32_t)(uint32_t)w;
  a.head = (uint32_t)(w >> 32) & 1u;
  return a;
}

/* First half of the decision pass for one thread's kDecItems consecutive
 * sorted elements: decode, admission threshold u, position r inside the own
 * queue, and the thread's running segmented reduction (admitted mode: minimum
 * of u_t - t; raw mode: number of kept requests). */
struct TileCtx {
  const unsigned long long* src;
  const PardSegConst* ktab;
  const uint32_t* seg_off;
  uint32_t n, ibits, imask, kshift;
  unsigned long long dmask;
  bool narrow;               /* deadline offsets have at most 29 bits */
  PlanHeader* hdr;
};

template <bool RAW>
__device__ __forceinline__ void tile_first_half(const TileCtx& T, uint64_t base, unsigned long long (&e)[kDecItems],
                                                uint32_t (&idx)[kDecItems], uint32_t (&u)[kDecItems],
                                                uint32_t (&r)[kDecItems], int32_t (&lv)[kDecItems],
                                                uint32_t& lheadbits, SegVal& run, PardSegConst& K,
                                                uint32_t& sstart, uint32_t& seg_first, bool& one_seg) {
  static_assert(kDecItems == 8, "two 32-byte loads per thread");
  const bool full = base + kDecItems <= T.n;
  if (full) {
    load4(T.src + base, e);
    load4(T.src + base + 4, e + 4);
  } else {
#pragma unroll
    for (int i = 0; i < kDecItems; ++i) e[i] = base + i < T.n ? T.src[base + i] : 0;
  }
  seg_first = (uint32_t)(e[0] >> T.kshift);
  /* most threads see one queue only: its constants are then loaded once */
  one_seg = full && seg_first == (uint32_t)(e[kDecItems - 1] >> T.kshift);
  K = T.ktab[seg_first];
  sstart = T.seg_off[seg_first];
  uint32_t cur_seg = seg_first;
  lheadbits = 0;
  run = seg_identity<RAW>();
  if ((K.narrow & kSegNoStage) && base < T.n) set_status(T.hdr, PARD_EDATA);   /* queue of a stage the pipeline lacks */
  if (one_seg && T.narrow && (K.narrow & (kSegNarrow | kSegNoStage)) == kSegNarrow) {
    /* one queue, and every quantity fits 32 bits: the common case */
    const uint32_t r0 = (uint32_t)base - sstart;
    const bool high_first = K.narrow & kSegHighFirst;
    const int32_t A = narrow_A(K);
#pragma unroll
    for (int i = 0; i < kDecItems; ++i) {
      const uint32_t lo = (uint32_t)e[i], hi = (uint32_t)(e[i] >> 32);
      idx[i] = lo & T.imask;
      const uint32_t off = __funnelshift_r(lo, hi, T.ibits) & (uint32_t)T.dmask;
      const int32_t X = high_first ? A - (int32_t)off : (int32_t)off - A;
      const unsigned long long uu = (unsigned long long)(div_magic32((uint32_t)X, K.d_magic) + 1u) * K.cap;
      u[i] = X < 0 ? 0u : (uu > kUClamp ? kUClamp : (uint32_t)uu);
      r[i] = r0 + i;
      if (r[i] == 0) { run = seg_identity<RAW>(); run.head = 1; }
      lv[i] = run.m;
      lheadbits |= run.head << i;
      if (RAW) run.m += r[i] < u[i] ? 1 : 0;
      else run.m = min(run.m, (int32_t)u[i] - (int32_t)r[i]);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < kDecItems; ++i) {
    const uint64_t j = base + i;
    if (j < T.n) {
      idx[i] = (uint32_t)e[i] & T.imask;
      const unsigned long long off = (e[i] >> T.ibits) & T.dmask;
      if (!one_seg) {
        const uint32_t sg = (uint32_t)(e[i] >> T.kshift);
        if (sg != cur_seg) {
          cur_seg = sg;
          K = T.ktab[sg];
          sstart = T.seg_off[sg];
          if (K.narrow & kSegNoStage) set_status(T.hdr, PARD_EDATA);
        }
      }
      r[i] = (uint32_t)j - sstart;
      u[i] = threshold_u(slack_of(off, K), K);
    } else {
      idx[i] = 0; r[i] = 0; u[i] = kUClamp;                    /* acts as a head, never read */
    }
    if (r[i] == 0) { run = seg_identity<RAW>(); run.head = 1; }
    lv[i] = run.m;
    lheadbits |= run.head << i;
    if (RAW) run.m += (r[i] < u[i] && j < T.n) ? 1 : 0;
    else run.m = min(run.m, (int32_t)u[i] - (int32_t)r[i]);
  }
}

__device__ __forceinline__ TileCtx make_tile_ctx(const PlanHeader* hdr, const unsigned long long* buf_a,
                                                 const unsigned long long* buf_b, uint32_t n, uint32_t ibits,
                                                 const PardSegConst* ktab, const uint32_t* seg_off) {
  TileCtx T;
  const uint32_t dbits = hdr->dbits;
  T.src = (hdr->npass & 1) ? buf_b : buf_a;
  T.ktab = ktab;
  T.seg_off = seg_off;
  T.n = n;
  T.ibits = ibits;
  T.imask = (1u << ibits) - 1;                                 /* ibits <= 30 */
  T.kshift = ibits + dbits;                                    /* < 64 */
  T.dmask = dbits >= 64 ? ~0ull : ((1ull << dbits) - 1);
  /* the offsets that occur, not the field they sit in (a call whose element format is fixed by
   * the host may have a wider field than its deadline spans need) */
  T.narrow = dbits <= 29 || (hdr->span_max >> 29) == 0;
  T.hdr = const_cast<PlanHeader*>(hdr);
  return T;
}

/* Exclusive segmented scan of the tile aggregates by one block, eight tiles
 * per thread and round: carry[t] is the reduction over the elements that
 * precede tile t in the queue that is open at the start of tile t. */
template <bool RAW, int THREADS>
__device__ void tile_scan_block(const unsigned long long* tile_agg, uint32_t n_tiles, int32_t* carry) {
  constexpr int PER = 8, WARPS = THREADS / 32;
  __shared__ int32_t s_wm[32];
  __shared__ uint32_t s_wh[32];
  __shared__ int32_t s_cm;
  __shared__ uint32_t s_ch;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) { s_cm = seg_identity<RAW>().m; s_ch = 0; }
  __syncthreads();
  for (uint32_t b = 0; b < n_tiles; b += THREADS * PER) {
    const uint32_t t0 = b + threadIdx.x * PER;
    SegVal v[PER];
    SegVal run = seg_identity<RAW>();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      v[k] = t0 + k < n_tiles ? unpack_val(__ldcg(&tile_agg[t0 + k])) : seg_identity<RAW>();
      run = seg_combine<RAW>(run, v[k]);
    }
    const SegVal inc = warp_scan<RAW>(run, lane);
    SegVal exc;
    exc.m = __shfl_up_sync(0xffffffffu, inc.m, 1);
    exc.head = __shfl_up_sync(0xffffffffu, inc.head, 1);
    if (lane == 0) exc = seg_identity<RAW>();
    if (lane == 31) { s_wm[warp] = inc.m; s_wh[warp] = inc.head; }
    __syncthreads();
    if (warp == 0) {                        /* scan of the warp aggregates, led by the carry */
      SegVal a = seg_identity<RAW>();
      if (lane < WARPS) { a.m = s_wm[lane]; a.head = s_wh[lane]; }
      SegVal ai = warp_scan<RAW>(a, lane);
      SegVal ae;
      ae.m = __shfl_up_sync(0xffffffffu, ai.m, 1);
      ae.head = __shfl_up_sync(0xffffffffu, ai.head, 1);
      if (lane == 0) ae = seg_identity<RAW>();
      SegVal c0; c0.m = s_cm; c0.head = s_ch;
      ae = seg_combine<RAW>(c0, ae);
      const SegVal all = seg_combine<RAW>(c0, ai);
      __syncwarp();
      s_wm[lane] = ae.m; s_wh[lane] = ae.head;
      if (lane == 31) { s_cm = all.m; s_ch = all.head; }
    }
    __syncthreads();
    SegVal pre; pre.m = s_wm[warp]; pre.head = s_wh[warp];
    pre = seg_combine<RAW>(pre, exc);
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      if (t0 + k < n_tiles) carry[t0 + k] = pre.m;
      pre = seg_combine<RAW>(pre, v[k]);
    }
    __syncthreads();
  }
}

/* Tile aggregates: the segmented reduction over each tile of kDecTile sorted
 * elements, for tiles [first, end).  Tiles are independent. */
template <bool RAW>
__device__ void tile_agg_tiles(const PlanHeader* __restrict__ hdr, const unsigned long long* __restrict__ buf_a,
                               const unsigned long long* __restrict__ buf_b, uint32_t n, uint32_t ibits,
                               const PardSegConst* __restrict__ ktab, const uint32_t* __restrict__ seg_off,
                               unsigned long long* __restrict__ tile_agg, uint32_t first, uint32_t end) {
  constexpr int WARPS = kDecThreads / 32;
  __shared__ int32_t s_wm[WARPS];
  __shared__ uint32_t s_wh[WARPS];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const TileCtx T = make_tile_ctx(hdr, buf_a, buf_b, n, ibits, ktab, seg_off);
  for (uint32_t tile = first; tile < end; ++tile) {
    const uint64_t base = (uint64_t)tile * kDecTile + (uint64_t)tid * kDecItems;
    unsigned long long e[kDecItems];
    uint32_t idx[kDecItems], u[kDecItems], r[kDecItems], lheadbits, sstart, seg_first;
    int32_t lv[kDecItems];
    SegVal run;
    PardSegConst K;
    bool one_seg;
    tile_first_half<RAW>(T, base, e, idx, u, r, lv, lheadbits, run, K, sstart, seg_first, one_seg);
    const SegVal inc = warp_scan<RAW>(run, lane);
    if (lane == 31) { s_wm[warp] = inc.m; s_wh[warp] = inc.head; }
    __syncthreads();
    if (tid == 0) {
      SegVal agg = seg_identity<RAW>();
#pragma unroll
      for (int w = 0; w < WARPS; ++w) {
        SegVal a; a.m = s_wm[w]; a.head = s_wh[w];
        agg = seg_combine<RAW>(agg, a);
      }
      tile_agg[tile] = pack_val(agg, 0);
    }
    __syncthreads();
  }
}

/* Decision pass over tiles [first, end) of kDecTile sorted elements; a thread owns kDecItems consecutive
 * elements of a tile.
 *
 * Admitted mode: c_r = min(r, r-1 + min_{t<r}(u_t - t)) by a segmented
 * exclusive prefix-min; raw mode: c_r = r, and the kept requests ahead in the
 * queue are counted by a segmented exclusive prefix-sum.  Either way the
 * number k_r of kept requests ahead in the own queue is known per request, and
 * a kept request's index goes to kept_tmp[first position of its queue + k_r]:
 * every queue's survivors end up contiguous, kept_move_jobs packs the queues. */
template <bool RAW>
__device__ void decide_tiles(const PlanHeader* __restrict__ hdr, const unsigned long long* __restrict__ buf_a,
         const unsigned long long* __restrict__ buf_b, uint32_t n, uint32_t ibits,
         const PardSegConst* __restrict__ ktab, const uint32_t* __restrict__ seg_off,
         const uint32_t* __restrict__ win_off, const int32_t* __restrict__ carry,
         uint8_t* __restrict__ out_keep, long long* __restrict__ out_est, uint32_t* __restrict__ out_perm,
         uint32_t* __restrict__ kept_tmp, uint32_t* __restrict__ seg_kept, uint32_t first, uint32_t end) {
  constexpr int WARPS = kDecThreads / 32;
  __shared__ int32_t s_wm[WARPS];
  __shared__ uint32_t s_wh[WARPS];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const TileCtx T = make_tile_ctx(hdr, buf_a, buf_b, n, ibits, ktab, seg_off);
  for (uint32_t tile = first; tile < end; ++tile) {
  const uint64_t base = (uint64_t)tile * kDecTile + (uint64_t)tid * kDecItems;
  const bool full = base + kDecItems <= n;
  const int32_t tile_carry = __ldcg(&carry[tile]);       /* written by another block of this kernel */

  unsigned long long e[kDecItems];
  uint32_t idx[kDecItems], u[kDecItems], r[kDecItems], lheadbits, sstart, seg_first;
  int32_t lv[kDecItems];     /* reduction over this thread's earlier items of the same queue */
  SegVal run;
  PardSegConst K;
  bool one_seg;
  tile_first_half<RAW>(T, base, e, idx, u, r, lv, lheadbits, run, K, sstart, seg_first, one_seg);

  /* exclusive segmented scan of the threads' aggregates: warp, block, then the tile's carry */
  const SegVal inc = warp_scan<RAW>(run, lane);
  SegVal exc;
  exc.m = __shfl_up_sync(0xffffffffu, inc.m, 1);
  exc.head = __shfl_up_sync(0xffffffffu, inc.head, 1);
  if (lane == 0) exc = seg_identity<RAW>();
  if (lane == 31) { s_wm[warp] = inc.m; s_wh[warp] = inc.head; }
  __syncthreads();
  SegVal wprefix; wprefix.m = tile_carry; wprefix.head = 0;
#pragma unroll
  for (int w = 0; w < WARPS; ++w) {
    SegVal a; a.m = s_wm[w]; a.head = s_wh[w];
    if (w < (int)warp) wprefix = seg_combine<RAW>(wprefix, a);
  }
  exc = seg_combine<RAW>(wprefix, exc);

  /* admitted position, estimate, decision */
  uint32_t keepbits = 0;
  long long est[kDecItems];
  uint32_t cur_seg = seg_first;
  uint32_t send = seg_off[seg_first + 1];
  if (!one_seg) {
    K = ktab[seg_first];
    sstart = seg_off[seg_first];
  }
  /* A queue served high budget first keeps a prefix (thresholds fall along the queue while
   * positions rise); win_off holds the length of that prefix, and the admitted position is
   * the raw one capped by it. */
  uint32_t hb_kept = (K.narrow & kSegHighFirst) ? win_off[seg_first] : 0u;
  const bool fast = one_seg && T.narrow && (K.narrow & (kSegNarrow | kSegNoStage)) == kSegNarrow;
  if (fast) {
    const bool high_first = K.narrow & kSegHighFirst;
#pragma unroll
    for (int i = 0; i < kDecItems; ++i) {
      const bool local = (lheadbits >> i) & 1u;
      const int32_t pre = local ? lv[i] : (RAW ? lv[i] + exc.m : min(lv[i], exc.m));
      uint32_t c, ahead;
      if (RAW) {
        c = r[i];
        ahead = r[i] == 0 ? 0u : (uint32_t)pre;
      } else {
        c = r[i] == 0 ? 0u : (uint32_t)min((int32_t)r[i] - 1 + pre, (int32_t)r[i]);   /* both below 2^31 */
        if (high_first) c = min(r[i], hb_kept);
        ahead = c;
      }
      const uint32_t round = K.cap_magic ? div_magic32(c, K.cap_magic) : c;
      est[i] = K.A + (long long)((unsigned long long)round * (uint32_t)K.d);
      const uint32_t kept = c < u[i] ? 1u : 0u;
      keepbits |= kept << i;
      if (kept && kept_tmp) kept_tmp[sstart + ahead] = idx[i];
      if ((uint32_t)(base + i) + 1 == send) seg_kept[cur_seg] = ahead + kept;
    }
  } else
#pragma unroll
  for (int i = 0; i < kDecItems; ++i) {
    const bool valid = base + i < n;
    if (!one_seg && valid) {
      const uint32_t sg = (uint32_t)(e[i] >> T.kshift);
      if (sg != cur_seg) {
        cur_seg = sg;
        K = ktab[sg];
        sstart = seg_off[sg];
        send = seg_off[sg + 1];
        hb_kept = (K.narrow & kSegHighFirst) ? win_off[sg] : 0u;
      }
    }
    /* reduction over the earlier requests of the same queue */
    const bool local = (lheadbits >> i) & 1u;
    const int32_t pre = local ? lv[i] : (RAW ? lv[i] + exc.m : min(lv[i], exc.m));
    uint32_t c, ahead;            /* batch-slot position; kept requests ahead in the queue */
    if (RAW) {
      c = r[i];
      ahead = r[i] == 0 ? 0u : (uint32_t)pre;
    } else {
      if (r[i] == 0) {
        c = 0;
      } else {
        const int64_t cc = (int64_t)r[i] - 1 + pre;               /* r-1 + min over t < r of (u_t - t) */
        c = cc < (int64_t)r[i] ? (uint32_t)cc : r[i];
      }
      if (K.narrow & kSegHighFirst) c = min(r[i], hb_kept);
      ahead = c;
    }
    const uint32_t round = K.cap_magic ? div_magic32(c, K.cap_magic) : c;     /* floor(c / cap) */
    est[i] = K.A + (long long)round * K.d;
    const uint32_t kept = (c < u[i] && valid) ? 1u : 0u;
    keepbits |= kept << i;
    if (kept && kept_tmp) kept_tmp[sstart + ahead] = idx[i];
    /* the last request of a queue knows the queue's kept count */
    if (valid && (uint32_t)(base + i) + 1 == send) seg_kept[cur_seg] = ahead + kept;
  }

  if (full) {
    if (out_keep) {
      /* bit k of a nibble -> byte k of a word */
      const uint32_t klo = ((keepbits & 15u) * 0x00204081u) & 0x01010101u;
      const uint32_t khi = (((keepbits >> 4) & 15u) * 0x00204081u) & 0x01010101u;
      *reinterpret_cast<uint2*>(out_keep + base) = make_uint2(klo, khi);
    }
    if (out_est) {
      store4(out_est + base, est[0], est[1], est[2], est[3]);
      store4(out_est + base + 4, est[4], est[5], est[6], est[7]);
    }
    if (out_perm)
      store4(out_perm + base, idx[0] | ((unsigned long long)idx[1] << 32),
             idx[2] | ((unsigned long long)idx[3] << 32), idx[4] | ((unsigned long long)idx[5] << 32),
             idx[6] | ((unsigned long long)idx[7] << 32));
  } else {
#pragma unroll
    for (int i = 0; i < kDecItems; ++i)
      if (base + i < n) {
        if (out_keep) out_keep[base + i] = (keepbits >> i) & 1u;
        if (out_est) out_est[base + i] = est[i];
        if (out_perm) out_perm[base + i] = idx[i];
      }
  }
  __syncthreads();
  }
}

__global__ void __launch_bounds__(1024)
k_kept_scan(const uint32_t* __restrict__ seg_kept, uint32_t n_seg, uint32_t* __restrict__ kept_base,
            uint32_t* __restrict__ chunk_base, uint32_t* __restrict__ out_seg_kept,
            unsigned long long* __restrict__ out_n_kept) {
  pdl_wait();
  kept_scan_block<1024>(seg_kept, n_seg, kept_base, chunk_base, out_seg_kept, out_n_kept);
}

/* Queue boundaries, window tables and output offsets of kWinQueues queues per block, from the sorted
 * elements:
 *   - every queue's first position: read off the last pass's digit counts when the queue id lies inside
 *     that digit, else a warp's 32-ary search for it in the elements' upper bits;
 *   - its number of windows, from its latest deadline, and a range of table entries for the block's
 *     queues from a shared counter (none left, or a queue with thousands: the scan path decides);
 *   - P of every entry, a lane each: four-way search of the window's first deadline in the queue;
 *   - E, Kp and the queue's kept count, a warp per queue; for a queue served high budget first the
 *     length of its kept prefix instead (win_off), by a warp's 32-ary search: its thresholds fall along
 *     the queue while the positions rise;
 *   - in the last block to finish, the output offsets of all queues' survivors.
 * Bound by dependent loads: the queue's constants are requested beside the boundaries, and P stays in shared memory until
 * E and Kp are there (8,192 queues of 305 requests 36.3 -> 29.2 us, 256 of 4,096 16.5 -> 15.0; seven probes per step of the
 * search instead of three: no gain).  As four launches (boundaries, entries of short queues by a lane and of long
 * ones by a warp each, prefixes, offsets) the same took 9 us more for 256 queues of 4,096 requests (a
 * replay epoch: 73 -> 64 us) and 12 more for 4,096 of them. */
constexpr int kWinQueues = 16;
constexpr int kWinThreads = 32 * kWinQueues;
constexpr uint32_t kWinEntries = 4096;           /* entries of a block whose P stay in shared memory until E and Kp are there */
__global__ void __launch_bounds__(kWinThreads, 2)
k_windows(PlanHeader* hdr, const unsigned long long* __restrict__ buf_a, const unsigned long long* __restrict__ buf_b, uint32_t n,
          uint32_t ibits, uint32_t n_seg, const PardSegConst* __restrict__ ktab, uint32_t* __restrict__ seg_off,
          uint32_t* __restrict__ out_seg_off, uint32_t* __restrict__ win_off, uint32_t* __restrict__ win_cnt,
          WinEntry* __restrict__ wtab, uint32_t capacity, uint32_t force_scan, const uint32_t* __restrict__ hist, uint32_t sbits,
          uint32_t local_candidate, uint32_t tables, uint32_t raw, uint32_t* __restrict__ seg_kept,
          uint32_t* __restrict__ kept_base, uint32_t* __restrict__ chunk_base, uint32_t* __restrict__ out_seg_kept,
          unsigned long long* __restrict__ out_n_kept, uint32_t direct) {
  pdl_wait();
  if (direct && hdr->direct) return;               /* (direct: the call may have its plan already) */
  __shared__ uint32_t s_lo[kWinQueues + 1], s_w[kWinQueues], s_first[kWinQueues + 1];
  __shared__ long long s_A[kWinQueues], s_d[kWinQueues];
  __shared__ uint32_t s_base, s_scan, s_P[kWinEntries];
  const uint32_t tid = threadIdx.x, lane = tid & 31, q = tid >> 5;
  const uint32_t s0 = blockIdx.x * kWinQueues, s = s0 + q;
  const PardSegConst K = ktab[min(s, n_seg - 1)];  /* (requested beside the boundaries) */
  const bool usable = hdr->wide == 0 && hdr->aborted == 0 && n > 0;       /* else nothing was sorted */
  const uint32_t npass = hdr->npass, dbits = hdr->dbits;
  const unsigned long long* src = (npass & 1) ? buf_b : buf_a;
  const unsigned long long dmask = dbits >= 64 ? ~0ull : ((1ull << dbits) - 1);
  /* first element whose queue id is >= s (warp 0 also: >= s0 + kWinQueues) */
  uint32_t lo[2] = {0, 0};
  const uint32_t want[2] = {s, q == 0 ? s0 + kWinQueues : s};
  if (usable) {
    const uint32_t top_bits = npass ? hdr->keybits - 8 * (npass - 1) : 0;   /* width of the last pass's digit */
    if (npass && sbits <= top_bits && !sort_is_local(hdr, local_candidate)) {
      /* the queue id is the upper part of that digit: the queue starts where the digits below
       * (s << (top_bits - sbits)) end */
      const uint32_t* h = hist + (npass - 1) * kBins;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const uint32_t limit = (uint32_t)min((unsigned long long)want[k] << (top_bits - sbits), (unsigned long long)kBins);
        uint32_t sum = 0;
        for (uint32_t d = lane; d < limit; d += 32) sum += h[d];
        lo[k] = __reduce_add_sync(0xffffffffu, sum);
      }
    } else {
      const uint32_t kshift = ibits + dbits;
      uint32_t hi[2] = {n, q == 0 ? n : 0u};
      while (lo[0] < hi[0] || lo[1] < hi[1]) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (lo[k] < hi[k]) {                     /* uniform across the warp */
            const uint32_t span = hi[k] - lo[k];
            const uint32_t p = lo[k] + (uint32_t)(((unsigned long long)(lane + 1) * span) / 33u);   /* lo <= p < hi */
            const bool less = (uint32_t)(__ldg(src + p) >> kshift) < want[k];
            const uint32_t c = __popc(__ballot_sync(0xffffffffu, less));   /* lanes 0..c-1 saw a smaller id */
            const uint32_t p_below = __shfl_sync(0xffffffffu, p, c > 0 ? c - 1 : 0);
            const uint32_t p_at = __shfl_sync(0xffffffffu, p, c < 32 ? c : 31);
            if (c > 0) lo[k] = p_below + 1;
            if (c < 32) hi[k] = p_at;
          }
        }
      }
    }
  }
  if (lane == 0) {
    s_lo[q] = lo[0];
    if (q == 0) s_lo[kWinQueues] = lo[1];
    if (s <= n_seg) {
      seg_off[s] = lo[0];
      if (out_seg_off) out_seg_off[s] = lo[0];
    }
    if (q == 0 && s0 + kWinQueues == n_seg) {
      seg_off[n_seg] = lo[1];
      if (out_seg_off) out_seg_off[n_seg] = lo[1];
    }
  }
  if (!tables) return;                             /* the boundaries are all the sequential rules need */
  if (tid == 0) s_scan = force_scan;
  __syncthreads();
  const uint32_t begin = s_lo[q], end = s_lo[q + 1];
  const bool mine = s < n_seg && usable && end > begin;
  bool high_first = false;
  {
    uint32_t w = 0;
    if (mine) {                                    /* whole warps */
      if (K.narrow & kSegNoStage) {
        if (lane == 0) set_status(hdr, PARD_EDATA);   /* requests queued at a stage the pipeline lacks */
      } else if (K.narrow & kSegHighFirst) {
        high_first = true;
        uint32_t a = begin, b = end;
        while (a < b) {                            /* uniform across the warp */
          const uint32_t span = b - a;
          const uint32_t p = a + (uint32_t)(((unsigned long long)(lane + 1) * span) / 33u);   /* a <= p < b */
          const bool kept = p - begin < threshold_u(slack_of((__ldg(src + p) >> ibits) & dmask, K), K);
          const uint32_t c = __popc(__ballot_sync(0xffffffffu, kept));   /* lanes 0..c-1 probe kept requests */
          const uint32_t p_below = __shfl_sync(0xffffffffu, p, c > 0 ? c - 1 : 0);
          const uint32_t p_at = __shfl_sync(0xffffffffu, p, c < 32 ? c : 31);
          if (c > 0) a = p_below + 1;
          if (c < 32) b = p_at;
        }
        if (lane == 0) { win_off[s] = a - begin; win_cnt[s] = 0; seg_kept[s] = a - begin; }   /* the kept prefix is the queue's kept count */
      } else {
        const long long X = (long long)((src[end - 1] >> ibits) & dmask) - K.A_rel;   /* latest deadline of the queue */
        const unsigned long long nb = X < 0 ? 0 : win_of((unsigned long long)X, K) + 1;
        if (nb >= kWinMaxPerSeg) { if (lane == 0) s_scan = 1; }
        else w = (uint32_t)nb + 1;                 /* windows 0..nb-1 and the end marker */
        if (lane == 0) { s_A[q] = K.A_rel; s_d[q] = K.d; }
      }
    }
    if (lane == 0) s_w[q] = w;
  }
  __syncthreads();
  if (tid < 32) {
    const uint32_t w = lane < kWinQueues ? s_w[lane] : 0u;
    uint32_t x = w;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    if (lane < kWinQueues) s_first[lane] = x - w;
    if (lane == 31) {
      s_first[kWinQueues] = x;
      const unsigned long long at = x && !s_scan ? atomicAdd(&hdr->win_total, (unsigned long long)x) : 0ull;
      if (at + x > (unsigned long long)capacity) s_scan = 1;
      s_base = (uint32_t)at;
      if (s_scan) hdr->use_scan = 1;
    }
  }
  __syncthreads();
  const uint32_t total = s_scan ? 0u : s_first[kWinQueues], base = s_base;
  if (lane == 0 && s < n_seg && !high_first) {
    win_off[s] = base + s_first[q];
    win_cnt[s] = total ? s_w[q] : 0u;
  }
  for (uint32_t e = tid; e < total; e += kWinThreads) {
    uint32_t k = 0;
#pragma unroll
    for (int b = kWinQueues / 2; b; b >>= 1)
      if (s_first[k + b] <= e) k += b;             /* last queue whose entries begin at or before e */
    const long long thr = s_A[k] + (long long)(e - s_first[k]) * s_d[k];     /* window >= b  <=>  deadline offset >= thr */
    const uint32_t first = s_lo[k];
    uint32_t a = first, b = s_lo[k + 1];
    while (a < b) {                                /* first position whose offset is >= thr; three probes per step */
      const uint32_t quarter = (b - a) / 4, m1 = a + quarter, m2 = a + 2 * quarter, m3 = a + 3 * quarter;   /* a <= m1 <= m2 <= m3 < b */
      const bool l1 = (long long)((__ldg(src + m1) >> ibits) & dmask) < thr, l2 = (long long)((__ldg(src + m2) >> ibits) & dmask) < thr,
                 l3 = (long long)((__ldg(src + m3) >> ibits) & dmask) < thr;
      if (l3) a = m3 + 1;
      else if (l2) { a = m2 + 1; b = m3; }
      else if (l1) { a = m1 + 1; b = m2; }
      else b = m1;
    }
    if (total <= kWinEntries) s_P[e] = a - first;
    else wtab[base + e].P = a - first;
  }
  __syncthreads();
  if (total && mine && !high_first && s_w[q]) {
    WinEntry* tab = wtab + base + s_first[q];
    const uint32_t kept = total <= kWinEntries ? win_prefix_warp<true>(K.cap, tab, s_w[q], lane, raw, s_P + s_first[q])
                                               : win_prefix_warp(K.cap, tab, s_w[q], lane, raw);
    if (lane == 0) seg_kept[s] = kept;             /* known before any request has been decided */
  }
  if (!last_block_done(&hdr->win_done)) return;
  kept_scan_block<kWinThreads>(seg_kept, n_seg, kept_base, chunk_base, out_seg_kept, out_n_kept);
}

/* The same for calls with very many short queues: a thread per queue (plain binary searches whose early
 * probes coincide across the lanes; its windows one after the other), 511 queues per block.  A thread's
 * chain of dependent loads is longer than a warp's, and the longer the more requests a queue has; but
 * k_windows keeps 4,736 queues in flight on 148 multiprocessors, so it walks its chain once per so many.
 * Whole calls, interleaved contexts, a warp / a thread per queue:
 *   queues              8,192      16,384     20,480     32,768     65,536
 *     32 requests each  113 / 123  185 / 181  177 / 165  235 / 200  415 / 290 us
 *    128                141 / 165  227 / 229  253 / 251  362 / 324  671 / 540
 *    256                197 / 224  315 / 323  364 / 370  549 / 523  1109 / 988
 *    512                279 / 316  487 / 512  634 / 687  967 / 963
 * so: from 16,384 queues on, with more than 128 queues per request of the average queue. */
constexpr uint32_t kManyQueues = 16384, kManyPerRequest = 128;
inline bool many_short_queues(uint64_t n, uint64_t n_seg) { return n_seg >= kManyQueues && n_seg * n_seg > kManyPerRequest * n; }
__global__ void __launch_bounds__(kWinThreads)
k_windows_many(PlanHeader* hdr, const unsigned long long* __restrict__ buf_a, const unsigned long long* __restrict__ buf_b, uint32_t n,
               uint32_t ibits, uint32_t n_seg, const PardSegConst* __restrict__ ktab, uint32_t* __restrict__ seg_off,
               uint32_t* __restrict__ out_seg_off, uint32_t* __restrict__ win_off, uint32_t* __restrict__ win_cnt,
               WinEntry* __restrict__ wtab, uint32_t capacity, uint32_t force_scan, uint32_t tables, uint32_t raw,
               uint32_t* __restrict__ seg_kept, uint32_t* __restrict__ kept_base, uint32_t* __restrict__ chunk_base,
               uint32_t* __restrict__ out_seg_kept, unsigned long long* __restrict__ out_n_kept, uint32_t direct) {
  pdl_wait();
  if (direct && hdr->direct) return;               /* (direct: the call may have its plan already) */
  __shared__ uint32_t s_lo[kWinThreads], s_warp[kWinThreads / 32], s_base, s_scan;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t s = blockIdx.x * (kWinThreads - 1u) + tid;          /* the last thread only finds the end of the one before */
  const bool usable = hdr->wide == 0 && hdr->aborted == 0 && n > 0;
  const uint32_t dbits = hdr->dbits, kshift = ibits + dbits;
  const unsigned long long* src = (hdr->npass & 1) ? buf_b : buf_a;
  const unsigned long long dmask = dbits >= 64 ? ~0ull : ((1ull << dbits) - 1);
  auto first_with = [&](uint32_t a, uint32_t b, auto below) {        /* first position in [a, b) that is not below */
    while (a < b) {
      const uint32_t mid = a + (b - a) / 2;
      if (below(mid, __ldg(src + mid))) a = mid + 1; else b = mid;
    }
    return a;
  };
  uint32_t lo = 0;
  if (usable && s <= n_seg) lo = first_with(0u, n, [&](uint32_t, unsigned long long e) { return (uint32_t)(e >> kshift) < s; });
  s_lo[tid] = lo;
  if (tid == 0) s_scan = force_scan;
  if (s <= n_seg && (tid + 1 < kWinThreads || s == n_seg)) {
    seg_off[s] = lo;
    if (out_seg_off) out_seg_off[s] = lo;
  }
  if (!tables) return;
  __syncthreads();
  const bool owner = tid + 1 < kWinThreads && s < n_seg;
  const uint32_t end = owner ? s_lo[tid + 1] : lo;
  uint32_t w = 0;
  bool high_first = false;
  if (owner && usable && end > lo) {
    const PardSegConst K = ktab[s];
    if (K.narrow & kSegNoStage) {
      set_status(hdr, PARD_EDATA);
    } else if (K.narrow & kSegHighFirst) {
      high_first = true;
      const uint32_t k = first_with(lo, end, [&](uint32_t p, unsigned long long e) { return p - lo < threshold_u(slack_of((e >> ibits) & dmask, K), K); }) - lo;
      win_off[s] = k;
      win_cnt[s] = 0;
      seg_kept[s] = k;
    } else {
      const long long X = (long long)((src[end - 1] >> ibits) & dmask) - K.A_rel;
      const unsigned long long nb = X < 0 ? 0 : win_of((unsigned long long)X, K) + 1;
      if (nb >= kWinMaxPerSeg) s_scan = 1;
      else w = (uint32_t)nb + 1;
    }
  }
  uint32_t x = w;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= (uint32_t)o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  const uint32_t v = lane < kWinThreads / 32 ? s_warp[lane] : 0u;
  const uint32_t total = __reduce_add_sync(0xffffffffu, v), before = x - w + __reduce_add_sync(0xffffffffu, lane < warp ? v : 0u);
  if (tid == 0) {
    const unsigned long long at = total && !s_scan ? atomicAdd(&hdr->win_total, (unsigned long long)total) : 0ull;
    if (at + total > (unsigned long long)capacity) s_scan = 1;
    s_base = (uint32_t)at;
    if (s_scan) hdr->use_scan = 1;
  }
  __syncthreads();
  if (owner && !high_first) {
    const bool scan = s_scan != 0;
    WinEntry* tab = wtab + s_base + before;
    win_off[s] = s_base + before;
    win_cnt[s] = scan ? 0u : w;
    if (!scan && w) {
      const PardSegConst K = ktab[s];
      uint32_t P = lo, kept = 0;
      int32_t E = kWinInf;
      for (uint32_t b = 0; b < w; ++b) {           /* entry b from what window b - 1 (at first: deadline < A) holds */
        const long long thr = K.A_rel + (long long)b * K.d;
        const uint32_t next = first_with(P, end, [&](uint32_t, unsigned long long e) { return (long long)((e >> ibits) & dmask) < thr; });
        const uint32_t p = P - lo, q = next - lo;
        if (q > p) {
          const uint32_t u = b ? win_u(b - 1, K.cap) : 0u;
          E = min(E, (int32_t)u - (int32_t)(q - 1));
          const uint32_t top = u < q ? u : q;
          kept += top > p ? top - p : 0;
        }
        tab[b].P = q;
        tab[b].E = E;
        tab[b].Kp = kept;
        P = next;
      }
      seg_kept[s] = raw ? kept : (uint32_t)((int32_t)(end - lo) - 1 + min(E, 1));
    }
  }
  if (!last_block_done(&hdr->win_done)) return;
  kept_scan_block<kWinThreads>(seg_kept, n_seg, kept_base, chunk_base, out_seg_kept, out_n_kept);
}

/* Decision pass from the window tables: every request on its own.  HF: some
 * queue may be served high budget first (the caller gave priorities). */
template <bool RAW, bool HF>
__device__ __forceinline__ void decide_tile(uint32_t tile, const PlanHeader* __restrict__ hdr, const unsigned long long* __restrict__ buf_a,
             const unsigned long long* __restrict__ buf_b, uint32_t n, uint32_t ibits,
             const PardSegConst* __restrict__ ktab, const uint32_t* __restrict__ seg_off,
             const uint32_t* __restrict__ win_off, const uint32_t* __restrict__ win_cnt,
             const WinEntry* __restrict__ wtab,
             uint8_t* __restrict__ out_keep, long long* __restrict__ out_est,
             uint32_t* __restrict__ out_perm, uint32_t* __restrict__ out_kept_idx, const uint32_t* __restrict__ kept_base) {
  /* The queues' kept counts followed from their tables, so the survivors go straight to their final
   * place: kept_base holds the queues' output offsets. */
  const TileCtx T = make_tile_ctx(hdr, buf_a, buf_b, n, ibits, ktab, seg_off);
  const uint64_t base = ((uint64_t)tile * kDecThreads + threadIdx.x) * kDecItems;
  if (threadIdx.x == 0) l2_ahead(T.src, base, (uint64_t)kDecAhead * kDecTile, kDecTile, n);
  if (base >= n) return;
  const bool full = base + kDecItems <= n;
  unsigned long long e[kDecItems];
  if (full) {
    load4(T.src + base, e);
    load4(T.src + base + 4, e + 4);
  } else {
#pragma unroll
    for (int i = 0; i < kDecItems; ++i) e[i] = base + i < n ? T.src[base + i] : 0;
  }
  uint32_t cur_seg = (uint32_t)(e[0] >> T.kshift);
  PardSegConst K = ktab[cur_seg];
  uint32_t sstart = seg_off[cur_seg], woff = win_off[cur_seg], wcnt = win_cnt[cur_seg];
  uint32_t koff = out_kept_idx ? kept_base[cur_seg] : 0u;
  const bool narrow = T.narrow && (K.narrow & (kSegNarrow | kSegNoStage)) == kSegNarrow && full &&
                      cur_seg == (uint32_t)(e[kDecItems - 1] >> T.kshift);
  const int32_t A32 = narrow_A(K);

  uint32_t keepbits = 0, idx[kDecItems];
  long long est[kDecItems];
#pragma unroll
  for (int i = 0; i < kDecItems; ++i) {
    const uint64_t j = base + i;
    const bool valid = j < n;
    uint32_t c = 0, ahead = 0, kept = 0;
    idx[i] = (uint32_t)e[i] & T.imask;
    if (valid) {
      long long X;
      if (narrow) {
        const int32_t off = (int32_t)(__funnelshift_r((uint32_t)e[i], (uint32_t)(e[i] >> 32), T.ibits) & (uint32_t)T.dmask);
        X = (HF && (K.narrow & kSegHighFirst)) ? A32 - off : off - A32;
      } else {
        const uint32_t sg = (uint32_t)(e[i] >> T.kshift);
        if (sg != cur_seg) {
          cur_seg = sg;
          K = ktab[sg];
          sstart = seg_off[sg];
          koff = out_kept_idx ? kept_base[sg] : 0u;
          woff = win_off[sg];
          wcnt = win_cnt[sg];
        }
        X = HF ? slack_of((e[i] >> T.ibits) & T.dmask, K) : (long long)((e[i] >> T.ibits) & T.dmask) - K.A_rel;
      }
      const uint32_t r = (uint32_t)j - sstart;
      uint32_t u = 0;
      if (HF && (K.narrow & kSegHighFirst)) {                 /* the kept requests are the first woff of the queue */
        u = threshold_u(X, K);
        ahead = min(r, woff);
        c = RAW ? r : ahead;
      } else if (X >= 0) {                            /* window b of the request and its table entry */
        const unsigned long long b64 = win_of((unsigned long long)X, K);
        /* The queue's table has an entry for every window up to its latest deadline's.  A queue
         * without a table (input errors: a stage its pipeline lacks, constants left at their
         * defaults) must not index one: its requests count as dropped, the call reports PARD_EDATA. */
        if (b64 >= (unsigned long long)wcnt) {
          set_status(T.hdr, PARD_EDATA);
          est[i] = K.A;
          continue;
        }
        const uint32_t b = (uint32_t)b64;
        u = win_u(b, K.cap);
        const WinEntry w = wtab[woff + b];
        if (RAW) {
          const uint32_t top = r < u ? r : u;
          ahead = w.Kp + (top > w.P ? top - w.P : 0);
          c = r;
        } else {
          /* min over t < r of (u_t - t); values above 1 cannot lower the position */
          int32_t m = w.E;
          if (r > w.P) m = min(m, (int32_t)u - (int32_t)(r - 1));
          c = r == 0 ? 0u : r - 1 + (uint32_t)min(m, 1);
          ahead = c;
        }
      } else {                                        /* deadline before even position 0 completes */
        c = RAW ? r : 0u;
      }
      kept = c < u ? 1u : 0u;
      const uint32_t round = K.cap_magic ? div_magic32(c, K.cap_magic) : c;
      est[i] = K.A + (long long)((unsigned long long)round * (unsigned long long)K.d);
      if (kept && out_kept_idx) out_kept_idx[koff + ahead] = idx[i];
    }
    keepbits |= kept << i;
  }
  if (full) {
    if (out_keep) {
      const uint32_t klo = ((keepbits & 15u) * 0x00204081u) & 0x01010101u;
      const uint32_t khi = (((keepbits >> 4) & 15u) * 0x00204081u) & 0x01010101u;
      *reinterpret_cast<uint2*>(out_keep + base) = make_uint2(klo, khi);
    }
    if (out_est) {
      store4(out_est + base, est[0], est[1], est[2], est[3]);
      store4(out_est + base + 4, est[4], est[5], est[6], est[7]);
    }
    if (out_perm)
      store4(out_perm + base, idx[0] | ((unsigned long long)idx[1] << 32),
             idx[2] | ((unsigned long long)idx[3] << 32), idx[4] | ((unsigned long long)idx[5] << 32),
             idx[6] | ((unsigned long long)idx[7] << 32));
  } else {
#pragma unroll
    for (int i = 0; i < kDecItems; ++i)
      if (base + i < n) {
        if (out_keep) out_keep[base + i] = (keepbits >> i) & 1u;
        if (out_est) out_est[base + i] = est[i];
        if (out_perm) out_perm[base + i] = idx[i];
      }
  }
}

/* A tile per block. */
template <bool RAW, bool HF>
__global__ void __launch_bounds__(kDecThreads, 8)
k_decide_win(const PlanHeader* __restrict__ hdr, const unsigned long long* __restrict__ buf_a, const unsigned long long* __restrict__ buf_b, uint32_t n,
             uint32_t ibits, const PardSegConst* __restrict__ ktab, const uint32_t* __restrict__ seg_off, const uint32_t* __restrict__ win_off,
             const uint32_t* __restrict__ win_cnt, const WinEntry* __restrict__ wtab, uint8_t* __restrict__ out_keep,
             long long* __restrict__ out_est, uint32_t* __restrict__ out_perm, uint32_t* __restrict__ out_kept_idx,
             const uint32_t* __restrict__ kept_base) {
  pdl_wait();
  if (hdr->direct | hdr->use_scan | hdr->wide | hdr->aborted) return;
  decide_tile<RAW, HF>(blockIdx.x, hdr, buf_a, buf_b, n, ibits, ktab, seg_off, win_off, win_cnt, wtab, out_keep, out_est, out_perm, out_kept_idx, kept_base);
}
/* For calls that mostly have their plan by then (pard_direct.cuh): fewer blocks, which take one tile after the other.  A
 * block per tile, 16,384 at 2^24 requests, took 11 us to find that there is nothing to do; a block that goes on to a next
 * tile decides a little slower than a new one.  Five rounds of the seven blocks that fit a multiprocessor: 2^24 requests of 64
 * contexts out of order 537.6 us with a block per tile, 542.5 with four rounds, 539.7 like this, of 256 contexts 545.7, 545,
 * 545; those in order 244.8, 233.2, 233.7. */
constexpr uint32_t kRestBlocks = 7, kRestRounds = 5;
__global__ void __launch_bounds__(kDecThreads, kRestBlocks)
k_decide_rest(const PlanHeader* __restrict__ hdr, const unsigned long long* __restrict__ buf_a, const unsigned long long* __restrict__ buf_b, uint32_t n,
              uint32_t ibits, const PardSegConst* __restrict__ ktab, const uint32_t* __restrict__ seg_off, const uint32_t* __restrict__ win_off,
              const uint32_t* __restrict__ win_cnt, const WinEntry* __restrict__ wtab, uint8_t* __restrict__ out_keep,
              long long* __restrict__ out_est, uint32_t* __restrict__ out_perm, uint32_t* __restrict__ out_kept_idx,
              const uint32_t* __restrict__ kept_base) {
  pdl_wait();
  if (hdr->direct | hdr->use_scan | hdr->wide | hdr->aborted) return;
  const uint32_t tiles = (uint32_t)(((uint64_t)n + kDecTile - 1) / kDecTile);
  for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x)
    decide_tile<false, false>(tile, hdr, buf_a, buf_b, n, ibits, ktab, seg_off, win_off, win_cnt, wtab, out_keep, out_est, out_perm, out_kept_idx, kept_base);
}

/* Packs the queues' survivors: copy job j moves up to kCompactChunk indices of one queue; a
 * warp per job. */
__device__ __forceinline__ void kept_move_jobs(const uint32_t* __restrict__ kept_tmp, const uint32_t* __restrict__ seg_off,
                                               const uint32_t* __restrict__ seg_kept, const uint32_t* __restrict__ kept_base,
                                               const uint32_t* __restrict__ chunk_base, uint32_t n_seg,
                                               uint32_t* __restrict__ out_kept_idx) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t jobs = __ldcg(&chunk_base[n_seg]), step = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t job = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; job < jobs; job += step) {
    uint32_t lo = 0, hi = n_seg;                 /* last queue whose first job is <= job */
    while (hi - lo > 1) {
      const uint32_t mid = lo + (hi - lo) / 2;
      if (__ldcg(&chunk_base[mid]) <= job) lo = mid; else hi = mid;
    }
    const uint32_t s = lo;
    const uint32_t first = (job - __ldcg(&chunk_base[s])) * kCompactChunk;
    const uint32_t count = min((uint32_t)kCompactChunk, __ldcg(&seg_kept[s]) - first);
    const uint32_t* src = kept_tmp + seg_off[s] + first;
    uint32_t* dst = out_kept_idx + __ldcg(&kept_base[s]) + first;
    uint32_t i = lane;
    for (; i + 224 < count; i += 256) {            /* eight loads in flight per lane */
      uint32_t v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = __ldcg(&src[i + 32 * k]);
#pragma unroll
      for (int k = 0; k < 8; ++k) dst[i + 32 * k] = v[k];
    }
    for (; i < count; i += 32) dst[i] = __ldcg(&src[i]);
  }
}

/* The decision by scanning, from the sorted elements to the packed survivors, as ONE kernel: the
 * fallback for calls whose queues have too many batch windows for the tables (and what
 * PARD_MODE_SCAN asks for).  Launched on every call; returns at once when the tables did the
 * work.  Five steps: tile aggregates, their scan, the decision, the queues' kept counts into output
 * offsets, the packing of the survivors.  The tiles of a step are taken by ticket, a run of them at a
 * time, and every block hands in how many runs it has done; the block that completes the step also does
 * the one-block step behind it and then sets a flag, which the others wait for before they go on.  So a wait
 * is only ever for blocks that run already, and those that run finish the call, however few of the grid
 * are placed at a time; each wait is bounded all the same (PARD_ETIMEOUT, every block gives up, nothing
 * hangs).  Bound by the two reads of the elements and by the one-block steps: forced for 2^24 requests the
 * call takes 726 us, for a million 62.0 (713 and 58.9 when a wait was for every block of the grid; every run
 * handed in by itself: 733 and 66). */
constexpr uint32_t kScanRuns = 4;                /* runs of tiles per block of the grid: blocks that start late find less to do */
/* The block's share of a step: work(first tile, end) for every run it gets hold of, the next ticket fetched
 * while a run is worked on.  True in the block that completes the step.  stall: testing aid, the first run
 * is never handed in. */
template <typename Work>
__device__ __forceinline__ bool scan_step(uint32_t* ticket, uint32_t* done, uint32_t n_tiles, bool stall, Work work) {
  __shared__ uint32_t s_next;
  const uint32_t per = (n_tiles + kScanRuns * gridDim.x - 1) / (kScanRuns * gridDim.x), runs = (n_tiles + per - 1) / per;
  uint32_t mine = 0, next = 0;
  if (threadIdx.x == 0) s_next = atomicAdd(ticket, 1u);
  __syncthreads();
  for (uint32_t t = s_next; t < runs; t = s_next) {
    if (threadIdx.x == 0) next = atomicAdd(ticket, 1u);
    work(t * per, min((t + 1) * per, n_tiles));
    mine += stall && t == 0 ? 0u : 1u;
    __syncthreads();
    if (threadIdx.x == 0) s_next = next;
    __syncthreads();
  }
  return last_arrival(done, mine, runs);
}
__device__ __forceinline__ void set_flag(uint32_t* word) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) atomicExch(word, 1u);
}
template <bool RAW>
__global__ void __launch_bounds__(kDecThreads, 3)
k_scan_path(PlanHeader* hdr, const unsigned long long* __restrict__ buf_a,
            const unsigned long long* __restrict__ buf_b, uint32_t n, uint32_t ibits, uint32_t n_seg,
            const PardSegConst* __restrict__ ktab, const uint32_t* __restrict__ seg_off,
            const uint32_t* __restrict__ win_off, unsigned long long* __restrict__ tile_agg, int32_t* __restrict__ carry,
            uint8_t* __restrict__ out_keep, long long* __restrict__ out_est, uint32_t* __restrict__ out_perm,
            uint32_t* __restrict__ kept_tmp, uint32_t* __restrict__ seg_kept, uint32_t* __restrict__ kept_base,
            uint32_t* __restrict__ chunk_base, uint32_t* __restrict__ out_seg_kept,
            unsigned long long* __restrict__ out_n_kept, uint32_t* __restrict__ out_kept_idx, uint32_t stall) {
  pdl_wait();
  if (hdr->wide || !hdr->use_scan || gave_up(hdr)) return;
  const uint32_t n_tiles = (n + kDecTile - 1) / kDecTile;
  if (scan_step(&hdr->scan_ticket[0], &hdr->scan_done[0], n_tiles, stall != 0, [&](uint32_t first, uint32_t end) {
        tile_agg_tiles<RAW>(hdr, buf_a, buf_b, n, ibits, ktab, seg_off, tile_agg, first, end);
      })) {
    tile_scan_block<RAW, kDecThreads>(tile_agg, n_tiles, carry);
    set_flag(&hdr->scan_flag[0]);
  }
  if (!finish_pieces(hdr, &hdr->scan_flag[0], 0u, 1u)) return;
  if (scan_step(&hdr->scan_ticket[1], &hdr->scan_done[1], n_tiles, false, [&](uint32_t first, uint32_t end) {
        decide_tiles<RAW>(hdr, buf_a, buf_b, n, ibits, ktab, seg_off, win_off, carry, out_keep, out_est, out_perm, kept_tmp, seg_kept, first, end);
      })) {
    kept_scan_block<kDecThreads>(seg_kept, n_seg, kept_base, chunk_base, out_seg_kept, out_n_kept);
    set_flag(&hdr->scan_flag[1]);
  }
  if (!finish_pieces(hdr, &hdr->scan_flag[1], 0u, 1u)) return;
  if (out_kept_idx) kept_move_jobs(kept_tmp, seg_off, seg_kept, kept_base, chunk_base, n_seg, out_kept_idx);
}

/* ------------------------------------------------------------------------ */
/* keys wider than one sort element                                          */
/* ------------------------------------------------------------------------ */
/* When segment, deadline and index bits together exceed 64 (deadline spans of years, millions
 * of queues and requests at once) the key (segment | deadline offset, up to 84 bits) is sorted
 * in chunks, least significant first, each chunk by the ordinary passes: a chunk's element is
 * chunk << ibits | current position, so every super-pass is a stable sort of the current
 * order by one more chunk, and the positions it yields are chased back to request indices.
 * The last super-pass leaves the order of the requests; the elements are then rewritten as
 * segment | index (no deadline bits) and the decision is taken by the queue walk, which looks
 * the deadlines up in the request array.  A slow path for legal but extreme inputs.
 * Once a wait of the passes has run out (`aborted`) the elements are no longer positions, and none of
 * these kernels may follow them. */
__device__ __forceinline__ uint32_t wide_chunk_bits(const PlanHeader* hdr, uint32_t sbits, uint32_t ibits, uint32_t super) {
  const uint32_t kb = sbits + hdr->dbits, cw = 64 - ibits, lo = super * cw;
  return lo < kb ? min(cw, kb - lo) : 0u;
}

__global__ void __launch_bounds__(256)
k_wide_reset(PlanHeader* hdr, uint32_t* __restrict__ hist, uint32_t* __restrict__ lookback, unsigned long long lb_words,
             uint32_t sbits, uint32_t ibits, uint32_t super) {
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    hdr->npass = (wide_chunk_bits(hdr, sbits, ibits, super) + 7) / 8;
    hdr->keybits = wide_chunk_bits(hdr, sbits, ibits, super);   /* what the passes of this super-pass sort */
    hdr->pshift = 0;
    for (int i = 0; i <= kMaxPasses; ++i) hdr->ticket[i] = 0;
    for (int i = 0; i < kMaxPasses; ++i) hdr->sort_bar[i] = 0;
    if (super == 0) {
      hdr->wide = 2;                                      /* the chunked sort is under way */
      hdr->status = hdr->bad_input ? (uint32_t)(-PARD_EDATA) : 0u;   /* the width was not an error after all */
    }
  }
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < lb_words + kMaxPasses * kBins; i += step) {
    if (i < lb_words) lookback[i] = 0;
    else hist[i - lb_words] = 0;
  }
}

__global__ void __launch_bounds__(256)
k_wide_pack(const uint4* __restrict__ req, uint32_t n, uint32_t n_ctx, uint32_t S,
            const unsigned long long* __restrict__ ctx_dmin_inv, const unsigned long long* __restrict__ ctx_dmax,
            const uint8_t* __restrict__ priority, uint32_t sbits, uint32_t ibits, uint32_t super,
            const PlanHeader* __restrict__ hdr, const uint32_t* __restrict__ order,
            unsigned long long* __restrict__ dst, uint32_t* __restrict__ hist) {
  pdl_wait();
  __shared__ uint32_t s_hist[kMaxPasses * kBins];
  if (hdr->aborted) return;
  const uint32_t bits = wide_chunk_bits(hdr, sbits, ibits, super), npass = (bits + 7) / 8;
  const uint32_t dbits = hdr->dbits, lo = super * (64 - ibits);
  for (uint32_t i = threadIdx.x; i < npass * kBins; i += blockDim.x) s_hist[i] = 0;
  __syncthreads();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride) {
    const uint32_t orig = super == 0 ? (uint32_t)p : order[p];
    const uint4 r = __ldg(&req[orig]);
    const unsigned long long D = ((unsigned long long)r.y << 32) | r.x;
    const uint32_t ctx = r.z, stage = r.w & 0xffffu;
    unsigned long long chunk = 0;
    if (ctx < n_ctx && stage < S && D < (unsigned long long)PARD_TIME_LIMIT_US && bits) {
      const uint32_t seg = ctx * S + stage;
      const bool high_first = priority && __ldg(&priority[seg]) != 0;
      const unsigned long long off = high_first ? ctx_dmax[ctx] - D : D - ~ctx_dmin_inv[ctx];
      const unsigned __int128 key = ((unsigned __int128)seg << dbits) | off;
      chunk = (unsigned long long)(key >> lo) & (bits >= 64 ? ~0ull : ((1ull << bits) - 1));
    }
    dst[p] = (chunk << ibits) | p;                        /* flagged requests sort first, into queue 0 */
    for (uint32_t q = 0; q < npass; ++q) atomicAdd(&s_hist[q * kBins + ((chunk >> (8 * q)) & 255u)], 1u);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < npass * kBins; i += blockDim.x)
    if (s_hist[i]) atomicAdd(&hist[i], s_hist[i]);
}

/* positions of a super-pass -> request indices, into the buffer the sort has left free */
__global__ void __launch_bounds__(256)
k_wide_chase(const PlanHeader* __restrict__ hdr, const unsigned long long* __restrict__ buf_a,
             unsigned long long* __restrict__ buf_b, uint32_t n, uint32_t ibits, uint32_t super,
             const uint32_t* __restrict__ order) {
  pdl_wait();
  if (hdr->aborted) return;
  const bool odd = hdr->npass & 1;
  const unsigned long long* sorted = odd ? buf_b : buf_a;
  uint32_t* tmp = reinterpret_cast<uint32_t*>(odd ? const_cast<unsigned long long*>(buf_a) : buf_b);
  const uint32_t imask = (1u << ibits) - 1;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride) {
    const uint32_t pos = (uint32_t)sorted[q] & imask;
    tmp[q] = super == 0 ? pos : order[pos];
  }
}

__global__ void __launch_bounds__(256)
k_wide_keep(const PlanHeader* __restrict__ hdr, const unsigned long long* __restrict__ buf_a,
            const unsigned long long* __restrict__ buf_b, uint32_t n, uint32_t* __restrict__ order) {
  pdl_wait();
  if (hdr->aborted) return;
  const uint32_t* tmp = reinterpret_cast<const uint32_t*>((hdr->npass & 1) ? buf_a : buf_b);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride) order[q] = tmp[q];
}

/* the sorted order as elements without deadline bits: segment | request index, in buf_a */
__global__ void __launch_bounds__(256)
k_wide_final(const uint4* __restrict__ req, uint32_t n, uint32_t n_ctx, uint32_t S, uint32_t sbits, uint32_t ibits,
             PlanHeader* hdr, const uint32_t* __restrict__ order, unsigned long long* __restrict__ buf_a) {
  pdl_wait();
  if (hdr->aborted) return;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride) {
    const uint32_t orig = order[q];
    const uint4 r = __ldg(&req[orig]);
    const unsigned long long D = ((unsigned long long)r.y << 32) | r.x;
    const uint32_t ctx = r.z, stage = r.w & 0xffffu;
    const bool ok = ctx < n_ctx && stage < S && D < (unsigned long long)PARD_TIME_LIMIT_US;
    buf_a[q] = ((unsigned long long)(ok ? ctx * S + stage : 0u) << ibits) | orig;
  }
}

/* after k_wide_final: the header as the kernels behind the sort expect it */
__global__ void k_wide_done(PlanHeader* hdr, uint32_t sbits) {
  pdl_wait();
  hdr->dbits = 0;
  hdr->keybits = sbits;
  hdr->npass = 0;
  hdr->wide = 0;
  hdr->lookup = 1;
}

/* ---- optional phase timing (process-wide) ---- */
constexpr int kEventsPerSample = PARD_N_PHASES + 1;
static_assert(PARD_N_PHASES == 4 + kMaxPasses + 3, "phase list");
struct Profiler {
  std::mutex mu;
  cudaEvent_t* last = nullptr;       /* events of the most recent sampled call */
  std::atomic<bool> on{false};       /* read without the lock by every pard_plan call */
  bool coarse = false;
  uint32_t every = 1, max_samples = 0, calls = 0, n_samples = 0;
  std::vector<cudaEvent_t> ev;
};
Profiler g_prof;

constexpr int kPhaseTables = 4 + kMaxPasses;       /* "tables", then "decide", "compact" */

/* events of this call if it is a sampled one, else nullptr */
cudaEvent_t* profile_acquire(bool* coarse) {
  if (!g_prof.on.load(std::memory_order_acquire)) return nullptr;   /* the usual case: no lock taken */
  std::lock_guard<std::mutex> lock(g_prof.mu);
  if (!g_prof.on.load(std::memory_order_relaxed)) return nullptr;
  *coarse = g_prof.coarse;
  uint32_t call = g_prof.calls++;
  g_prof.last = nullptr;
  if (call % g_prof.every != 0 || g_prof.n_samples >= g_prof.max_samples) return nullptr;
  g_prof.last = g_prof.ev.data() + (size_t)(g_prof.n_samples++) * kEventsPerSample;
  return g_prof.last;
}

/* the sort pass needs more dynamic shared memory than the default limit: opt in once per device */
int allow_sort_smem(int dev) {
  static std::mutex mu;
  static std::atomic<bool> done[64];
  if (dev < 0 || dev >= 64) return PARD_ERANGE;
  if (done[dev].load(std::memory_order_acquire)) return PARD_OK;    /* every call but the first on a device */
  std::lock_guard<std::mutex> lock(mu);
  if (!done[dev].load(std::memory_order_relaxed)) {
    PARD_CUDA_OK(cudaFuncSetAttribute(k_sort_pass<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem)));
    PARD_CUDA_OK(cudaFuncSetAttribute(k_sort_pass<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem)));
    PARD_CUDA_OK(cudaFuncSetAttribute(k_sort_rest<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem)));
    PARD_CUDA_OK(cudaFuncSetAttribute(k_sort_rest<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem)));
    PARD_CUDA_OK(cudaFuncSetAttribute(k_sort_rest<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem)));
    PARD_CUDA_OK(cudaFuncSetAttribute(k_sort_local, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(SortSmem)));
    PARD_CUDA_OK(cudaFuncSetAttribute(k_sort_requests<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem)));
    PARD_CUDA_OK(cudaFuncSetAttribute(k_sort_requests<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem)));
    int rc = allow_local_smem();
    if (rc == PARD_OK) rc = allow_walk_smem();
    if (rc != PARD_OK) return rc;
    done[dev].store(true, std::memory_order_release);
  }
  return PARD_OK;
}


int check_state(const pard_queue_state_t* st, uint32_t n_ctx) {
  if (!st) return PARD_EINVAL;
  if (st->stage_stride < 1) return PARD_EINVAL;
  if (st->stage_stride > PARD_MAX_STAGES) return PARD_ERANGE;
  if (!st->d_now_us || !st->d_batch || !st->d_free_at_us || !st->d_q_us) return PARD_EINVAL;
  if (st->d_w_us && st->slot_stride < 0) return PARD_EINVAL;
  if (n_ctx < 1) return PARD_EINVAL;
  if ((uint64_t)n_ctx * (uint64_t)st->stage_stride > PARD_MAX_SEGMENTS) return PARD_ERANGE;
  return PARD_OK;
}

}  // namespace

/* pard_goodput follows pard_plan on the same stream and belongs to the same pass over the
 * sorted queues: when the plan call just before it was a sampled one, the end of its last phase
 * moves behind the goodput kernel. */
void pard_profile_extend_last(cudaStream_t stream) {
  if (!g_prof.on.load(std::memory_order_acquire)) return;
  std::lock_guard<std::mutex> lock(g_prof.mu);
  if (g_prof.on.load(std::memory_order_relaxed) && g_prof.last) cudaEventRecord(g_prof.last[PARD_N_PHASES], stream);
}

extern "C" int pard_plan_workspace_bytes(uint64_t n, uint32_t n_ctx, int32_t stage_stride,
                                         uint64_t* bytes) {
  if (!bytes || n_ctx < 1 || stage_stride < 1) return PARD_EINVAL;
  if (n >= PARD_MAX_REQUESTS || stage_stride > PARD_MAX_STAGES ||
      (uint64_t)n_ctx * (uint64_t)stage_stride > PARD_MAX_SEGMENTS)
    return PARD_ERANGE;
  *bytes = make_layout(n, n_ctx, stage_stride).total;
  return PARD_OK;
}

extern "C" int pard_plan(const pard_pipeline_t* const* pipelines, uint32_t n_pipelines,
                         const pard_request_t* d_requests, uint64_t n,
                         const pard_queue_state_t* state, uint32_t n_ctx, uint32_t mode,
                         const pard_plan_out_t* out, void* d_workspace, uint64_t workspace_bytes,
                         void* cuda_stream) {
  return pard_plan_policy(pipelines, n_pipelines, d_requests, nullptr, n, state, n_ctx, mode, out, d_workspace,
                          workspace_bytes, cuda_stream);
}

extern "C" int pard_plan_policy(const pard_pipeline_t* const* pipelines, uint32_t n_pipelines,
                                const pard_request_t* d_requests, const pard_arrival_t* d_arrivals, uint64_t n,
                                const pard_queue_state_t* state, uint32_t n_ctx, uint32_t mode,
                                const pard_plan_out_t* out, void* d_workspace, uint64_t workspace_bytes,
                                void* cuda_stream) {
  /* ---- host-side checks, nothing launched before they pass ---- */
  if (!pipelines || n_pipelines < 1 || !out) return PARD_EINVAL;
  if (n_pipelines > kMaxPipelinesPerCall) return PARD_ERANGE;
  constexpr uint32_t kRuleBits = PARD_MODE_PATH_MASK | PARD_MODE_FCFS | PARD_MODE_NEXUS | PARD_MODE_CLIPPER;
  if (mode & ~(PARD_MODE_RAW | PARD_MODE_NOWAIT | PARD_MODE_SCAN | PARD_MODE_TEST_STALL | PARD_MODE_GROUPED | kRuleBits))
    return PARD_EINVAL;
  /* the rules decided by a walk of every queue, and what they combine with */
  const bool rule_walk = (mode & kRuleBits) != 0;
  const bool arrival_order = (mode & (PARD_MODE_FCFS | PARD_MODE_NEXUS | PARD_MODE_CLIPPER)) != 0;
  if (rule_walk && (mode & PARD_MODE_RAW)) return PARD_EINVAL;
  if ((mode & PARD_MODE_NEXUS) && (mode & (PARD_MODE_CLIPPER | PARD_MODE_PATH_MASK))) return PARD_EINVAL;
  if ((mode & PARD_MODE_CLIPPER) && (mode & PARD_MODE_PATH_MASK)) return PARD_EINVAL;
  if ((mode & PARD_MODE_CLIPPER) && n > 0 && (!d_arrivals || ((uintptr_t)d_arrivals & 15))) return PARD_EINVAL;
  if (arrival_order && state && state->d_priority) return PARD_EINVAL;
  int rc = check_state(state, n_ctx);
  if (rc != PARD_OK) return rc;
  if (n >= PARD_MAX_REQUESTS) return PARD_ERANGE;
  if (n > 0 && !d_requests) return PARD_EINVAL;
  if ((uintptr_t)d_requests & 15) return PARD_EINVAL;
  int dev = -1;
  PARD_CUDA_OK(cudaGetDevice(&dev));
  int32_t max_slots = 0;
  for (uint32_t i = 0; i < n_pipelines; ++i) {
    const pard_pipeline_t* p = pipelines[i];
    if (!p || !p->d_blob || p->device != dev) return PARD_EINVAL;
    if (p->n_stages > state->stage_stride) return PARD_EINVAL;
    max_slots = std::max(max_slots, p->n_slots);
  }
  if (state->d_w_us && state->slot_stride < max_slots) return PARD_EINVAL;
  if (!d_workspace || ((uintptr_t)d_workspace & 255)) return PARD_EINVAL;
  const Layout L = make_layout(n, n_ctx, state->stage_stride);
  if (workspace_bytes < L.total) return PARD_EWORKSPACE;
  if ((out->d_est_us && ((uintptr_t)out->d_est_us & 15)) ||
      (out->d_perm && ((uintptr_t)out->d_perm & 15)) ||
      (out->d_keep && ((uintptr_t)out->d_keep & 7)))
    return PARD_EINVAL;

  cudaStream_t stream = (cudaStream_t)cuda_stream;
  char* ws = (char*)d_workspace;
  PlanHeader* hdr = (PlanHeader*)(ws + L.hdr);
  unsigned long long* ctx_dmin = (unsigned long long*)(ws + L.ctx_dmin);
  unsigned long long* ctx_dmax = (unsigned long long*)(ws + L.ctx_dmax);
  uint32_t* seg_off = (uint32_t*)(ws + L.seg_off);
  PardSegConst* ktab = (PardSegConst*)(ws + L.ktab);
  uint32_t* hist = (uint32_t*)(ws + L.hist);
  uint32_t* lookback = (uint32_t*)(ws + L.lookback);
  const size_t lb_words = (size_t)L.lb_rows * kBins;
  unsigned long long* tile_agg = (unsigned long long*)(ws + L.tile_agg);
  int32_t* tile_carry = (int32_t*)(ws + L.tile_carry);
  uint32_t* seg_kept = (uint32_t*)(ws + L.seg_kept);
  uint32_t* kept_base = (uint32_t*)(ws + L.kept_base);
  uint32_t* chunk_base = (uint32_t*)(ws + L.chunk_base);
  uint32_t* kept_tmp = (uint32_t*)(ws + L.kept_tmp);
  uint32_t* win_off = (uint32_t*)(ws + L.win_off);
  WinEntry* wtab = (WinEntry*)(ws + L.wtab);
  uint32_t* win_cnt = (uint32_t*)(ws + L.win_cnt);
  uint32_t* whist = (uint32_t*)(ws + L.whist);
  unsigned long long* buf_a = (unsigned long long*)(ws + L.buf_a);
  unsigned long long* buf_b = (unsigned long long*)(ws + L.buf_b);
  const uint32_t n32 = (uint32_t)n;
  const uint32_t S = (uint32_t)state->stage_stride;
  const uint32_t ibits = std::max(1u, ceil_log2(n));
  const uint32_t sbits = ceil_log2(L.n_seg);

  bool prof_coarse = false;
  /* requests grouped by ctx, no ctx beyond a tile: worth testing for when the sizes allow it */
  const uint32_t local_cand = local_sort_candidate(n, n_ctx) ? 1u : 0u;
  /* one ctx that fits a tile: the local sort is certain, no range search, no order check, no fallback passes */
  const bool local_sure = local_cand && n_ctx == 1;
  uint32_t* ctx_start = (uint32_t*)(ws + L.ctx_start);
  cudaEvent_t* evs = profile_acquire(&prof_coarse);
  int phase = 0;
  auto mark = [&]() {                      /* boundary between two phases */
    const bool inner = phase == kPhaseTables + 1 || phase == kPhaseTables + 2;   /* inside the decision pass */
    if (evs && !(prof_coarse && inner)) cudaEventRecord(evs[phase], stream);
    ++phase;
  };
  mark();
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  PipeTable pipe_table;
  rc = pard_pipe_table(pipelines, n_pipelines, ws + L.pipes, stream, &pipe_table);
  if (rc != PARD_OK) return rc;
  rc = allow_sort_smem(dev);
  if (rc != PARD_OK) return rc;
  const uint4* req4 = (const uint4*)d_requests;

  /* the decision by a walk of every queue (pard_policy.cu), between the sort and the outputs */
  auto decide_by_walk = [&](PolicyArgs& pa) -> int {
    pa.rounds = win_cnt; pa.tail = win_off; pa.tile_x = (uint32_t*)tile_carry;
    pa.out_keep = out->d_keep; pa.out_est = (long long*)out->d_est_us; pa.out_perm = out->d_perm;
    pa.out_kept_idx = out->d_kept_idx; pa.kept_base = kept_base; pa.seg_kept = seg_kept;
    int wrc = launch_policy_walk(pa, sms, stream);
    if (wrc != PARD_OK) return wrc;
    launch_pdl(k_kept_scan, 1, 1024, 0, stream, seg_kept, L.n_seg, kept_base, chunk_base, out->d_seg_kept,
               (unsigned long long*)out->d_n_kept);
    return launch_policy_emit(pa, stream);
  };

  /* queue boundaries, and for the planner's own rule the window tables and output offsets; id_bits > 8:
   * the boundaries are searched, never read off the digit counts */
  auto launch_windows = [&](bool tables, uint32_t local_candidate, uint32_t id_bits = 64u, bool direct = false) {
    if (many_short_queues(n, L.n_seg))
      launch_pdl(k_windows_many, L.n_seg / (kWinThreads - 1u) + 1, kWinThreads, 0, stream, hdr, (const unsigned long long*)buf_a,
                 (const unsigned long long*)buf_b, n32, ibits, L.n_seg, (const PardSegConst*)ktab, seg_off, out->d_seg_offsets,
                 win_off, win_cnt, wtab, L.win_capacity, (mode & PARD_MODE_SCAN) ? 1u : 0u, tables ? 1u : 0u,
                 (mode & PARD_MODE_RAW) ? 1u : 0u, seg_kept, kept_base, chunk_base, out->d_seg_kept,
                 (unsigned long long*)out->d_n_kept, direct ? 1u : 0u);
    else
      launch_pdl(k_windows, L.n_seg / kWinQueues + 1, kWinThreads, 0, stream, hdr, (const unsigned long long*)buf_a,
               (const unsigned long long*)buf_b, n32, ibits, L.n_seg, (const PardSegConst*)ktab, seg_off, out->d_seg_offsets, win_off,
               win_cnt, wtab, L.win_capacity, (mode & PARD_MODE_SCAN) ? 1u : 0u, (const uint32_t*)hist, id_bits, local_candidate,
               tables ? 1u : 0u, (mode & PARD_MODE_RAW) ? 1u : 0u, seg_kept, kept_base, chunk_base, out->d_seg_kept,
               (unsigned long long*)out->d_n_kept, direct ? 1u : 0u);
  };

  auto const_args = [&]() {
    ConstArgs ca = {};
    ca.pipes = pipe_table; ca.st = *state; ca.n_pipelines = n_pipelines; ca.n_ctx = n_ctx; ca.ktab = ktab;
    ca.sbits = sbits; ca.ibits = ibits; ca.key_sbits = sbits; ca.win_off = win_off; ca.win_cnt = win_cnt;
    return ca;
  };

  /* ---- keys wider than one sort element: see k_wide_reset.  Run only when a finished call has
   * reported that width (the host cannot know the deadline span beforehand), hence not for
   * PARD_MODE_NOWAIT, whose caller gets PARD_ERANGE from pard_plan_status as before. ---- */
  auto plan_wide = [&]() -> int {
    uint32_t h_wide = 0;
    PARD_CUDA_OK(cudaMemcpyAsync(&h_wide, &hdr->wide, 4, cudaMemcpyDeviceToHost, stream));
    PARD_CUDA_OK(cudaStreamSynchronize(stream));
    if (!h_wide) return PARD_ERANGE;
    const uint32_t grid_n = (uint32_t)std::min<uint64_t>((n + 255) / 256, (uint64_t)sms * 8);
    {
      const unsigned long long n16 = L.zero_end / 16;
      launch_pdl(k_clear, (uint32_t)std::min<unsigned long long>((n16 + 255) / 256, (unsigned long long)sms * 4), 256, 0,
                 stream, (uint4*)(ws + L.hdr), n16);
    }
    ConstArgs ca = const_args();
    launch_prepass(req4, n32, n_ctx, S, ctx_dmin, ctx_dmax, hdr, 0u, ca, sms, stream);
    launch_pdl(k_ctx_span, (n_ctx + 255) / 256, 256, 0, stream, ctx_dmin, ctx_dmax, n_ctx, hdr);
    launch_pdl(k_key_width, 1, 1, 0, stream, sbits, ibits, hdr, 0u, sbits, 1u);
    launch_pdl(k_seg_const, n_ctx, kConstThreads, 0, stream, ca, (const unsigned long long*)ctx_dmin, (const unsigned long long*)ctx_dmax, hdr);
    const uint32_t cw = 64 - ibits;                         /* key bits per super-pass */
    const uint32_t supers = (sbits + 60 + cw - 1) / cw;     /* for the widest legal span; chunks beyond the key are empty */
    const uint32_t chunk_passes = std::min<uint32_t>(kMaxPasses, (cw + 7) / 8);
    uint32_t* order = kept_tmp;
    const uint32_t stall = (mode & PARD_MODE_TEST_STALL) ? 1u : 0u;
    for (uint32_t sp = 0; sp < supers; ++sp) {
      launch_pdl(k_wide_reset, (uint32_t)std::min<uint64_t>((lb_words + kMaxPasses * kBins + 255) / 256, (uint64_t)sms * 4), 256,
                 0, stream, hdr, hist, lookback, (unsigned long long)lb_words, sbits, ibits, sp);
      launch_pdl(k_wide_pack, grid_n, 256, 0, stream, req4, n32, n_ctx, S, ctx_dmin, ctx_dmax, state->d_priority, sbits, ibits,
                 sp, (const PlanHeader*)hdr, (const uint32_t*)order, buf_a, hist);
      if (L.small_tiles)
        launch_pdl(k_sort_rest<false, true>, std::min<uint32_t>(L.sort_tiles, 2u * (uint32_t)sms), kSortThreads, sizeof(SortSmem), stream, 0u,
                   hdr, buf_a, buf_b, (const uint32_t*)hist, lookback, lb_words, n32, ibits, stall, 0u, CtxTiles{}, WinCountArgs{}, L.geometry);
      else
        for (uint32_t p = 0; p < chunk_passes; ++p)
          launch_pdl(k_sort_pass<false>, L.sort_tiles, kSortThreads, sizeof(SortSmem), stream, p, hdr, buf_a, buf_b, hist,
                     lookback + (p & 1) * lb_words, lookback + ((p + 1) & 1) * lb_words, n32, ibits, p == 0 ? stall : 0u, 0u, CtxTiles{}, WinCountArgs{});
      launch_pdl(k_wide_chase, grid_n, 256, 0, stream, (const PlanHeader*)hdr, (const unsigned long long*)buf_a, buf_b, n32,
                 ibits, sp, (const uint32_t*)order);
      launch_pdl(k_wide_keep, grid_n, 256, 0, stream, (const PlanHeader*)hdr, (const unsigned long long*)buf_a,
                 (const unsigned long long*)buf_b, n32, order);
    }
    launch_pdl(k_wide_final, grid_n, 256, 0, stream, req4, n32, n_ctx, S, sbits, ibits, hdr, (const uint32_t*)order, buf_a);
    launch_pdl(k_wide_done, 1, 1, 0, stream, hdr, sbits);
    launch_windows(false, 0u, sbits);
    PolicyArgs pa = {};
    pa.hdr = hdr; pa.buf_a = buf_a; pa.buf_b = buf_b;
    pa.n = n32; pa.ibits = ibits; pa.n_seg = L.n_seg; pa.mode = mode;
    pa.ktab = ktab; pa.seg_off = seg_off; pa.req = req4; pa.arrivals = d_arrivals;
    pa.pipes = pipe_table; pa.n_pipelines = n_pipelines; pa.st = *state;
    const int wrc = decide_by_walk(pa);
    if (wrc != PARD_OK) return wrc;
    return pard_plan_status(d_workspace, cuda_stream);
  };

  /* ---- a block per ctx does everything (pard_local.cu): a single ctx within one tile, or the
   * caller's word that the requests come grouped by ctx with no ctx beyond a tile ---- */
  const bool local_single = local_sure && !rule_walk;
  if (local_single || ((mode & PARD_MODE_GROUPED) && n_ctx > 1 && n > 0 && !rule_walk && !L.ctx_passes)) {
    LocalArgs la = {};
    la.req = req4; la.ctx_start = local_single ? nullptr : ctx_start;
    la.n = n32; la.n_ctx = n_ctx; la.ibits = ibits; la.force_scan = (mode & PARD_MODE_SCAN) ? 1u : 0u;
    la.pipes = pipe_table; la.n_pipelines = n_pipelines; la.st = *state;
    la.out_keep = out->d_keep; la.out_est = (long long*)out->d_est_us; la.out_perm = out->d_perm;
    la.out_kept_idx = out->d_kept_idx; la.out_n_kept = (unsigned long long*)out->d_n_kept;
    la.out_seg_off = out->d_seg_offsets; la.out_seg_kept = out->d_seg_kept;
    la.ktab = ktab; la.kept_words = (uint32_t*)ctx_dmin; la.kept_tmp = out->d_kept_idx ? kept_tmp : nullptr;
    const bool answered = local_single && !(mode & PARD_MODE_NOWAIT);
    if (answered) la.answer = pard_report_ticket();
    if (!local_single) {
      launch_pdl(k_clear, std::min<uint32_t>((n_ctx + 1023) / 1024 + 1, (uint32_t)sms), 256, 0, stream, (uint4*)(ws + L.hdr),
                 (unsigned long long)((L.ctx_dmin + 4ull * n_ctx + 15) / 16));
      rc = launch_ctx_prep(la, ktab, ctx_start, hdr, stream);
      if (rc != PARD_OK) return rc;
    }
    rc = launch_plan_local(la, hdr, (mode & PARD_MODE_RAW) != 0, stream);
    if (rc != PARD_OK) return rc;
    while (phase <= PARD_N_PHASES) mark();             /* the phases are those of the other path: all of this counts as the first */
    PARD_CUDA_OK(cudaGetLastError());
    if (mode & PARD_MODE_NOWAIT) return PARD_OK;
    rc = answered ? pard_report_wait(la.answer, &hdr->status, stream, nullptr) : pard_plan_status(d_workspace, cuda_stream);
    return rc == PARD_ERANGE ? plan_wide() : rc;
  }

  /* Requests grouped by ctx (the caller's word) with contexts of more than a tile on average: the
   * radix passes stay inside every ctx's range -- tiles cut at ctx boundaries, digit counts per
   * ctx, look-back up to the ctx's first tile -- and sort the stage and deadline bits only; the
   * ctx bits of the key need no pass (C5: four passes instead of five).  Needs the stage in the low
   * bits of the queue id: stage_stride a power of two. */
  const bool ctx_sort = (mode & PARD_MODE_GROUPED) && L.ctx_passes && (S & (S - 1)) == 0 && !rule_walk && n > 0;

  /* ---- such requests may stand in order already: planned without a sort if they do (pard_direct.cuh).  2^24 requests of 256 contexts in order 345 -> 232 us,
   * 288 k of 24 contexts 71 -> 51.  Out of order the try cost 7 of 568 us, 2 of 71; the tiles of the passes behind it on
   * their way into L2 brought that to 544 and 74, at which it stands (k_decide_rest).  In order, but with a constant that the path does not take, 608 -> 609 and 70 -> 74.
   * The path itself would take any stride up to 16 (12 stages: 243 us, by the general sort 434); but the kernels of that sort would have to look,
   * ahead of their first loads, whether the plan is made, and every other call of theirs paid 0.7 us for it.  Without the
   * caller's word a call would pay 8 to 11 us, of 85 to 210, for finding out that its contexts come mixed. ---- */
  DirectArgs da = {};
  const bool direct = ctx_sort && !(mode & (PARD_MODE_RAW | PARD_MODE_SCAN)) &&
                      !state->d_priority && dir_layout(n, n_ctx, S, sms, (char*)buf_b, &da);
  da.req = req4; da.n = n32; da.n_ctx = n_ctx; da.S = S; da.sbits = sbits; da.ibits = ibits;
  da.ktab = ktab; da.ctx_start = ctx_start; da.const_bad = kept_tmp; da.stall = (mode & PARD_MODE_TEST_STALL) ? 1u : 0u;

  /* ---- clear the scratch that must start at zero: one contiguous region ---- */
  if (!direct) {
    const unsigned long long n16 = (n > 0 ? L.zero_end : L.lookback) / 16;   /* offsets are multiples of 256 */
    launch_pdl(k_clear, (uint32_t)std::min<unsigned long long>((n16 + 255) / 256, (unsigned long long)sms * 4), 256, 0,
               stream, (uint4*)(ws + L.hdr), n16);
  }

  const uint32_t key_sbits = ctx_sort ? ceil_log2(S) : sbits;
  const CtxTiles ctx_tiles = {ctx_start, (const uint32_t*)(ws + L.tile_first), (const uint32_t*)(ws + L.hist_ctx), n_ctx};
  /* few queues, decided by the planner's own rule in budget order from the start of every queue:
   * the window tables are counted while the requests are packed */
  const bool win_hist = n > 0 && L.n_seg <= kHistSegs && !rule_walk && !state->d_priority && !local_cand && !ctx_sort;
  ConstArgs ca = const_args();
  ca.key_sbits = key_sbits;
  ca.with_key_width = n_ctx <= kFoldCtx ? 1u : 0u;       /* few contexts: the last block to finish finds the key width */
  ca.arrival_order = arrival_order ? 1u : 0u; ca.win_hist = win_hist ? 1u : 0u; ca.force_scan = (mode & PARD_MODE_SCAN) ? 1u : 0u;
  /* known paths: the paths' sums are written down beside the constants, in the survivors' scratch, where
   * they fit (queues of 32 requests on average); else blocks work them out again (stage_paths) */
  ca.path_sums = (mode & PARD_MODE_PATH_MASK) && n >= 2ull * kMaskPaths * L.n_seg ? (long long*)kept_tmp : nullptr;
  const bool const_fold = n > 0 && L.n_seg <= kFoldSegs && ca.with_key_width;
  /* arrival order, a queue id of one digit: sorted straight from the requests (k_sort_requests) */
  const bool from_requests = arrival_order && L.n_seg > 1 && L.n_seg <= kCountSegs && !local_cand && n > 0;
  const bool with_rounds = from_requests && !(mode & (PARD_MODE_CLIPPER | PARD_MODE_PATH_MASK));
  if (direct) {
    const unsigned long long n16 = L.zero_end / 16;
    const uint32_t range_blocks = (n_ctx + kDirWarps - 1) / kDirWarps;
    launch_pdl(k_dir_begin, n_ctx + range_blocks + (uint32_t)std::min<unsigned long long>((n16 + 255) / 256, (unsigned long long)sms * 4), kDirThreads, 0,
               stream, da, ca, (uint4*)(ws + L.hdr), n16, range_blocks);
  }
  mark();
  if (direct)
    launch_pdl(S > 8 ? k_dir_count<4> : k_dir_count<3>, da.n_pieces, kDirThreads, 0, stream, da, ca, hdr, ctx_dmin, ctx_dmax);
  if (n > 0 && !direct) launch_prepass(req4, n32, n_ctx, S, ctx_dmin, ctx_dmax, hdr, const_fold ? n_ctx : 0u, ca, sms, stream, from_requests ? hist : nullptr);
  mark();
  if (!ca.with_key_width) {
    if (n > 0) launch_pdl(k_ctx_span, (n_ctx + 255) / 256, 256, 0, stream, ctx_dmin, ctx_dmax, n_ctx, hdr);
    launch_pdl(k_key_width, 1, 1, 0, stream, sbits, ibits, hdr, arrival_order ? 1u : 0u, key_sbits, state->d_priority ? 1u : 0u);
  }
  if (!const_fold && direct)
    launch_pdl(k_seg_finish, (L.n_seg + 1023) / 1024 + 1, 1024, 0, stream, ca, (const unsigned long long*)ctx_dmin, (const unsigned long long*)ctx_dmax, hdr,
               (const uint32_t*)ctx_start, (uint32_t*)(ws + L.tile_first));
  else if (!const_fold)
    launch_pdl(k_seg_const, n_ctx, kConstThreads, 0, stream, ca, (const unsigned long long*)ctx_dmin, (const unsigned long long*)ctx_dmax, hdr);
  if ((local_cand && !local_sure) || (ctx_sort && !direct))
    launch_pdl(k_ctx_ranges, (n_ctx + 1 + 7) / 8, 256, 0, stream, req4, n32, n_ctx, ctx_start, hdr);
  if (ctx_sort && (const_fold || !direct)) launch_pdl(k_tile_table, 1, 1024, 0, stream, (const uint32_t*)ctx_start, n_ctx, (uint32_t*)(ws + L.tile_first), (const PlanHeader*)hdr);
  mark();
  if (direct) {
    const DirScanOut scan_out = {seg_off, out->d_seg_offsets, seg_kept, kept_base, chunk_base, out->d_seg_kept, (unsigned long long*)out->d_n_kept};
    launch_pdl(k_dir_scan, n_ctx, kDirScanThreads, 0, stream, da, hdr, scan_out);
    launch_pdl(S > 8 ? k_dir_emit<4> : k_dir_emit<3>, std::min<uint32_t>(da.n_pieces, (uint32_t)sms * 4), kDirThreads, sizeof(EmitSmem), stream,
               da, hdr, (const uint32_t*)seg_off, (const uint32_t*)kept_base, out->d_keep, (long long*)out->d_est_us, out->d_perm,
               out->d_kept_idx);
  }
  if (local_cand)                                /* every ctx inside one tile: sorted block by block, straight from the requests */
    launch_pdl(k_sort_local, n_ctx, kSortThreads, sizeof(SortSmem), stream, hdr, local_cand, req4, ctx_dmin, ctx_dmax,
               state->d_priority, buf_a, buf_b, local_sure ? (const uint32_t*)nullptr : (const uint32_t*)ctx_start, n32, S,
               ceil_log2(S), ibits);
  if (ctx_sort) {
    launch_pdl(k_pack_ctx, L.ctx_tiles, 256, 0, stream, req4, S, ctx_dmin, ctx_dmax, state->d_priority, ibits, hdr, buf_a,
               (uint32_t*)(ws + L.hist_ctx), ctx_tiles);
  } else if (from_requests) {
    /* (by the sort below) */
  } else if (n > 0 && !local_sure) {             /* returns at once when the blocks above did the work */
    /* every block adds its digit counts to the call's, up to 256 additions per pass: the fewer blocks the
     * better, down to two per multiprocessor and up to the four that are resident (a million requests with 1,184
     * blocks: 7 us more; 2^24: 3 us more) */
    const uint64_t blocks = std::min<uint64_t>(std::max<uint64_t>(n / 4096, 2ull * sms), 4ull * sms);
    const uint32_t grid = (uint32_t)std::min<uint64_t>((n + 255) / 256, blocks);
    launch_pdl(win_hist ? k_pack<true> : k_pack<false>, grid, 256, 0, stream, req4, n32, n_ctx, S, ctx_dmin, ctx_dmax,
               state->d_priority, ibits, hdr, buf_a, hist, local_cand, (const PardSegConst*)ktab, (const uint32_t*)win_off,
               (const uint32_t*)win_cnt, whist);
  }
  /* passes with a launch of their own, then the rest in one kernel (see k_sort_rest) */
  const uint32_t sort_tiles = ctx_sort ? L.ctx_tiles : L.sort_tiles;
  /* the passes that the widest possible key needs; in arrival order the key is the queue id alone (see
   * set_key_width), so that no launch turns out empty (three of them, 11 us a call at 2^24) */
  const uint32_t max_passes = arrival_order ? (key_sbits + 7) / 8
                            : ctx_sort ? std::min<uint32_t>(kMaxPasses, (key_sbits + 60 + 7) / 8) : L.max_passes;
  const bool small = L.small_tiles && !ctx_sort;
  const uint32_t own_passes = small || local_cand ? 0u : std::min(kOwnPasses, max_passes);
  const uint32_t rest_grid = std::min<uint32_t>(sort_tiles, 2u * (uint32_t)sms);
  const uint32_t stall = (mode & PARD_MODE_TEST_STALL) && !ctx_sort ? 1u : 0u;
  WinCountArgs wc = {};
  wc.on = win_hist ? 1u : 0u; wc.n_seg = L.n_seg; wc.raw = (mode & PARD_MODE_RAW) ? 1u : 0u; wc.sbits = sbits;
  wc.ktab = ktab; wc.whist = whist; wc.win_off = win_off; wc.win_cnt = win_cnt; wc.wtab = wtab;
  wc.seg_off = seg_off; wc.out_seg_off = out->d_seg_offsets; wc.seg_kept = seg_kept; wc.out_seg_kept = out->d_seg_kept;
  wc.kept_base = kept_base; wc.out_n_kept = (unsigned long long*)out->d_n_kept; wc.hist = hist;
  for (uint32_t p = 0; p < (uint32_t)kMaxPasses; ++p) {
    mark();
    if (n == 0 || local_sure || p >= max_passes) continue;
    if (from_requests) {                                   /* (one pass: max_passes is 1) */
      const RequestPass rp = {req4, ctx_dmin, n_ctx, S, (mode & PARD_MODE_NEXUS) ? 1u : 0u, ktab, with_rounds ? (uint32_t*)buf_a : nullptr};
      launch_pdl(small ? k_sort_requests<true> : k_sort_requests<false>, sort_tiles, kSortThreads, sizeof(SortSmem), stream, hdr, buf_a, buf_b,
                 (const uint32_t*)hist, lookback, lookback + lb_words, n32, ibits, stall, L.geometry, rp);
    } else if (p < own_passes)
      launch_pdl(ctx_sort ? k_sort_pass<true> : k_sort_pass<false>, sort_tiles + wc.on, kSortThreads, sizeof(SortSmem), stream, p, hdr, buf_a,
                 buf_b, hist, lookback + (p & 1) * lb_words, lookback + ((p + 1) & 1) * lb_words, n32, ibits, p == 0 ? stall : 0u,
                 local_cand, ctx_tiles, wc);
    else if (p == own_passes)
      launch_pdl(ctx_sort ? k_sort_rest<true, false> : small ? k_sort_rest<false, true> : k_sort_rest<false, false>, rest_grid + wc.on, kSortThreads, sizeof(SortSmem), stream, p, hdr, buf_a,
                 buf_b, hist, lookback, lb_words, n32, ibits, stall, local_cand, ctx_tiles, wc, L.geometry);
    wc.on = 0;                                             /* the first launch has done it */
  }
  mark();
  if (win_hist) {
    /* boundaries and tables are there already */
  } else {
    launch_windows(!rule_walk, local_cand, ctx_sort ? 64u : sbits, direct);
  }
  if (n > 0 && rule_walk) {
    /* a rule without rising thresholds: every queue is walked in order (pard_policy.cu) */
    PolicyArgs pa = {};
    pa.hdr = hdr; pa.buf_a = buf_a; pa.buf_b = buf_b;
    pa.n = n32; pa.ibits = ibits; pa.n_seg = L.n_seg; pa.mode = mode;
    pa.ktab = ktab; pa.seg_off = seg_off; pa.req = req4; pa.arrivals = d_arrivals;
    pa.pipes = pipe_table; pa.n_pipelines = n_pipelines; pa.st = *state; pa.path_sums = ca.path_sums;
    pa.rounds_there = with_rounds ? 1u : 0u;
    mark();
    rc = decide_by_walk(pa);
    if (rc != PARD_OK) return rc;
  } else if (n > 0) {
    long long* est = (long long*)out->d_est_us;
    const bool raw = mode & PARD_MODE_RAW;
    uint32_t* tmp = out->d_kept_idx ? kept_tmp : nullptr;
    /* window tables, and the decision from them */
    mark();
    const uint32_t win_grid = (uint32_t)((n + (uint64_t)kDecTile - 1) / kDecTile);
    auto decide_win = raw ? (state->d_priority ? k_decide_win<true, true> : k_decide_win<true, false>)
                          : (state->d_priority ? k_decide_win<false, true> : k_decide_win<false, false>);
    /* the survivors go straight to their place in the output */
    if (direct)
      launch_pdl(k_decide_rest, std::min<uint32_t>(win_grid, kRestRounds * kRestBlocks * (uint32_t)sms), kDecThreads, 0, stream, hdr, buf_a, buf_b, n32, ibits, ktab, seg_off,
                 win_off, win_cnt, wtab, out->d_keep, est, out->d_perm, out->d_kept_idx, (const uint32_t*)kept_base);
    else
      launch_pdl(decide_win, win_grid, kDecThreads, 0, stream, hdr, buf_a, buf_b, n32, ibits, ktab, seg_off, win_off, win_cnt, wtab,
                 out->d_keep, est, out->d_perm, out->d_kept_idx, (const uint32_t*)kept_base);
    /* fallback when a queue has too many batch windows: the same decision by scanning, one kernel
     * that returns at once otherwise */
    const uint32_t scan_grid = std::min<uint32_t>(L.dec_tiles, (uint32_t)sms * 2);
    launch_pdl(raw ? k_scan_path<true> : k_scan_path<false>, scan_grid, kDecThreads, 0, stream, hdr, buf_a, buf_b, n32, ibits,
               L.n_seg, ktab, seg_off, win_off, tile_agg, tile_carry, out->d_keep, est, out->d_perm, tmp, seg_kept, kept_base,
               chunk_base, out->d_seg_kept, (unsigned long long*)out->d_n_kept, out->d_kept_idx,
               (mode & PARD_MODE_TEST_STALL) ? 1u : 0u);
  }
  if (n == 0) mark();
  mark();
  if (n == 0)                                      /* an empty call still owes its zeros */
    launch_pdl(k_kept_scan, 1, 1024, 0, stream, seg_kept, L.n_seg, kept_base, chunk_base, out->d_seg_kept,
               (unsigned long long*)out->d_n_kept);
  mark();
  PARD_CUDA_OK(cudaGetLastError());
  if (mode & PARD_MODE_NOWAIT) return PARD_OK;
  rc = pard_plan_status(d_workspace, cuda_stream);
  return (rc == PARD_ERANGE && n > 0) ? plan_wide() : rc;
}

extern "C" int pard_plan_status(const void* d_workspace, void* cuda_stream) {
  if (!d_workspace) return PARD_EINVAL;
  return pard_wait_status(&((const PlanHeader*)d_workspace)->status, (cudaStream_t)cuda_stream);
}

extern "C" int pard_plan_kernel_launches(uint64_t n, uint32_t n_ctx, int32_t stage_stride,
                                         uint32_t* launches) {
  uint64_t bytes;
  if (!launches) return PARD_EINVAL;
  int rc = pard_plan_workspace_bytes(n, n_ctx, stage_stride, &bytes);
  if (rc != PARD_OK) return rc;
  /* For the planner's own rule without priorities and without PARD_MODE_GROUPED.  One ctx of at
   * most a sort tile: one kernel.  Else always clear, and seg_const (few queues: inside the
   * prepass); with many contexts also key_width (and, when n > 0, ctx_span); when n > 0: prepass, pack, the radix passes, decide_win
   * and the scan path (one kernel that returns at once); with more than 64 queues also the
   * queue boundaries and the searched window tables (windows). */
  const uint64_t n_seg = (uint64_t)n_ctx * (uint64_t)stage_stride;
  const uint32_t width_kernels = n_ctx <= kFoldCtx ? 0 : 1;     /* key_width (+ ctx_span when n > 0) */
  const uint32_t const_kernels = n > 0 && n_seg <= kFoldSegs ? 0 : 1;   /* seg_const, unless the prepass does its work */
  const bool local_cand = local_sort_candidate(n, n_ctx);
  const uint32_t local_kernels = local_cand ? 2 : 0;            /* ctx_ranges, sort_local */
  const Layout L = make_layout(n, n_ctx, stage_stride);
  const uint32_t own = L.small_tiles || local_sort_candidate(n, n_ctx) ? 0u : std::min(kOwnPasses, L.max_passes);
  const uint32_t passes = own + (own < L.max_passes ? 1 : 0);   /* and the kernel that does the rest */
  if (n_ctx == 1 && n > 0 && n <= (uint64_t)kSortTile) *launches = 1;
  else if (n == 0) *launches = 4 + width_kernels;               /* clear, (key_width,) seg_const, windows, kept_scan */
  else *launches = 1 + const_kernels + 2 * width_kernels + 2 + local_kernels + passes + 2 + (n_seg <= kHistSegs && !local_cand ? 0 : 1);
  return PARD_OK;
}

extern "C" int pard_profile_begin(uint32_t every, uint32_t max_samples) {
  const bool coarse = (every & PARD_PROFILE_COARSE) != 0;
  every &= ~PARD_PROFILE_COARSE;
  if (every < 1 || max_samples < 1 || max_samples > 65536) return PARD_EINVAL;
  std::lock_guard<std::mutex> lock(g_prof.mu);
  if (g_prof.on.load()) return PARD_EINVAL;
  try {
    g_prof.ev.assign((size_t)max_samples * kEventsPerSample, nullptr);
  } catch (const std::bad_alloc&) {
    return PARD_ENOMEM;
  }
  for (auto& e : g_prof.ev)
    if (cudaEventCreate(&e) != cudaSuccess) {
      for (auto& f : g_prof.ev) if (f) cudaEventDestroy(f);
      g_prof.ev.clear();
      return PARD_ECUDA;
    }
  g_prof.every = every;
  g_prof.coarse = coarse;
  g_prof.max_samples = max_samples;
  g_prof.calls = 0;
  g_prof.n_samples = 0;
  g_prof.last = nullptr;
  g_prof.on.store(true, std::memory_order_release);
  return PARD_OK;
}

extern "C" int pard_profile_end(float* ms_sum, uint32_t* n_samples) {
  std::lock_guard<std::mutex> lock(g_prof.mu);
  if (!g_prof.on.load()) return PARD_EINVAL;
  int rc = PARD_OK;
  if (ms_sum) for (int i = 0; i < PARD_N_PHASES; ++i) ms_sum[i] = 0.f;
  for (uint32_t s = 0; s < g_prof.n_samples; ++s) {
    cudaEvent_t* e = g_prof.ev.data() + (size_t)s * kEventsPerSample;
    if (cudaEventSynchronize(e[PARD_N_PHASES]) != cudaSuccess) { rc = PARD_ECUDA; break; }
    for (int i = 0; i < PARD_N_PHASES && ms_sum; ++i) {
      float ms = 0.f;
      int to = i + 1;
      if (g_prof.coarse && i == kPhaseTables) to = PARD_N_PHASES;       /* the decision pass as one phase */
      if (g_prof.coarse && i > kPhaseTables) continue;
      if (cudaEventElapsedTime(&ms, e[i], e[to]) != cudaSuccess) rc = PARD_ECUDA;
      ms_sum[i] += ms;
    }
  }
  if (n_samples) *n_samples = g_prof.n_samples;
  for (auto& e : g_prof.ev) cudaEventDestroy(e);
  g_prof.ev.clear();
  g_prof.last = nullptr;
  g_prof.on.store(false, std::memory_order_release);
  return rc;
}

extern "C" const char* pard_profile_phase_name(uint32_t phase) {
  static const char* names[PARD_N_PHASES] = {"clear", "prepass", "segments", "pack", "sort0", "sort1",
                                              "sort2", "sort3", "sort4", "sort5", "sort6", "sort7",
                                              "tables", "decide", "compact"};
  return phase < PARD_N_PHASES ? names[phase] : "";
}
