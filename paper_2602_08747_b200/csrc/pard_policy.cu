/* Decision rules that need a sequential walk of every queue.
 *
 * The planner's own rule in budget order has thresholds that only rise along a queue, which
 * turns the Request Broker's loop into a prefix minimum (pard_plan.cu).  That no longer holds
 *   - when requests carry the downstream path they will take (Sec. 5.2, dynamic-path DAGs):
 *     L_sub, and with it the threshold, differs from request to request;
 *   - in arrival order (Table 1 and Sec. 5.3, PARD-FCFS);
 *   - for Clipper++'s per-module share of the objective (Sec. 5.1, Baseline), arrival order;
 *   - for Nexus' window scan (Sec. 5.1, Baseline), a rule of its own.
 * For the first three the loop is  x <- x + [x < u_r]  with x the admitted count and u_r a multiple
 * of the batch round's size: u_r = cap * v_r, v_r the number of rounds r still fits.  So r is
 * admitted iff floor(x / cap) < v_r, and while one round fills up -- until cap more requests are
 * admitted -- the test is the same for every request: v_r > b, b the number of the round.  A walk
 * is therefore a chain of rounds, not of requests: in round b, count the requests with v_r > b
 * until there are cap of them, which any number of threads can do side by side.  Nexus' scan has
 * the same shape (find the first cap consecutive requests with v_r > b).
 *   k_policy_terms   every request on its own: v_r                                -> T[n]; calls in arrival order
 *                    that look no further than the deadline have it from their sort (k_sort_requests)
 *   k_policy_walk    a group of threads per queue (16 requests each and step) closes round after
 *                    round; round b's end goes to C[first position of the queue + b]
 *   k_policy_emit    every request on its own again: its round by a search in the ends, estimate,
 *                    decision, survivors straight to their final place
 * T and C live in the sort buffer that does not hold the elements.
 * Nexus on 16 queues of 2^20 requests: the walk takes 0.053 ms by clusters of eight blocks (0.080 by one block,
 * 0.093 without copies ahead) where one warp per queue, 32 requests per step, took 23.8 ms; a call of 2^24
 * requests 452 -> 402 us, 309 since the sort takes the requests themselves and k_policy_emit eight in a row. */
#include <type_traits>

#include "pard_plan_internal.cuh"

using namespace pard_plan_detail;

namespace {

constexpr int kPolThreads = 128;
constexpr int kPolItems = 8;
constexpr int kPolTile = kPolThreads * kPolItems;
constexpr int kStageSegs = 16;           /* queues whose path sums a block keeps in shared memory */

struct SortedView {
  const unsigned long long* src;
  uint32_t* T;
  uint32_t* C;
  uint32_t kshift, imask;
  unsigned long long dmask;
};

__device__ __forceinline__ SortedView sorted_view(const PolicyArgs& a) {
  SortedView v;
  const bool odd = a.hdr->npass & 1;
  v.src = odd ? a.buf_b : a.buf_a;
  uint32_t* spare = reinterpret_cast<uint32_t*>(odd ? a.buf_a : a.buf_b);
  v.T = spare;
  v.C = spare + a.n;                     /* 8 bytes per request: two 32-bit arrays */
  v.kshift = a.ibits + a.hdr->dbits;
  v.imask = (1u << a.ibits) - 1;
  v.dmask = a.hdr->dbits >= 64 ? ~0ull : ((1ull << a.hdr->dbits) - 1);
  return v;
}

__device__ __forceinline__ const PardPipeDev* pipe_of(const PolicyArgs& a, uint32_t c) {
  int32_t pi = a.st.d_pipeline_of_ctx ? a.st.d_pipeline_of_ctx[c] : 0;
  if (pi < 0 || (uint32_t)pi >= a.n_pipelines) pi = 0;          /* reported by k_seg_const */
  return a.n_pipelines <= (uint32_t)kFewPipelines ? a.pipes.few[pi] : a.pipes.many[pi];
}

/* sum over the path in slot `s` of q_i + d_i(B_i), plus w of the slot (Eq. 3, State Planner part) */
__device__ long long path_sum(const PolicyArgs& a, const PardPipeDev* p, uint32_t c, int32_t s) {
  const uint32_t S = (uint32_t)a.st.stage_stride;
  long long acc = a.st.d_w_us ? a.st.d_w_us[(size_t)c * a.st.slot_stride + s] : 0;
  for (int32_t e = p->path_off[s]; e < p->path_off[s + 1]; ++e) {
    const int32_t i = p->path_stage[e];
    int32_t Bi = a.st.d_batch[(size_t)c * S + i];
    if (Bi < 1 || Bi > p->bmax[i]) Bi = 1;                      /* reported by k_seg_const */
    acc += a.st.d_q_us[(size_t)c * S + i] + p->lat_us[p->lat_offsets[i] + Bi - 1];
  }
  return acc;
}

/* Path sums of the first kStageSegs queues a block's tile touches, kept in shared memory. */
struct StagedPaths {
  long long sum[kStageSegs][kMaskPaths];
  int32_t n_paths[kStageSegs];
  uint32_t seg0;
};

__device__ void stage_paths(const PolicyArgs& a, const SortedView& v, uint64_t tile0, StagedPaths& sp) {
  const uint32_t S = (uint32_t)a.st.stage_stride;
  const uint64_t end = tile0 + kPolTile < a.n ? tile0 + kPolTile : a.n;
  const uint32_t seg0 = (uint32_t)(v.src[tile0] >> v.kshift);
  const uint32_t segs = (uint32_t)(v.src[end - 1] >> v.kshift) - seg0 + 1;
  if (threadIdx.x == 0) sp.seg0 = seg0;
  for (uint32_t t = threadIdx.x; t < min(segs, (uint32_t)kStageSegs) * kMaskPaths; t += blockDim.x) {
    const uint32_t q = t / kMaskPaths, j = t % kMaskPaths, seg = seg0 + q;
    if (seg >= a.n_seg) { if (j == 0) sp.n_paths[q] = 0; continue; }
    const uint32_t c = seg / S, k = seg % S;
    const PardPipeDev* p = pipe_of(a, c);
    int32_t np = 0;
    if (k < (uint32_t)p->n_stages) {
      const int32_t s0 = p->stage_slot_off[k];
      np = p->stage_slot_off[k + 1] - s0;
      if ((int32_t)j < np) sp.sum[q][j] = path_sum(a, p, c, s0 + (int32_t)j);
    }
    if (j == 0) sp.n_paths[q] = np;
  }
  __syncthreads();
}

/* The downstream estimate of a request whose path is known: the maximum over the paths its mask
 * names; K.lsub when the mask names none of the stage's (input error) or the stage is a sink. */
__device__ __noinline__ long long masked_lsub(const PolicyArgs& a, const StagedPaths& sp, uint32_t seg, uint32_t flags,
                                 const PardSegConst& K) {
  const uint32_t q = seg - sp.seg0;
  long long best = -1;
  int32_t np;
  if (q < (uint32_t)kStageSegs) {
    np = sp.n_paths[q];
    for (int32_t j = 0; j < np && j < kMaskPaths; ++j)
      if ((flags >> j) & 1u) best = sp.sum[q][j] > best ? sp.sum[q][j] : best;
  } else {                                       /* a queue beyond the staged ones: straight from the tables */
    const uint32_t S = (uint32_t)a.st.stage_stride, c = seg / S, k = seg % S;
    const PardPipeDev* p = pipe_of(a, c);
    const int32_t s0 = p->stage_slot_off[k];
    np = p->stage_slot_off[k + 1] - s0;
    for (int32_t j = 0; j < np && j < kMaskPaths; ++j)
      if ((flags >> j) & 1u) {
        const long long v = path_sum(a, p, c, s0 + j);
        best = v > best ? v : best;
      }
  }
  if (np <= 0) return K.lsub;                    /* a sink has nothing downstream whatever the mask says */
  if (best < 0) { set_status(a.hdr, PARD_EDATA); return K.lsub; }   /* the mask names no path of this stage */
  return best;
}

/* The same from the sums written down beside the queue's constants.  (A request mostly names one path or two: their
 * loads do not wait for each other, nor those of several requests.) */
__device__ __forceinline__ long long masked_lsub_at_hand(const PolicyArgs& a, uint32_t seg, uint32_t flags, long long lsub) {
  const long long* t = a.path_sums + (size_t)seg * kMaskPaths;
  const uint32_t rest = flags & (flags - 1);
  const long long one = __ldg(t + __ffs((int)flags) - 1), two = rest ? __ldg(t + __ffs((int)rest) - 1) : -1ll;
  long long best = one > two ? one : two;
  for (uint32_t m = rest & (rest - 1); m; m &= m - 1) {
    const long long v = __ldg(t + __ffs((int)m) - 1);
    best = v > best ? v : best;
  }
  if (best >= 0) return best;
  if (__ldg(t) >= 0) set_status(a.hdr, PARD_EDATA);      /* the mask names no path of this stage (a sink has none) */
  return lsub;
}

/* How the kernels of one request each get at its downstream estimate: all paths, as in the constants;
 * by its mask, path sums worked out by the block; by its mask, path sums at hand.  (Working them out is
 * a chain of dependent loads per path and block: a million requests with known paths, 27 -> 14 us for the rounds and 32 -> 19 us for the estimates.) */
enum { kAllPaths, kMaskStaged, kMaskAtHand };

/* One request's rounds and, for PARD_MODE_PATH_MASK, its own downstream estimate.  What it takes from
 * the queue's constants stays in registers while a thread's requests are of one queue, which they
 * mostly are: bound by instructions otherwise (2^24 requests under the window scan: 111 us with the
 * table entry read for every request). */
/* (The kernels of this file are kept to 64 registers, 32 warps per multiprocessor, but for those that
 * work out path sums.) */
template <int MASK>
__global__ void __launch_bounds__(kPolThreads, MASK == kMaskStaged ? 5 : 8)
k_policy_terms(const __grid_constant__ PolicyArgs a) {
  pdl_wait();
  __shared__ __align__(16) unsigned char sp_raw[MASK == kMaskStaged ? sizeof(StagedPaths) : 16];
  StagedPaths& sp = *reinterpret_cast<StagedPaths*>(sp_raw);
  if (a.hdr->wide || a.hdr->aborted) return;
  const SortedView v = sorted_view(a);
  const bool lookup = a.hdr->lookup != 0;
  const uint64_t tile0 = (uint64_t)blockIdx.x * kPolTile;
  if (MASK == kAllPaths && threadIdx.x == 0) l2_ahead(v.src, tile0, (uint64_t)kDecAhead * kPolTile, kPolTile, a.n);   /* (the others have no registers left for it) */
  if (MASK == kMaskStaged) stage_paths(a, v, tile0, sp);
  constexpr int kUn = 4;                           /* elements, then their records, requested together */
  uint32_t cur = 0xffffffffu;
  long long from = 0;                              /* deadline - A = offset (or deadline) - from, or from - offset */
  unsigned long long magic = 0;
  bool none = false, falls = false;
#pragma unroll 1
  for (int i0 = 0; i0 < kPolItems; i0 += kUn) {
    unsigned long long e[kUn], D[kUn];
    uint32_t flags[kUn];
#pragma unroll
    for (int u = 0; u < kUn; ++u) {
      const uint64_t j = tile0 + (uint64_t)(i0 + u) * kPolThreads + threadIdx.x;
      e[u] = j < a.n ? v.src[j] : 0ull;
    }
#pragma unroll
    for (int u = 0; u < kUn; ++u) {
      const uint64_t j = tile0 + (uint64_t)(i0 + u) * kPolThreads + threadIdx.x;
      const uint32_t idx = (uint32_t)e[u] & v.imask;
      D[u] = 0;
      flags[u] = 0;
      if (j >= a.n) continue;
      if (lookup) D[u] = __ldg(reinterpret_cast<const unsigned long long*>(&a.req[idx]));
      if (MASK) flags[u] = __ldg(&reinterpret_cast<const uint32_t*>(&a.req[idx])[3]) >> 16;
    }
#pragma unroll
    for (int u = 0; u < kUn; ++u) {
      const uint64_t j = tile0 + (uint64_t)(i0 + u) * kPolThreads + threadIdx.x;
      if (j >= a.n) continue;
      const uint32_t seg = (uint32_t)(e[u] >> v.kshift), idx = (uint32_t)e[u] & v.imask;
      const PardSegConst& K = a.ktab[seg];
      if (seg != cur) {
        cur = seg;
        from = lookup ? K.A : K.A_rel;
        if (a.mode & PARD_MODE_NEXUS) from -= K.lsub;           /* the current module only: base + d */
        falls = !lookup && (K.narrow & kSegHighFirst);          /* offsets counted down from the ctx's largest deadline */
        magic = K.d_magic;
        none = K.narrow & kSegNoStage;
      }
      if (none) { set_status(a.hdr, PARD_EDATA); v.T[j] = 0; continue; }
      long long X = (long long)(lookup ? D[u] : (e[u] >> a.ibits) & v.dmask) - from;
      if (falls) X = -X;
      if (a.mode & PARD_MODE_CLIPPER) {
        /* the module's share of the request's objective, counted from its arrival at the module; the
         * request is kept iff its batch starts within the share: start <= arrive + share, i.e.
         * start + d <= arrive + share + d */
        const pard_arrival_t ar = a.arrivals[idx];
        if (ar.arrive_us < 0 || ar.arrive_us >= PARD_TIME_LIMIT_US || ar.slo_us < 0 || ar.slo_us >= (1ll << 31) ||
            K.d >= (1ll << 32)) {
          set_status(a.hdr, PARD_EDATA);
          X = -1;
        } else {
          const long long share = (long long)((unsigned long long)ar.slo_us * (unsigned long long)K.d / (unsigned long long)K.dsum);
          X = ar.arrive_us + share + K.d - (K.A - K.lsub);
        }
      }
      if (MASK && flags[u]) X += K.lsub - (MASK == kMaskAtHand ? masked_lsub_at_hand(a, seg, flags[u], K.lsub) : masked_lsub(a, sp, seg, flags[u], K));
      v.T[j] = rounds_fit(X, magic, (unsigned long long)K.d);
    }
  }
}

/* The blocks of a cluster: this one's rank, a word stored in block `to`'s shared memory, all of them brought
 * together. */
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_store(uint32_t* p, uint32_t to, uint32_t v) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(to));
  asm volatile("st.shared::cluster.u32 [%0], %1;" :: "r"(remote), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

/* What a group of WARPS warps in each of CTAS blocks that walks one queue together exchanges: running sums and maxima
 * over its threads, in thread order.  One barrier each, of the block or of the cluster; the slots are used in turn. */
template <int WARPS, int CTAS>
struct WalkGroup {
  static constexpr int kAll = WARPS * CTAS, kPer = kAll > 32 ? kAll / 32 : 1;   /* warps of the group; figures that a lane adds up */
  struct Shared {
    __align__(16) uint32_t of_warp[2][2][kAll];    /* every block has all of them */
    uint32_t pos;
  };
  Shared& sh;
  uint32_t lane, warp, rank;
  uint32_t turn;
  __device__ uint32_t thread() const { return (rank * WARPS + warp) * 32 + lane; }
  __device__ void sync() const {
    if (CTAS > 1) cluster_sync();
    else if (WARPS > 1) __syncthreads();
    else __syncwarp();
  }
  /* the warps' figures x (and y), the same in all lanes of a warp, to everybody: op(index, x, y) for this lane's share of them */
  template <bool TWO, typename Op>
  __device__ void exchange(uint32_t x, uint32_t y, Op op) {
    const uint32_t me = rank * WARPS + warp;
    turn ^= 1;
    if (CTAS > 1) {
      if (lane < CTAS) {
        cluster_store(&sh.of_warp[turn][0][me], lane, x);
        if (TWO) cluster_store(&sh.of_warp[turn][1][me], lane, y);
      }
    } else if (lane == 0) {
      sh.of_warp[turn][0][me] = x;
      if (TWO) sh.of_warp[turn][1][me] = y;
    }
    sync();
    if (lane * kPer < kAll)
#pragma unroll
      for (int k = 0; k < kPer; ++k) op(lane * kPer + k, sh.of_warp[turn][0][lane * kPer + k], TWO ? sh.of_warp[turn][1][lane * kPer + k] : 0u);
  }
  /* sum over the earlier threads; *total: over all */
  __device__ uint32_t sum_before(uint32_t x, uint32_t* total) {
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    const uint32_t mine = __shfl_sync(0xffffffffu, incl, 31), me = rank * WARPS + warp;
    if (kAll == 1) {
      *total = mine;
      return incl - x;
    }
    uint32_t all = 0, before = 0;
    exchange<false>(mine, 0u, [&](uint32_t k, uint32_t v, uint32_t) { all += v; before += k < me ? v : 0u; });
    *total = __reduce_add_sync(0xffffffffu, all);
    return incl - x + __reduce_add_sync(0xffffffffu, before);
  }
  /* maximum over the earlier threads (at least `floor`); *total: over all */
  __device__ int32_t max_before(int32_t x, int32_t floor, int32_t* total) {
    int32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= (uint32_t)o) incl = max(incl, y);
    }
    int32_t before = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) before = floor;
    const int32_t mine = __shfl_sync(0xffffffffu, incl, 31);
    if (kAll == 1) {
      *total = max(floor, mine);
      return max(floor, before);
    }
    const uint32_t me = rank * WARPS + warp;
    int32_t all = floor, ahead = floor;
    exchange<false>((uint32_t)mine, 0u, [&](uint32_t k, uint32_t v, uint32_t) { all = max(all, (int32_t)v); ahead = k < me ? max(ahead, (int32_t)v) : ahead; });
    *total = __reduce_max_sync(0xffffffffu, all);
    return max(max(floor, before), __reduce_max_sync(0xffffffffu, ahead));
  }
  /* smallest and largest x of the group */
  __device__ void range_all(uint32_t lo, int32_t hi, uint32_t* least, int32_t* most) {
    uint32_t m = __reduce_min_sync(0xffffffffu, lo);
    int32_t t = __reduce_max_sync(0xffffffffu, hi);
    if (kAll > 1) {
      uint32_t ms = 0xffffffffu;
      int32_t ts = -1;
      exchange<true>(m, (uint32_t)t, [&](uint32_t, uint32_t x, uint32_t y) { ms = min(ms, x); ts = max(ts, (int32_t)y); });
      m = __reduce_min_sync(0xffffffffu, ms);
      t = __reduce_max_sync(0xffffffffu, ts);
    }
    *least = m;
    *most = t;
  }
  /* smallest x of the group */
  __device__ uint32_t min_all(uint32_t x) {
    uint32_t m = __reduce_min_sync(0xffffffffu, x);
    if (kAll > 1) {
      uint32_t ms = 0xffffffffu;
      exchange<false>(m, 0u, [&](uint32_t, uint32_t v, uint32_t) { ms = min(ms, v); });
      m = __reduce_min_sync(0xffffffffu, ms);
    }
    return m;
  }
  /* by one thread: a position for all, who see it behind the next sync() */
  __device__ void tell(uint32_t pos) {
    if (CTAS > 1)
      for (int k = 0; k < CTAS; ++k) cluster_store(&sh.pos, (uint32_t)k, pos);
    else
      sh.pos = pos;
  }
};

constexpr int kWalkItems = 16;                     /* consecutive requests per thread and step */
constexpr uint32_t kWalkWarps = 32;                /* warps of a group that walks a long queue (16: 123 us instead of 94 at 16 x 2^20) */
constexpr uint32_t kWalkLong = 2048;               /* requests per queue on average from which a block, not a warp, walks one:
                                                      an eighth of the 16,384 requests a block takes in one step */
constexpr int kWalkCtas = 8;                       /* blocks of a cluster that walks a queue */
constexpr uint32_t kWalkShare = kWalkWarps * 32 * kWalkItems;           /* requests a block takes in one step */
constexpr uint32_t kWalkClusterLong = 4 * kWalkCtas * kWalkShare;       /* shorter queues, and ... */
constexpr uint32_t kWalkClusterCap = 4 * kWalkShare;                    /* ... queues of smaller rounds are walked by one block: a round costs */
constexpr uint32_t kWalkClusterWindow = kWalkShare;                     /* two of the cluster's barriers; windows of Nexus seldom fill */
constexpr int kWalkClusterRounds = 2;              /* most queues: as many clusters as two rounds of the device's blocks (37) */
constexpr uint32_t kWalkCopiesLong = 4 * kWalkShare;   /* from so many requests per queue on, and up to a queue per multiprocessor, one block's
                                                      thresholds are copied ahead: the room leaves one block there instead of two */
constexpr uint32_t kWalkSmallRound = 64;           /* rounds below this size are walked by one warp, 32 requests per step: a step
                                                      closes several of them, where a group needs a barrier for each */

/* The thresholds of step after step, 16 consecutive ones per thread; the array may be read up to the next multiple
 * of 16 (workspace).
 * COPIES: a block has them copied into shared memory, kFeedDepth steps ahead, and reads them there four at a
 * time, the four vectors of a thread in an order that starts a place further with every second thread: as loads of
 * 64 bytes per lane from global memory they took 16 wavefronts an instruction, and a step 1.45 us of which the rest
 * of the work needs 0.5 (16 queues of 2^20, Nexus: the walk 93 us). */
constexpr int kFeedDepth = 3;
template <int WARPS, int CTAS, bool COPIES>
struct WalkFeed {
  static constexpr uint32_t kStep = WARPS * 32 * kWalkItems;
  const uint32_t* T;
  uint32_t at, hi, next[kWalkItems];
  static constexpr uint32_t rot = 0;
  __device__ void load() {
#pragma unroll
    for (int q = 0; q < kWalkItems / 4; ++q) {
      uint4 x = make_uint4(0u, 0u, 0u, 0u);
      if (at + 4 * q < hi) x = *reinterpret_cast<const uint4*>(T + at + 4 * q);
      next[4 * q] = x.x; next[4 * q + 1] = x.y; next[4 * q + 2] = x.z; next[4 * q + 3] = x.w;
    }
    at += kStep;
  }
  __device__ WalkFeed(const PolicyArgs&, const uint32_t* T_, uint32_t first, uint32_t hi_, uint32_t t, uint32_t) : T(T_), at(first + t * kWalkItems), hi(hi_) { load(); }
  /* this step's, and the next one's on their way */
  __device__ void step(uint32_t (&u)[kWalkItems]) {
#pragma unroll
    for (int i = 0; i < kWalkItems; ++i) u[i] = next[i];
    load();
  }
  __device__ uint32_t in_order(uint32_t bits) const { return bits; }
};
struct FeedSmem {
  uint32_t ring[kFeedDepth][kWalkWarps * 32 * kWalkItems];
  unsigned long long full[kFeedDepth];             /* mbarriers */
};
__device__ __forceinline__ FeedSmem* feed_smem() {
  extern __shared__ __align__(16) unsigned char walk_raw[];
  return reinterpret_cast<FeedSmem*>(walk_raw);
}
template <int CTAS>
struct WalkFeed<(int)kWalkWarps, CTAS, true> {
  static constexpr uint32_t kShare = kWalkWarps * 32 * kWalkItems;      /* of a block; the step's are the blocks' shares in order of rank */
  FeedSmem& Sm;
  const PolicyArgs& a;
  const uint32_t* T;
  uint32_t from, hi, t, slot, parity, rot;         /* from: first of the next share to fetch; rot: the vector a thread begins with */
  uint32_t left;                                   /* steps for which this block has a share */
  __device__ void fetch(uint32_t to) {             /* by thread 0 */
    if (from >= hi) return;
    bulk_fetch(&Sm.full[to], Sm.ring[to], T + from, ((min(hi - from, kShare) + 3) & ~3u) * 4);
    from += CTAS * kShare;
  }
  __device__ WalkFeed(const PolicyArgs& a_, const uint32_t* T_, uint32_t first, uint32_t hi_, uint32_t t_, uint32_t rank)
      : Sm(*feed_smem()), a(a_), T(T_), from(first + rank * kShare), hi(hi_), t(t_), slot(0), parity(0), rot((t_ >> 1) & 3u),
        left(from < hi_ ? (hi_ - from + CTAS * kShare - 1) / (CTAS * kShare) : 0u) {
    if (t == 0) {
      for (int k = 0; k < kFeedDepth; ++k) bulk_init(&Sm.full[k]);
      for (int k = 0; k < kFeedDepth; ++k) {
        if (k == 0 && (a.mode & PARD_MODE_TEST_STALL) && blockIdx.x == 0) from += CTAS * kShare;     /* testing aid: a share never asked for */
        else fetch(k);
      }
    }
    __syncthreads();
  }
  /* A wait that runs out does not end the walk here: blocks of a cluster store into each other's shared memory, so
   * they go on together, this one without requests that fit. */
  __device__ void step(uint32_t (&u)[kWalkItems]) {
#pragma unroll
    for (int i = 0; i < kWalkItems; ++i) u[i] = 0;
    if (!left) return;
    --left;
    const bool late = !bulk_arrived(&Sm.full[slot], parity);
    const uint4* mine = reinterpret_cast<const uint4*>(Sm.ring[slot]) + t * (kWalkItems / 4);
#pragma unroll
    for (uint32_t q = 0; q < kWalkItems / 4; ++q) {
      const uint4 x = mine[(q + rot) & 3u];
      u[4 * q] = x.x; u[4 * q + 1] = x.y; u[4 * q + 2] = x.z; u[4 * q + 3] = x.w;
    }
    if (__syncthreads_or(late)) {                  /* (also: everybody has read the slot) */
#pragma unroll
      for (int i = 0; i < kWalkItems; ++i) u[i] = 0;
      left = 0;
      if (t == 0) {
        for (int k = 0; k < kFeedDepth; ++k) bulk_arrived(&Sm.full[k], k < (int)slot ? parity ^ 1 : parity);   /* no copy is under way when the block ends */
        a.hdr->walk_late = 1;
        set_status(a.hdr, PARD_ETIMEOUT);
      }
      return;
    }
    if (t == 0) fetch(slot);
    if (++slot == kFeedDepth) { slot = 0; parity ^= 1; }
  }
  /* bit i of `bits`: the i-th value as read; of the result: the i-th in the array */
  __device__ uint32_t in_order(uint32_t bits) const { return ((bits << (4 * rot)) | (bits >> (16 - 4 * rot))) & 0xffffu; }
};
/* bits of this thread's requests that fit round b (in the order of u) */
__device__ __forceinline__ uint32_t walk_fit(const uint32_t (&v)[kWalkItems], uint32_t b) {
  uint32_t g = 0;
#pragma unroll
  for (int i = kWalkItems - 1; i >= 0; --i) g = __funnelshift_l(b - v[i], g, 1);      /* both at most 2^30: the sign says it */
  return g;
}

/* bits of the positions at .. at+15 that lie in [from, hi) */
__device__ __forceinline__ uint32_t walk_range(uint32_t at, uint32_t from, uint32_t hi) {
  uint32_t m = 0xffffu;
  if (from > at) m = from - at >= 16 ? 0u : m & (0xffffu << (from - at));
  if (hi < at + 16) m = hi <= at ? 0u : m & (0xffffu >> (at + 16 - hi));
  return m;
}

/* The general rule in rounds of at least kWalkSmallRound.  RAW: every request ahead takes a slot,
 * so a request's round is its position's and no round has to be waited for. */
template <int WARPS, int CTAS, bool COPIES, bool RAW>
__device__ void walk_admit(WalkGroup<WARPS, CTAS>& G, const PolicyArgs& a, const SortedView& v, uint32_t s, uint32_t lo,
                           uint32_t hi, const PardSegConst& K) {
  constexpr uint32_t kStep = CTAS * WARPS * 32 * kWalkItems;
  const uint32_t cap = K.cap, t = G.thread();
  uint32_t x = 0, b = 0, left = cap;
  uint32_t at = (lo & ~(uint32_t)(kWalkItems - 1)) + t * kWalkItems;
  WalkFeed<WARPS, CTAS, COPIES> feed(a, v.T, lo & ~(uint32_t)(kWalkItems - 1), hi, G.warp * 32 + G.lane, G.rank);
  for (uint32_t step = lo & ~(uint32_t)(kWalkItems - 1); step < hi; step += kStep, at += kStep) {
    uint32_t u[kWalkItems];
    feed.step(u);
    uint32_t open = walk_range(at, lo, hi), kept = 0, before = 0, total = 0;
    const uint32_t x0 = x;
    bool several = false;
    for (;;) {
      uint32_t fit = 0;
      if (RAW) {
#pragma unroll
        for (int i = 0; i < kWalkItems; ++i) {
          const uint32_t r = at + ((i + 4 * feed.rot) & (kWalkItems - 1)) - lo, round = K.cap_magic ? div_magic32(r, K.cap_magic) : r;
          fit |= (u[i] > round ? 1u : 0u) << i;
        }
      } else {
        fit = walk_fit(u, b);
      }
      fit = feed.in_order(fit) & open;
      const uint32_t mine = __popc(fit);
      before = G.sum_before(mine, &total);
      if (RAW || total < left) {                   /* the round does not close in this step */
        kept |= fit;
        x += total;
        left -= total;
        break;
      }
      several = true;
      if (before < left && left <= before + mine) {     /* it closes here, behind this thread's (left - before)-th fitting request */
        uint32_t m = fit;
        for (uint32_t k = left - before; k > 1; --k) m &= m - 1;
        const uint32_t end = at + __ffs(m);        /* position behind it */
        kept |= fit & (0xffffu >> (at + 16 - end));
        v.C[lo + b] = end;
        G.tell(end);
      } else if (before + mine < left) {
        kept |= fit;
      }
      G.sync();
      const uint32_t end = G.sh.pos;
      x += left;
      left = cap;
      ++b;
      open = walk_range(at, end, hi);
      if (end >= hi) { G.sync(); break; }          /* (the slot may be written again) */
    }
    if (several) before = G.sum_before(__popc(kept), &total);
    if ((at & (kPolTile - 1)) == 0 && at >= lo && at < hi) a.tile_x[at / kPolTile] = x0 + before;
  }
  if (t == 0) { a.seg_kept[s] = x; a.rounds[s] = b; }
}

/* The same in small rounds, by one warp: the keep mask of a step of 32 is the fixed point of
 * keep_i = [x + #kept among lanes below i < u_i] (bit i is final after i + 1 iterations). */
__device__ void walk_admit_small(const PolicyArgs& a, const SortedView& v, uint32_t s, uint32_t lo, uint32_t hi,
                                 const PardSegConst& K, uint32_t lane) {
  const uint32_t below = (1u << lane) - 1, cap = K.cap;
  uint32_t x = 0;
  uint32_t next = lo + lane < hi ? v.T[lo + lane] : 0u;
  for (uint32_t b0 = lo; b0 < hi; b0 += 32) {
    const uint32_t j = b0 + lane;
    const unsigned long long u64 = (unsigned long long)next * cap;
    const uint32_t u = u64 > kUClamp ? kUClamp : (uint32_t)u64;       /* beyond the queue: 0, never kept */
    next = j + 32 < hi ? v.T[j + 32] : 0u;
    uint32_t m = __ballot_sync(0xffffffffu, x < u);        /* as if nobody in the step were kept before */
    for (int round = 0; round < 34; ++round) {
      const uint32_t m2 = __ballot_sync(0xffffffffu, x + __popc(m & below) < u);
      if (m2 == m) break;
      m = m2;
    }
    const uint32_t c = x + __popc(m & below);
    if ((j & (kPolTile - 1)) == 0 && j < hi) a.tile_x[j / kPolTile] = c;
    if ((m >> lane) & 1u) {                        /* the c-th admitted request closes a round when c + 1 fills it */
      const uint32_t q = K.cap_magic ? div_magic32(c + 1, K.cap_magic) : c + 1;
      if (q * cap == c + 1) v.C[lo + q - 1] = j + 1;
    }
    x += __popc(m);
  }
  if (lane == 0) { a.seg_kept[s] = x; a.rounds[s] = K.cap_magic ? div_magic32(x, K.cap_magic) : x; }
}

/* Nexus: the batch is the first window of W = cap requests that all fit the round b being formed
 * (b < v_r), everything before it is dropped, b advances, the scan goes on behind it.  With `bad`
 * the last position that does not fit (or that ends the window before), a window closes at
 * bad + W, the first time that lies before the next misfit. */
template <int WARPS, int CTAS, bool COPIES>
__device__ void walk_nexus(WalkGroup<WARPS, CTAS>& G, const PolicyArgs& a, const SortedView& v, uint32_t s, uint32_t lo,
                           uint32_t hi, uint32_t W) {
  constexpr uint32_t kStep = CTAS * WARPS * 32 * kWalkItems;
  constexpr uint32_t kNone = 0xffffffffu;
  const uint32_t t = G.thread();
  uint32_t b = 0;
  int32_t bad = (int32_t)lo - 1;
  uint32_t at = (lo & ~(uint32_t)(kWalkItems - 1)) + t * kWalkItems;
  WalkFeed<WARPS, CTAS, COPIES> feed(a, v.T, lo & ~(uint32_t)(kWalkItems - 1), hi, G.warp * 32 + G.lane, G.rank);
  for (uint32_t step = lo & ~(uint32_t)(kWalkItems - 1); step < hi; step += kStep, at += kStep) {
    uint32_t u[kWalkItems];
    feed.step(u);
    uint32_t from = lo;
    for (;;) {
      const uint32_t open = walk_range(at, from, hi);
      const uint32_t miss = ~feed.in_order(walk_fit(u, b)) & open;
      if (W >= kStep) {                            /* a window cannot begin and end in one step: only the running one can close */
        uint32_t least;
        int32_t most;
        G.range_all(miss ? at + __ffs(miss) - 1 : kNone, miss ? (int32_t)at + 31 - __clz(miss) : -1, &least, &most);
        const unsigned long long full = (unsigned long long)((long long)bad + W);
        if (full < hi && full < least && full < (unsigned long long)step + kStep) {
          if (t == 0) v.C[lo + b] = (uint32_t)full + 1;
          ++b;
          bad = (int32_t)full;
          from = (uint32_t)full + 1;
          if (from >= hi) break;
          continue;                                /* the rest of the step, under the next round */
        }
        bad = max(bad, most);
        break;
      }
      int32_t top;
      const int32_t last = G.max_before(miss ? (int32_t)at + 31 - __clz(miss) : -1, bad, &top);
      uint32_t found = kNone;
      if (open) {                                  /* a window can only close ahead of the thread's first misfit: it is longer than a thread's share */
        const uint32_t end = miss ? at + __ffs(miss) - 1 : min(at + 16, hi);
        const unsigned long long full = (unsigned long long)((long long)last + W);   /* where a window would close */
        if (full < end && full >= max(at, from)) found = (uint32_t)full;
      }
      found = G.min_all(found);
      if (found == kNone) { bad = top; break; }
      if (t == 0) v.C[lo + b] = found + 1;
      ++b;
      bad = (int32_t)found;
      from = found + 1;
      if (from >= hi) break;
    }
  }
  if (t == 0) {
    const uint32_t run = (uint32_t)((int32_t)hi - 1 - bad);          /* a last, partly filled window runs as it is */
    a.rounds[s] = b;
    a.tail[s] = run;
    a.seg_kept[s] = b * W + run;
  }
}

/* Nexus in small windows, by one warp, 32 requests per step. */
__device__ void walk_nexus_small(const PolicyArgs& a, const SortedView& v, uint32_t s, uint32_t lo, uint32_t hi,
                                 uint32_t W, uint32_t lane) {
  uint32_t b = 0, run = 0;                         /* batches formed; length of the current run of fitting requests */
  uint32_t next = lo + lane < hi ? v.T[lo + lane] : 0u;
  for (uint32_t p0 = lo; p0 < hi; p0 += 32) {
    const uint32_t nvalid = min(32u, hi - p0);
    const uint32_t x = next;
    next = p0 + 32 + lane < hi ? v.T[p0 + 32 + lane] : 0u;
    const uint32_t valid = nvalid == 32 ? 0xffffffffu : ((1u << nvalid) - 1);
    uint32_t pos = 0;
    while (pos < nvalid) {                         /* uniform */
      const uint32_t fit = __ballot_sync(0xffffffffu, b < x) & valid;
      const uint32_t misfit = ~fit & valid & ~((1u << pos) - 1);
      const uint32_t firstbad = misfit ? (uint32_t)__ffs(misfit) - 1 : nvalid;
      const uint32_t fitlen = firstbad - pos, need = W - run;
      if (fitlen >= need) {                        /* the window is full at lane pos + need - 1 */
        pos += need;
        if (lane == 0) v.C[lo + b] = p0 + pos;
        ++b;
        run = 0;
      } else if (firstbad < nvalid) {              /* a request that does not fit: the run before it goes too */
        run = 0;
        pos = firstbad + 1;
      } else {                                     /* everything up to the end of the step fits: the run goes on */
        run += fitlen;
        pos = nvalid;
      }
    }
  }
  if (lane == 0) { a.rounds[s] = b; a.tail[s] = run; a.seg_kept[s] = b * W + run; }
}

/* CTAS > 1: a cluster per queue, for the queues where its barriers are worth it: many steps, few rounds.  The first
 * block of the cluster walks the others by itself.  (A step of one block 1.2 us, of a cluster some 1.5 for eight times
 * the requests, a round 0.6 and 1.5; 2^23 requests with known paths in 32 queues of 2^18: 612 by blocks, 621 by clusters.) */
template <int WARPS, int CTAS, bool COPIES>
__global__ void __launch_bounds__(WARPS == 1 ? kPolThreads : WARPS * 32)
k_policy_walk(const __grid_constant__ PolicyArgs a) {
  pdl_wait();
  constexpr int kGroups = WARPS == 1 ? kPolThreads / 32 : 1;
  __shared__ typename WalkGroup<WARPS, CTAS>::Shared sh[kGroups];
  if (a.hdr->wide || a.hdr->aborted) return;       /* (nothing sets them while this kernel runs) */
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rank = CTAS > 1 ? cluster_rank() : 0u;
  const uint32_t s = WARPS == 1 ? blockIdx.x * kGroups + warp : blockIdx.x / CTAS;
  if (s >= a.n_seg) return;                        /* whole groups leave together */
  const SortedView v = sorted_view(a);
  const uint32_t lo = a.seg_off[s], hi = a.seg_off[s + 1];
  if (hi <= lo) {
    if (rank == 0 && lane == 0 && (WARPS == 1 || warp == 0)) { a.rounds[s] = 0; a.tail[s] = 0; a.seg_kept[s] = 0; }
    return;
  }
  const PardSegConst K = a.ktab[s];
  const bool nexus = a.mode & PARD_MODE_NEXUS, raw = a.mode & PARD_MODE_RAW;
  if (K.cap < kWalkSmallRound && !raw) {
    if (rank || (WARPS > 1 && warp != 0)) return;
    if (nexus) walk_nexus_small(a, v, s, lo, hi, K.cap, lane);
    else walk_admit_small(a, v, s, lo, hi, K, lane);
    return;
  }
  auto walk = [&](auto ctas) {
    constexpr int N = decltype(ctas)::value;
    WalkGroup<WARPS, N> G{reinterpret_cast<typename WalkGroup<WARPS, N>::Shared&>(sh[WARPS == 1 ? warp : 0]), lane, WARPS == 1 ? 0u : warp, N > 1 ? rank : 0u, 0u};
    if (nexus) walk_nexus<WARPS, N, COPIES>(G, a, v, s, lo, hi, K.cap);
    else if (raw) walk_admit<WARPS, N, COPIES, true>(G, a, v, s, lo, hi, K);
    else walk_admit<WARPS, N, COPIES, false>(G, a, v, s, lo, hi, K);
  };
  if (CTAS > 1 && (raw || K.cap < (nexus ? kWalkClusterWindow : kWalkClusterCap) || hi - lo < kWalkClusterLong)) {
    if (rank == 0) walk(std::integral_constant<int, 1>());
  } else {
    if (CTAS > 1) cluster_sync();                  /* every block's shared memory is there before another stores into it */
    walk(std::integral_constant<int, CTAS>());
  }
}

/* Estimates, decisions and survivors, eight consecutive requests per thread.  A request's round is the number of rounds
 * of its queue that ended at or before it, found by a search in the ends: a warp's 32-ary search for the warp's first
 * request, from there a few steps for a thread's first one -- a round takes at least a batch of requests, so p positions
 * on it is at most p / cap rounds on --, and one round after the other behind that.  (A binary search over all of the
 * queue's rounds for every 128th request was a chain of up to 120 dependent loads: 2^24 requests in
 * queues of 2^15 rounds, 130 us.)  Its place among the survivors is, for Nexus, given by its window, else the kept requests
 * ahead of it: those ahead of the tile (a.tile_x) and those inside it.  Survivors of a warp that sees one queue only
 * follow one another and go out from shared memory, side by side.
 * Bound by instructions: 2^24 requests under the window scan 90 us with every 128th request to a thread (119 instructions
 * per request), 64 like this; 17 + 4f bytes each would take 45.
 * INDEX: the sort left the requests' indexes alone (k_sort_requests); a queue is known by its positions. */
template <int MASK, bool INDEX = false>
__global__ void __launch_bounds__(kPolThreads, MASK == kMaskStaged ? 5 : 8)
k_policy_emit(const __grid_constant__ PolicyArgs a) {
  pdl_wait();
  constexpr int kRows = kPolTile / 32;
  static_assert(kRows == 32 && kPolItems == 8, "one warp scans the rows of 32; a thread's flags are one byte");
  __shared__ __align__(16) unsigned char sp_raw[MASK == kMaskStaged ? sizeof(StagedPaths) : 16];
  StagedPaths& sp = *reinterpret_cast<StagedPaths*>(sp_raw);
  __shared__ uint32_t s_keep[kRows], s_before[kRows];
  if (a.hdr->wide | a.hdr->aborted | a.hdr->walk_late) return;
  const SortedView v = sorted_view(a);
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t tile0 = blockIdx.x * kPolTile, j0 = tile0 + threadIdx.x * kPolItems;
  const bool nexus = !MASK && (a.mode & PARD_MODE_NEXUS), full = j0 + kPolItems <= a.n;     /* (known paths do not combine with it) */
  /* raw positions: no rule takes them, but the planner's own comes here too when its key is wider than an element */
  const bool raw = !MASK && !INDEX && (a.mode & PARD_MODE_RAW);
  __shared__ uint32_t s_out[kPolThreads / 32][32 * kPolItems];
  if (MASK == kAllPaths && threadIdx.x == 0)       /* (the others have no registers left for it) */
    l2_ahead(v.src, INDEX ? tile0 / 2 : tile0, (uint64_t)kDecAhead * kPolTile / (INDEX ? 2 : 1), INDEX ? kPolTile / 2 : kPolTile, INDEX ? a.n / 2 : a.n);
  /* Path sums worked out on the spot: 32 requests in a row to a warp for that, which mostly are of one queue or two.  (Only a
   * tile's first queues are staged; eight in a row per thread leave all others to the last warps: a million requests in
   * queues of 30 290 -> 326 us for the call.) */
  __shared__ long long s_paths[MASK == kMaskStaged ? kPolTile : 1];
  if (MASK == kMaskStaged) {
    stage_paths(a, v, tile0, sp);
#pragma unroll 1
    for (uint32_t p = threadIdx.x; p < (uint32_t)kPolTile && tile0 + p < a.n; p += kPolThreads) {
      const unsigned long long e = v.src[tile0 + p];
      const uint32_t flags = __ldg(&reinterpret_cast<const uint32_t*>(&a.req[(uint32_t)e & v.imask])[3]) >> 16, seg = (uint32_t)(e >> v.kshift);
      const PardSegConst& K = a.ktab[seg];
      s_paths[p] = flags && !(K.narrow & kSegNoStage) ? masked_lsub(a, sp, seg, flags, K) - K.lsub : 0ll;
    }
    __syncthreads();
  }
  uint32_t idx[kPolItems], t[kPolItems], my_seg = 0, last_seg = 0;
  long long est[kPolItems];                        /* at first: by how much the paths that a request names take it from the queue's estimate */
#pragma unroll
  for (int k = 0; k < kPolItems; ++k) est[k] = MASK == kMaskStaged && j0 + k < a.n ? s_paths[threadIdx.x * kPolItems + k] : 0ll;
  if (INDEX) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(v.src);
    if (full) {
      const uint4 x = *reinterpret_cast<const uint4*>(src + j0), y = *reinterpret_cast<const uint4*>(src + j0 + 4);
      idx[0] = x.x; idx[1] = x.y; idx[2] = x.z; idx[3] = x.w; idx[4] = y.x; idx[5] = y.y; idx[6] = y.z; idx[7] = y.w;
    } else {
#pragma unroll
      for (int i = 0; i < kPolItems; ++i) idx[i] = j0 + i < a.n ? src[j0 + i] : 0u;
    }
  } else {
    unsigned long long e[kPolItems];
    if (full) {
      load4(v.src + j0, e);
      load4(v.src + j0 + 4, e + 4);
    } else {
#pragma unroll
      for (int i = 0; i < kPolItems; ++i) e[i] = j0 + i < a.n ? v.src[j0 + i] : 0ull;
    }
#pragma unroll
    for (int i = 0; i < kPolItems; ++i) idx[i] = (uint32_t)e[i] & v.imask;
    my_seg = (uint32_t)(e[0] >> v.kshift);
    last_seg = (uint32_t)(e[kPolItems - 1] >> v.kshift);
    if (MASK == kMaskAtHand) {
      uint32_t flags[kPolItems];
#pragma unroll
      for (int k = 0; k < kPolItems; ++k) flags[k] = j0 + k < a.n ? __ldg(&reinterpret_cast<const uint32_t*>(&a.req[idx[k]])[3]) >> 16 : 0u;
#pragma unroll
      for (int k = 0; k < kPolItems; ++k)
        if (flags[k]) {
          const uint32_t seg = (uint32_t)(e[k] >> v.kshift);
          const PardSegConst& K = a.ktab[seg];
          if (!(K.narrow & kSegNoStage)) est[k] = masked_lsub_at_hand(a, seg, flags[k], K.lsub) - K.lsub;
        }
    }
  }
  if (full && !nexus) {
    const uint4 x = *reinterpret_cast<const uint4*>(v.T + j0), y = *reinterpret_cast<const uint4*>(v.T + j0 + 4);
    t[0] = x.x; t[1] = x.y; t[2] = x.z; t[3] = x.w; t[4] = y.x; t[5] = y.y; t[6] = y.z; t[7] = y.w;
  } else {
#pragma unroll
    for (int i = 0; i < kPolItems; ++i) t[i] = j0 + i < a.n && !nexus ? v.T[j0 + i] : 0u;
  }
  /* the round of the warp's first request */
  const uint32_t p0 = tile0 + warp * (32 * kPolItems);
  uint32_t seg_first = 0;
  bool one_queue;                                  /* all of the warp's requests are there and of one queue */
  if (INDEX) {                                     /* the queues that end at or before p0 come before it */
    uint32_t before = 0;
    for (uint32_t q = lane; q < a.n_seg; q += 32) before += a.seg_off[q + 1] <= p0 ? 1u : 0u;
    seg_first = min(__reduce_add_sync(0xffffffffu, before), a.n_seg - 1);
    one_queue = p0 + 32 * kPolItems <= min(a.seg_off[seg_first + 1], a.n);
  } else {
    seg_first = __shfl_sync(0xffffffffu, my_seg, 0);
    one_queue = __all_sync(0xffffffffu, full && my_seg == seg_first && last_seg == seg_first);
  }
  /* The queue of position j, the last that begins at or before it; none before queue `from`, the nearest ones looked at
   * first.  (All later ones halved again and again: a million requests in 32,768 queues under Clipper++ 180 -> 174 us,
   * 4.2 M in as many in arrival order 342 -> 328.) */
  auto queue_at = [&](uint32_t j, uint32_t from) {
    uint32_t step = 1;
    for (; from + step < a.n_seg && a.seg_off[from + step] <= j; step *= 2) from += step;
    uint32_t z = min(from + step, a.n_seg);
    while (z - from > 1) {
      const uint32_t mid = from + (z - from) / 2;
      if (a.seg_off[mid] <= j) from = mid; else z = mid;
    }
    return from;
  };
  uint32_t b0 = 0;
  if (!raw && p0 < a.n) {
    const uint32_t* ends = v.C + a.seg_off[seg_first];
    uint32_t z = a.rounds[seg_first];
    while (b0 < z) {                               /* uniform across the warp */
      const uint32_t span = z - b0;
      const uint32_t p = b0 + (uint32_t)(((unsigned long long)(lane + 1) * span) / 33u);   /* b0 <= p < z */
      const uint32_t c = __popc(__ballot_sync(0xffffffffu, ends[p] <= p0));                /* the lanes before lane c */
      const uint32_t p_below = __shfl_sync(0xffffffffu, p, c > 0 ? c - 1 : 0);
      const uint32_t p_at = __shfl_sync(0xffffffffu, p, c < 32 ? c : 31);
      if (c > 0) b0 = p_below + 1;
      if (c < 32) z = p_at;
    }
  }
  /* span after span of requests of one queue and round: mostly the thread's eight are one */
  uint32_t lo = 0, hi = 0, nb = 0, b = 0, cap = 0, tail = 0, place = 0, keepbits = 0, at = 0;
  long long A0 = 0, d = 0;
  bool none = false;
  const uint32_t count = j0 < a.n ? min(a.n - j0, (uint32_t)kPolItems) : 0u;
  for (uint32_t i = 0; i < count;) {
    const uint32_t j = j0 + i;
    if (j >= hi) {                                 /* a queue begins, or the thread's share does */
      if (INDEX || i > 0) my_seg = one_queue ? seg_first : queue_at(j, i > 0 ? my_seg : seg_first);
      const PardSegConst& K = a.ktab[my_seg];
      lo = a.seg_off[my_seg];
      hi = a.seg_off[my_seg + 1];
      nb = raw ? 0u : a.rounds[my_seg];
      cap = K.cap;
      none = K.narrow & kSegNoStage;
      tail = nexus ? a.tail[my_seg] : 0u;
      A0 = K.A;
      d = none ? 0 : K.d;
      if (!MASK && !none && (a.mode & (PARD_MODE_NEXUS | PARD_MODE_CLIPPER))) A0 -= K.lsub;     /* the current module only */
      if (nexus && a.out_kept_idx) place = a.kept_base[my_seg];
      b = 0;                                       /* (a queue that begins inside the thread's share: its first round) */
      if (i == 0 && !raw) {
        if (my_seg == seg_first) b = b0;
        const uint32_t on = j - max(lo, p0);
        uint32_t z = min(nb, b + (K.cap_magic ? div_magic32(on, K.cap_magic) : on) + 1);     /* ends b .. z-1: how many are <= j */
        while (b < z) {
          const uint32_t mid = b + (z - b) / 2;
          if (v.C[lo + mid] <= j) b = mid + 1; else z = mid;
        }
      }
    } else {
      ++b;                                         /* (no round is empty) */
    }
    const uint32_t end = b < nb ? v.C[lo + b] : 0xffffffffu;
    uint32_t stop = max(min(min(end, hi) - j0, count), i + 1);           /* (i + 1: the loop ends whatever the arrays hold) */
    if (raw) {
      const unsigned long long magic = a.ktab[my_seg].cap_magic;
      b = magic ? div_magic32(j - lo, magic) : j - lo;
      stop = i + 1;
    }
    const long long now = A0 + (long long)b * d;
    const uint32_t from = b < nb ? end - cap : hi - tail;      /* Nexus: the window's first request */
    uint32_t kept = 0;
    if (!nexus) {
#pragma unroll
      for (int k = 0; k < kPolItems; ++k) kept |= (t[k] > b ? 1u : 0u) << k;
    } else {
      kept = from <= j0 ? 255u : 255u << min(from - j0, 8u);
    }
    const uint32_t span = (1u << stop) - (1u << i);
    kept = none ? 0u : kept & span;
#pragma unroll
    for (int k = 0; k < kPolItems; ++k) est[k] += (span >> k) & 1u ? now : 0ll;
    if (nexus && kept && a.out_kept_idx) {
      const uint32_t to = place + b * cap + (j0 - from);       /* of the thread's request 0, were it of this window */
      if (!one_queue) {
#pragma unroll
        for (int k = 0; k < kPolItems; ++k)
          if ((kept >> k) & 1u) a.out_kept_idx[to + k] = idx[k];
      } else if (!keepbits) {
        at = to + (uint32_t)__ffs((int)kept) - 1;  /* the thread's first */
      }
    }
    keepbits |= kept;
    i = stop;
  }
  if (full) {
    if (a.out_keep) *reinterpret_cast<uint2*>(a.out_keep + j0) = make_uint2(((keepbits & 15u) * 0x00204081u) & 0x01010101u, ((keepbits >> 4) * 0x00204081u) & 0x01010101u);
    if (a.out_est) {
      store4(a.out_est + j0, est[0], est[1], est[2], est[3]);
      store4(a.out_est + j0 + 4, est[4], est[5], est[6], est[7]);
    }
    if (a.out_perm) {
      auto two = [&](int i) { return idx[i] | (unsigned long long)idx[i + 1] << 32; };
      store4(a.out_perm + j0, two(0), two(2), two(4), two(6));
    }
  } else {
#pragma unroll
    for (int i = 0; i < kPolItems; ++i)
      if (j0 + i < a.n) {
        if (a.out_keep) a.out_keep[j0 + i] = (keepbits >> i) & 1u;
        if (a.out_est) a.out_est[j0 + i] = est[i];
        if (a.out_perm) a.out_perm[j0 + i] = idx[i];
      }
  }
  if (!a.out_kept_idx) return;
  /* a warp's survivors, to be written from position `to` of the output on */
  auto write_out = [&](uint32_t rank, uint32_t total, uint32_t to) {
    uint32_t* out = s_out[warp];
#pragma unroll
    for (int i = 0; i < kPolItems; ++i)
      if ((keepbits >> i) & 1u) out[rank + __popc(keepbits & ((1u << i) - 1))] = idx[i];
    __syncwarp();
    for (uint32_t k = lane; k < total; k += 32) a.out_kept_idx[to + k] = out[k];
  };
  if (nexus) {
    if (!one_queue) return;
    uint32_t rank = __popc(keepbits);
    const uint32_t mine = rank, any = __ballot_sync(0xffffffffu, mine != 0);
    if (!any) return;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, rank, o);
      if (lane >= (uint32_t)o) rank += y;
    }
    write_out(rank - mine, __shfl_sync(0xffffffffu, rank, 31), __shfl_sync(0xffffffffu, at, __ffs((int)any) - 1));
    return;
  }
  reinterpret_cast<uint8_t*>(s_keep)[threadIdx.x] = (uint8_t)keepbits;
  __syncthreads();
  if (warp == 0) {
    const uint32_t x = __popc(s_keep[lane]);
    uint32_t incl = x;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    s_before[lane] = incl - x;
  }
  __syncthreads();
  /* kept requests of the tile ahead of its position p */
  auto kept_before = [&](uint32_t p) { return s_before[p >> 5] + __popc(s_keep[p >> 5] & ((1u << (p & 31)) - 1)); };
  uint32_t c = kept_before(threadIdx.x * kPolItems);
  /* output position of the queue's survivors, less those of the tile ahead of its first */
  auto place_of = [&](uint32_t seg) {
    const uint32_t first = a.seg_off[seg];
    return a.kept_base[seg] + (first <= tile0 ? a.tile_x[blockIdx.x] : 0u - kept_before(first - tile0));
  };
  if (one_queue) {
    const uint32_t c0 = __shfl_sync(0xffffffffu, c, 0);
    write_out(c - c0, __shfl_sync(0xffffffffu, c + __popc(keepbits), 31) - c0, place_of(seg_first) + c0);
    return;
  }
  uint32_t seg = seg_first, behind = 0;            /* the queue at hand, its end */
#pragma unroll
  for (int i = 0; i < kPolItems; ++i) {
    if (!((keepbits >> i) & 1u)) continue;         /* (requests beyond the array are not kept) */
    if (j0 + i >= behind) {
      seg = queue_at(j0 + i, seg);
      at = place_of(seg);
      behind = a.seg_off[seg + 1];
    }
    a.out_kept_idx[at + c] = idx[i];
    ++c;
  }
}

}  // namespace

namespace pard_plan_detail {

int allow_walk_smem() {
  PARD_CUDA_OK(cudaFuncSetAttribute(k_policy_walk<kWalkWarps, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FeedSmem)));
  PARD_CUDA_OK(cudaFuncSetAttribute(k_policy_walk<kWalkWarps, kWalkCtas, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FeedSmem)));
  return PARD_OK;
}

/* A cluster's blocks are placed together.  Whether the device, or the share of it that this context may use, has room
 * for one at all is asked for every such call, not once: the share may change.  (The host's 25 us per call of 2^24
 * requests stay what they were; by one block each the 16 queues take 22 us more, 420 against 398.) */
static bool cluster_walk_fits() {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = kWalkCtas;
  cfg.blockDim = kWalkWarps * 32;
  cfg.dynamicSmemBytes = sizeof(FeedSmem);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kWalkCtas;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, k_policy_walk<kWalkWarps, kWalkCtas, true>, &cfg) == cudaSuccess) return clusters > 0;
  cudaGetLastError();                              /* an answer like any other: nothing of the call has failed */
  return false;
}

int launch_policy_walk(const PolicyArgs& a, int sms, cudaStream_t stream) {
  static_assert(kWalkItems < (int)kWalkSmallRound, "a window is longer than a thread's share of a step");
  static_assert(kPolTile == kDecTile, "tile_x is indexed by the planner's decision tiles");
  const uint32_t tiles = (uint32_t)(((uint64_t)a.n + kPolTile - 1) / kPolTile);
  if (!a.rounds_there)
    launch_pdl(!(a.mode & PARD_MODE_PATH_MASK) ? k_policy_terms<kAllPaths> : a.path_sums ? k_policy_terms<kMaskAtHand> : k_policy_terms<kMaskStaged>,
             tiles, kPolThreads, 0, stream, a);
  PARD_CUDA_OK(cudaGetLastError());
  const uint32_t per = a.n / a.n_seg;
  const bool copies = per >= kWalkCopiesLong && a.n_seg <= (uint32_t)sms;
  if (per >= kWalkClusterLong / 2 && a.n_seg <= (uint32_t)(kWalkClusterRounds * sms / kWalkCtas) && !(a.mode & PARD_MODE_SCAN) && cluster_walk_fits())
    PARD_CUDA_OK(launch_pdl_cluster(k_policy_walk<kWalkWarps, kWalkCtas, true>, a.n_seg * kWalkCtas, kWalkWarps * 32, sizeof(FeedSmem), kWalkCtas, stream, a));
  else if (per >= kWalkLong)
    launch_pdl(copies ? k_policy_walk<kWalkWarps, 1, true> : k_policy_walk<kWalkWarps, 1, false>, a.n_seg, kWalkWarps * 32, copies ? sizeof(FeedSmem) : 0, stream, a);
  else
    launch_pdl(k_policy_walk<1, 1, false>, (a.n_seg + kPolThreads / 32 - 1) / (kPolThreads / 32), kPolThreads, 0, stream, a);
  return cudaGetLastError() == cudaSuccess ? PARD_OK : PARD_ECUDA;
}

int launch_policy_emit(const PolicyArgs& a, cudaStream_t stream) {
  const uint32_t tiles = (uint32_t)(((uint64_t)a.n + kPolTile - 1) / kPolTile);
  launch_pdl(a.rounds_there ? k_policy_emit<kAllPaths, true> : !(a.mode & PARD_MODE_PATH_MASK) ? k_policy_emit<kAllPaths> : a.path_sums ? k_policy_emit<kMaskAtHand> : k_policy_emit<kMaskStaged>,
             tiles, kPolThreads, 0, stream, a);
  return cudaGetLastError() == cudaSuccess ? PARD_OK : PARD_ECUDA;
}

}  // namespace pard_plan_detail
