/* Declarations shared by the translation units that make up pard_plan: the
 * workspace header, the per-call pipeline table and a few arithmetic helpers. */
#ifndef PARD_PLAN_INTERNAL_CUH_
#define PARD_PLAN_INTERNAL_CUH_

#include <memory>
#include <new>

#include "pard_internal.h"

namespace pard_plan_detail {

constexpr int kMaxPasses = 8;
constexpr int kBins = 256;
constexpr uint32_t kUClamp = (1u << 30) - 1;       /* >= any request count      */
constexpr uint32_t kMaxPipelinesPerCall = 65536;
constexpr uint32_t kSegNarrow = 1u;                /* bits of PardSegConst::narrow */
constexpr uint32_t kSegNoStage = 2u;
constexpr uint32_t kSegHighFirst = 4u;
constexpr uint32_t kFoldSegs = 1024;              /* up to this many queues the constants are worked out beside the prepass */
constexpr uint32_t kFoldCtx = 1024;               /* up to this many contexts the key width is found by the last block of another kernel */
constexpr uint32_t kHistSegs = 64;                /* up to this many queues the batch-window tables are counted, not searched */
constexpr uint32_t kHistCap = 8192;               /* window-table entries a counted table may have in all */
constexpr uint32_t kSpinLimit = 1u << 18;          /* polling rounds (about a microsecond each) before giving up */

constexpr int kSortThreads = 512;
constexpr int kLoWarps = 8;                        /* warps 0..7 also do the look-back (one thread per digit) */
constexpr int kItemsLo = 10, kItemsHi = 22;        /* rounds of 32 elements per warp: look-back warps / others (measured best) */
constexpr int kSortTile = 32 * (kLoWarps * kItemsLo + (kSortThreads / 32 - kLoWarps) * kItemsHi);
constexpr int kSmallLo = 6, kSmallHi = 12;         /* the same for the tiles of calls that do not fill the device: at most */
constexpr uint32_t kSmallTile = 256 * (kSmallLo + kSmallHi), kSmallLeast = 8;    /* 4,608 elements, at least 2,048 */
constexpr uint32_t kResidentTiles = 296;           /* tiles in flight on the full chip: two blocks per multiprocessor */
constexpr int kLookGroup = 16;                     /* tiles whose counts are added up before the walk back */
constexpr int kDecThreads = 128;                   /* small blocks: a short tail when the grid drains (measured against 64 and 256) */
constexpr int kDecItems = 8;
constexpr int kDecTile = kDecThreads * kDecItems;
constexpr int kCompactChunk = 1024;                /* indices moved by one warp of kept_move_jobs */
constexpr int kLookBatch = 8;                      /* earlier tiles inspected per round trip in the sort */

/* look-back word of the sort: [31:30] state, [29:0] count */
constexpr uint32_t kLbAgg = 1u << 30;
constexpr uint32_t kLbIncl = 2u << 30;
constexpr uint32_t kLbMask = (1u << 30) - 1;

struct PlanHeader {
  uint32_t status;            /* 0, or the positive value of a pard_status */
  uint32_t dbits;             /* bits of the widest per-ctx deadline span  */
  uint32_t keybits;           /* segment bits + dbits                      */
  uint32_t npass;             /* radix passes that run                     */
  unsigned long long span_max;
  unsigned long long win_total;   /* window-table entries asked for (64 bits: 2^24 queues of up to 4,097 entries) */
  uint32_t ticket[kMaxPasses + 1];
  uint32_t wide;              /* 1: segment, deadline and index bits exceed 64; nothing is sorted */
  uint32_t use_scan;          /* 1: too many batch windows for the window tables: decide by scanning */
  uint32_t aborted;           /* 1: a bounded wait ran out; the sort is incomplete and every later kernel returns */
  uint32_t win_done;          /* blocks of k_windows that have finished */
  uint32_t seg_done;          /* blocks of k_seg_const (k_prepass) that have finished */
  uint32_t unsorted;          /* 1: some request's ctx is smaller than its predecessor's */
  uint32_t ctx_too_big;       /* 1: some ctx holds more requests than one sort tile */
  uint32_t bad_input;         /* 1: PARD_EDATA was found (kept apart from `status`, which holds the first error only) */
  uint32_t scan_ticket[2];    /* k_scan_path: runs of tiles taken, in the aggregates' step and in the decision's */
  uint32_t scan_done[2];      /* runs finished */
  uint32_t scan_flag[2];      /* 1: the one-block step behind it is done */
  uint32_t pshift;            /* low bits of the key that need no pass: the deadline field, when the requests come in its order */
  uint32_t time_steps_back;   /* 1: some request's deadline lies before its predecessor's */
  uint32_t pair_steps_back;   /* 1: some request's (ctx, deadline) lies before its predecessor's */
  uint32_t lookup;            /* 1: the elements hold no deadline: it has to be looked up in the request array */
  uint32_t sort_bar[kMaxPasses]; /* tiles of each of k_sort_rest's passes that are finished */
  uint32_t direct;            /* 1: the requests came in order, the plan is made without a sort (pard_direct.cuh) */
  uint32_t direct_off;        /* not 0: they did not, or something else that path does not take (kDirOff, kDirSteps) */
  uint32_t direct_done;       /* blocks of k_dir_count that have finished */
  uint32_t direct_ticket;     /* pieces taken by k_dir_emit */
  uint32_t walk_late;         /* 1: a wait of the rules' walk ran out: `aborted` for the kernels behind it (its own blocks go on together) */
  uint32_t pad[64 - 31 - kMaxPasses - (kMaxPasses + 1)];
};
static_assert(sizeof(PlanHeader) == 256, "header is 256 bytes");

__device__ __forceinline__ void set_status(PlanHeader* hdr, int status) {
  if (status == PARD_EDATA) hdr->bad_input = 1;
  atomicCAS(&hdr->status, 0u, (uint32_t)(-status));
}

/* A bounded wait ran out: the elements are only partly sorted from here on, so nothing after
 * this may use them as indices. */
__device__ __forceinline__ void set_aborted(PlanHeader* hdr) {
  hdr->aborted = 1;
  __threadfence();
  atomicExch(&hdr->status, (uint32_t)(-PARD_ETIMEOUT));
}

/* The device tables of the call's pipelines: handed over inside the kernel arguments when there are few
 * (no copy to enqueue, which also holds the first kernel up), else through a table in the workspace.
 * Every launch that needs the table carries all of it, whatever the call uses.  With 256 entries, 2 KB, 256
 * pipelines cost a grouped call of 256 k requests 43.5 us and of 5.1 M 154.9 us, copied 46.0 and 158.4 (257
 * of them, copied: 45.7 and 159.8).  512 entries, 4 KB: 257 pipelines 43.8 us, but a call of one pipeline
 * that needs no table pays: 96 epochs 35.4 -> 36.1 us, one small queue 41.0 -> 42.8 us. */
constexpr int kFewPipelines = 256;
struct PipeTable {
  const PardPipeDev* few[kFewPipelines];
  const PardPipeDev* const* many;
};

/* Fills the table for a call whose pipelines have been checked; d_many: room for their addresses in
 * the workspace, used when they do not fit the arguments. */
inline int pard_pipe_table(const pard_pipeline_t* const* pipelines, uint32_t n_pipelines, void* d_many, cudaStream_t stream,
                           PipeTable* out) {
  out->many = (const PardPipeDev* const*)d_many;
  if (n_pipelines <= (uint32_t)kFewPipelines) {
    for (uint32_t i = 0; i < (uint32_t)kFewPipelines; ++i)
      out->few[i] = i < n_pipelines ? (const PardPipeDev*)pipelines[i]->d_blob : nullptr;
    return PARD_OK;
  }
  std::unique_ptr<const PardPipeDev*[]> h(new (std::nothrow) const PardPipeDev*[n_pipelines]);
  if (!h) return PARD_ENOMEM;
  for (uint32_t i = 0; i < n_pipelines; ++i) h[i] = (const PardPipeDev*)pipelines[i]->d_blob;
  PARD_CUDA_OK(cudaMemcpyAsync(d_many, h.get(), 8ull * n_pipelines, cudaMemcpyHostToDevice, stream));
  return PARD_OK;
}

/* floor(2^64 / d) + 1 for d >= 2 */
__device__ __forceinline__ unsigned long long magic64(unsigned long long d) {
  unsigned long long q = ~0ull / d;
  if (~0ull % d == d - 1) ++q;          /* d divides 2^64 */
  return q + 1;
}

/* Whether a queue's constants allow 32-bit arithmetic against deadline offsets below 2^29.  Towards early
 * deadlines A may lie any distance away: a queue booked far ahead has late requests only, which narrow_A
 * keeps as they are.  (With a limit on that side too, one such queue among 16 sent a call of 2^24 requests
 * through the packing loop of 64-bit words, 517 -> 543 us.) */
__device__ __forceinline__ bool fits_narrow(uint64_t d_magic, int64_t d, int64_t A_rel, bool high_first) {
  const int64_t lim = (int64_t)1 << 29;
  return d_magic != 0 && d < ((int64_t)1 << 31) && (high_first ? A_rel < lim : A_rel > -lim);
}
/* A_rel of such a queue in 32 bits: cut off where every offset is late */
__device__ __forceinline__ int32_t narrow_A(const PardSegConst& K) {
  if (K.narrow & kSegHighFirst) return K.A_rel < 0 ? -1 : (int32_t)K.A_rel;
  return K.A_rel > (1ll << 29) ? 1 << 29 : (int32_t)K.A_rel;
}

/* The constants of all queues of ctx c, by one block: threads over the stages, then over the (stage,
 * downstream path) slots, then over the stages again.  dmin / dmax: smallest and largest deadline of
 * the ctx, the origins of the queues' deadline offsets.  True in the threads that met an input out
 * of range.  Bound by dependent loads (pipeline -> profile offsets -> durations; slot -> path ->
 * durations): with the durations of all stages fetched side by side first, a path costs one load
 * per stage instead of a chain of three.  One warp per queue that walked its paths on its own took
 * 10 us for 16 queues and 37 us for 32,768.  AHEAD: a thread requests what belongs to its own stage and slot at once
 * (9.0 -> 7.0 us for the constants of one ctx; not in k_plan_local, which has no registers left for it: 4,096 epochs
 * 391 -> 395 us).  BAR: by the threads from first_thread on, with a barrier of their own.  sums: the ctx's rows of PolicyArgs::path_sums, or null. */
constexpr int kMaskPaths = 16;                     /* bits of pard_request_t.flags: paths of a stage that a request can name */
constexpr int kConstThreads = 64;                  /* k_seg_const's blocks; any number of threads will do */
struct CtxScratch {
  long long delay[PARD_MAX_STAGES];                /* q_i + d_i(B_i), -1: out of range */
  long long dur[PARD_MAX_STAGES];                  /* d_i(B_i); d_i(1) for a batch size out of range */
  unsigned long long lsub[PARD_MAX_STAGES];
  int32_t slot_off[PARD_MAX_STAGES + 1];
};
template <bool AHEAD, int BAR = 0>
__device__ __forceinline__ bool ctx_constants(const PipeTable& pipes, uint32_t n_pipelines, const pard_queue_state_t& st, uint32_t c,
                                              unsigned long long dmin, unsigned long long dmax, PardSegConst* K_out,
                                              CtxScratch& sc, long long* sums = nullptr, uint32_t first_thread = 0) {
  const uint32_t S = (uint32_t)st.stage_stride, tid = threadIdx.x - first_thread, nt = blockDim.x - first_thread;
  auto sync = [&]() {
    if (BAR) asm volatile("bar.sync %0, %1;" :: "n"(BAR), "r"(nt) : "memory");
    else __syncthreads();
  };
  const int32_t pi = st.d_pipeline_of_ctx ? st.d_pipeline_of_ctx[c] : 0;
  /* a thread's own stage and slot: all that does not hang on the pipeline, requested at once */
  int32_t B_own = 1, m_own = 1;
  int64_t q_own = 0, fa_own = 0, w_own = 0, now_own = 0;
  bool high_own = false;
  if (AHEAD) {
    now_own = st.d_now_us[c];
    if (tid < S) {
      const size_t at = (size_t)c * S + tid;
      B_own = st.d_batch[at];
      q_own = st.d_q_us[at];
      fa_own = st.d_free_at_us[at];
      if (st.d_workers) m_own = st.d_workers[at];
      if (st.d_priority) high_own = st.d_priority[at] != 0;
    }
    if (st.d_w_us && tid < (uint32_t)st.slot_stride) w_own = st.d_w_us[(size_t)c * st.slot_stride + tid];
  }
  const PardPipeDev* p = nullptr;
  if (pi >= 0 && (uint32_t)pi < n_pipelines) p = n_pipelines <= (uint32_t)kFewPipelines ? pipes.few[pi] : pipes.many[pi];
  bool bad = p == nullptr;
  PardPipeDev head = {};
  if (AHEAD && p) head = *p;
  const PardPipeDev* const P = AHEAD ? &head : p;
  const uint32_t stages = p ? (uint32_t)P->n_stages : 0u;   /* <= S: checked on the host */
  const int32_t n_slots = p ? P->n_slots : 0;
  const size_t row = (size_t)c * S;
  int32_t e0_own = 0, e1_own = 0;
  if (AHEAD && (int32_t)tid < n_slots) { e0_own = P->path_off[tid]; e1_own = P->path_off[tid + 1]; }
  for (uint32_t k = tid; k < stages; k += nt) {
    const bool own = AHEAD && k == tid;
    const int32_t B = own ? B_own : st.d_batch[row + k];
    const int64_t q = own ? q_own : st.d_q_us[row + k];
    const bool ok = B >= 1 && B <= P->bmax[k];
    const long long d = P->lat_us[P->lat_offsets[k] + (ok ? B : 1) - 1];
    sc.dur[k] = d;
    sc.delay[k] = ok && q >= 0 && q < PARD_TIME_LIMIT_US ? q + d : -1;
    sc.lsub[k] = 0;
    sc.slot_off[k] = P->stage_slot_off[k];
  }
  sync();
  for (int32_t s = (int32_t)tid; s < n_slots; s += (int32_t)nt) {
    const bool own = AHEAD && s == (int32_t)tid;
    int64_t acc = own ? w_own : st.d_w_us ? st.d_w_us[(size_t)c * st.slot_stride + s] : 0;
    if (acc < 0 || acc >= PARD_TIME_LIMIT_US) { bad = true; acc = 0; }
    const int32_t e1 = own ? e1_own : P->path_off[s + 1];
    for (int32_t e = own ? e0_own : P->path_off[s]; e < e1; ++e) {
      const long long t = sc.delay[P->path_stage[e]];
      if (t < 0) bad = true;
      else acc += t;
    }
    uint32_t lo = 0, hi = stages;                  /* the slot's stage: the last whose slots begin at or before s */
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) / 2;
      if (sc.slot_off[mid] <= s) lo = mid; else hi = mid;
    }
    atomicMax(&sc.lsub[lo], (unsigned long long)acc);      /* maximum over the stage's paths; a sink has none: 0 */
    const int32_t j = s - sc.slot_off[lo];
    if (sums && j < kMaskPaths) sums[lo * kMaskPaths + j] = acc;
  }
  sync();
  for (uint32_t k = tid; k < S; k += nt) {
    PardSegConst out;
    out.A = 0; out.A_rel = 0; out.d = 1; out.cap = 1; out.d_magic = 0; out.cap_magic = 0;
    out.narrow = 0; out.lsub = 0; out.dsum = 1;
    if (sums && k < stages)                        /* paths the stage does not have */
      for (int32_t j = (k + 1 < stages ? sc.slot_off[k + 1] : n_slots) - sc.slot_off[k]; j < kMaskPaths; ++j) sums[k * kMaskPaths + j] = -1;
    if (p && k >= stages) {
      out.narrow = kSegNoStage;                    /* no such stage: a request found in this queue is an input error */
    } else if (p) {
      const bool own = AHEAD && k == tid;
      const int32_t B = own ? B_own : st.d_batch[row + k];
      const int64_t now = AHEAD ? now_own : st.d_now_us[c];
      const int64_t m = own ? m_own : st.d_workers ? st.d_workers[row + k] : 1;
      const int64_t fa = own ? fa_own : st.d_free_at_us[row + k];
      if (B < 1 || B > P->bmax[k] || m < 1 || now < 0 || now >= PARD_TIME_LIMIT_US || fa < 0 || fa >= PARD_TIME_LIMIT_US) {
        bad = true;
      } else {
        const int64_t d = sc.dur[k], lsub = (int64_t)sc.lsub[k], base = now > fa ? now : fa, cap = (int64_t)B * m;
        out.d = d;
        out.cap = (uint32_t)(cap > (int64_t)(1u << 30) ? (int64_t)(1u << 30) : cap);
        out.A = base + d + lsub;
        /* A against the origin of the queue's deadline offsets: offsets count up from the ctx's
         * smallest deadline, or, for a queue served high budget first, down from its largest */
        const bool high_first = own ? high_own : st.d_priority && st.d_priority[row + k] != 0;
        out.A_rel = high_first ? (int64_t)dmax - out.A : out.A - (int64_t)dmin;
        out.d_magic = (d >= 2 && d < ((int64_t)1 << 32)) ? magic64((uint64_t)d) : 0;
        out.cap_magic = out.cap >= 2 ? magic64(out.cap) : 0;
        out.narrow = fits_narrow(out.d_magic, d, out.A_rel, high_first) ? kSegNarrow : 0u;
        if (high_first) out.narrow |= kSegHighFirst;
        out.lsub = lsub;
        /* all stages' durations at their current batch sizes, for the rule that splits the objective
         * in proportion to them */
        long long dsum = 0;
        for (uint32_t i = 0; i < stages; ++i) dsum += sc.dur[i];
        out.dsum = dsum;
      }
    }
    K_out[k] = out;
  }
  return bad;
}

/* floor(x / d) for 32-bit x, with M = floor(2^64 / d) + 1 (d >= 2): exact
 * whenever x * d < 2^64, i.e. for every 32-bit x and d */
__device__ __forceinline__ uint32_t div_magic32(uint32_t x, unsigned long long M) {
  unsigned long long p0 = (unsigned long long)x * (uint32_t)M;
  unsigned long long p1 = (unsigned long long)x * (uint32_t)(M >> 32) + (p0 >> 32);
  return (uint32_t)(p1 >> 32);
}

__device__ __forceinline__ uint32_t threshold_u(int64_t X, const PardSegConst& K) {
  /* number of requests that may be admitted ahead of or at this one while it
   * still completes by its deadline: 0 if even position 0 is late, else
   * cap * (floor(X / d) + 1), saturated */
  if (X < 0) return 0;
  unsigned long long q;
  if (((unsigned long long)X >> 32) == 0 && K.d_magic)
    q = div_magic32((uint32_t)X, K.d_magic);
  else
    q = (unsigned long long)X / (unsigned long long)K.d;    /* d == 1 or operands beyond 32 bits */
  if (q >= kUClamp) return kUClamp;
  unsigned long long u = (q + 1) * K.cap;
  return u > kUClamp ? kUClamp : (uint32_t)u;
}

/* number of batch rounds b for which a request still fits, b < v: Nexus tests "base + b*d + d <= D" */
__device__ __forceinline__ uint32_t rounds_fit(long long X, unsigned long long magic, unsigned long long d) {
  if (X < 0) return 0;
  unsigned long long q;
  if (((unsigned long long)X >> 32) == 0 && magic) q = div_magic32((uint32_t)X, magic);
  else q = (unsigned long long)X / d;
  return q >= kUClamp ? kUClamp : (uint32_t)q + 1;
}

/* X = deadline - A of a request from its deadline offset: offsets of a queue served high
 * budget first count down from the ctx's largest deadline, and A_rel is that deadline - A */
__device__ __forceinline__ long long slack_of(unsigned long long off, const PardSegConst& K) {
  return (K.narrow & kSegHighFirst) ? K.A_rel - (long long)off : (long long)off - K.A_rel;
}

/* 32 bytes with one access, from the scratch (p 32-byte aligned) */
__device__ __forceinline__ void load4(const unsigned long long* p, unsigned long long* v) {
  asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];"
               : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(p));
}
/* 32 bytes of an output, which the caller may have put on a 16-byte boundary: with one access, or with two */
__device__ __forceinline__ void store4(void* p, unsigned long long a, unsigned long long b,
                                       unsigned long long c, unsigned long long d) {
  if (((uintptr_t)p & 31) == 0) {
    asm volatile("st.global.v4.u64 [%0], {%1, %2, %3, %4};" :: "l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
  } else {
    asm volatile("st.global.v2.u64 [%0], {%1, %2};" :: "l"(p), "l"(a), "l"(b) : "memory");
    asm volatile("st.global.v2.u64 [%0+16], {%1, %2};" :: "l"(p), "l"(c), "l"(d) : "memory");
  }
}

/* `count` elements of 8 bytes, `ahead` of them behind `from` in an array of n, on their way into L2 before the block
 * that will work on them asks for them, by one thread: a block's loads then wait for L2 instead of memory.  Blocks
 * are placed in the order of their tiles, so a tile's load phase comes about as many tiles later as are placed in
 * the meantime.  At 2^24 requests (us per call; before: 528): sort passes 16 tiles ahead (of 296 in flight) 512,
 * 32 ahead 513, 120 ahead 516, 296 ahead 521; the decision 600 tiles ahead another 4 (300 and 2,400: 2).  Not for
 * arrays that are in L2 as they were written or read before: 9 M elements 332 -> 320 us a call, 4 M 311 -> 313. */
constexpr uint64_t kAheadFrom = (48ull << 20) / 8;
__device__ __forceinline__ void l2_ahead(const unsigned long long* src, uint64_t from, uint64_t ahead, uint32_t count, uint64_t n) {
  if (n > kAheadFrom && count && from + ahead + count <= n)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(src + from + ahead), "r"(count * 8) : "memory");
}
constexpr uint32_t kSortAhead = 16, kDecAhead = 600;    /* tiles of kSortTile and of kDecTile */

/* loads and stores of look-back words: relaxed, device scope (other blocks write them) */
__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}

/* Copies into shared memory that report to an mbarrier (one arrival per phase).  All 16-byte aligned, the size a
 * multiple of 16. */
__device__ __forceinline__ void bulk_init(unsigned long long* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"((uint32_t)__cvta_generic_to_shared(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void bulk_fetch(unsigned long long* bar, void* dst, const void* src, uint32_t bytes) {
  const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar), d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(b), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               :: "r"(d), "l"(src), "r"(bytes), "r"(b) : "memory");
}
/* false: the copy has not arrived within about a second */
__device__ __forceinline__ bool bulk_arrived(unsigned long long* bar, uint32_t parity) {
  const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
  for (uint32_t spins = 0; spins < 1u << 18; ++spins) {
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(b), "r"(parity) : "memory");
    if (done) return true;
  }
  return false;
}

struct SegVal {            /* value of a segmented running reduction */
  int32_t m;               /* admitted mode: minimum of u_t - t; raw mode: number of kept requests;
                              over the elements since the last queue head (or since the span's start) */
  uint32_t head;           /* a queue head lies inside the span */
};

template <bool RAW>
__device__ __forceinline__ SegVal seg_identity() {
  SegVal a;
  a.m = RAW ? 0 : 0x7fffffff;
  a.head = 0;
  return a;
}

template <bool RAW>
__device__ __forceinline__ SegVal seg_combine(SegVal left, SegVal right) {
  SegVal r;
  r.m = right.head ? right.m : (RAW ? left.m + right.m : min(left.m, right.m));
  r.head = left.head | right.head;
  return r;
}

/* Inclusive segmented warp scan of the threads' values (in lane order). */
template <bool RAW>
__device__ __forceinline__ SegVal warp_scan(SegVal v, uint32_t lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    SegVal l;
    l.m = __shfl_up_sync(0xffffffffu, v.m, o);
    l.head = __shfl_up_sync(0xffffffffu, v.head, o);
    if (lane >= (uint32_t)o) v = seg_combine<RAW>(l, v);
  }
  return v;
}

constexpr int32_t kWinInf = 0x7fffffff;

/* u of window b (the saturation of threshold_u) */
__device__ __forceinline__ uint32_t win_u(uint32_t b, uint32_t cap) {
  const unsigned long long u = (unsigned long long)(b + 1) * cap;
  return u > kUClamp ? kUClamp : (uint32_t)u;
}

/* The first request whose ctx is >= c, by one warp's 32-ary search, into ctx_start[c].  That the
 * boundaries never step back and the ranges cover all requests is checked here; the planner's
 * blocks check that their ranges hold requests of their ctx only: both together prove the grouping. */
__device__ __forceinline__ void ctx_range_search(const uint4* __restrict__ req, uint32_t n, uint32_t n_ctx, uint32_t c,
                                                 uint32_t* __restrict__ ctx_start, PlanHeader* hdr, uint32_t limit) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t lo[2] = {0, 0}, hi[2] = {n, n};       /* first request whose ctx is >= c, >= c + 1 */
  while (lo[0] < hi[0] || lo[1] < hi[1]) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (lo[q] < hi[q]) {                       /* uniform across the warp */
        const uint32_t span = hi[q] - lo[q];
        const uint32_t p = lo[q] + (uint32_t)(((unsigned long long)(lane + 1) * span) / 33u);   /* lo <= p < hi */
        const bool less = __ldg(&req[p]).z < c + q;
        const uint32_t k = __popc(__ballot_sync(0xffffffffu, less));
        const uint32_t p_below = __shfl_sync(0xffffffffu, p, k > 0 ? k - 1 : 0);
        const uint32_t p_at = __shfl_sync(0xffffffffu, p, k < 32 ? k : 31);
        if (k > 0) lo[q] = p_below + 1;
        if (k < 32) hi[q] = p_at;
      }
    }
  }
  if (lane != 0) return;
  ctx_start[c] = lo[0];
  if (c == n_ctx && lo[0] != n) hdr->unsorted = 1;      /* requests past the last ctx's range (ctx out of range) */
  if (c < n_ctx) {
    if (lo[1] < lo[0]) hdr->unsorted = 1;
    else if (lo[1] - lo[0] > limit) hdr->ctx_too_big = 1;
  }
}

/* ---- one block plans one ctx (pard_local.cu) ---- */
constexpr uint32_t kLocalTile = 8192;             /* requests of one ctx a block can take */
struct LocalArgs {
  const uint4* req;
  const uint32_t* ctx_start;       /* NULL: the call has one ctx */
  uint32_t n, n_ctx, ibits, force_scan;
  PipeTable pipes;
  uint32_t n_pipelines;
  pard_queue_state_t st;
  uint8_t* out_keep;
  long long* out_est;
  uint32_t* out_perm;
  uint32_t* out_kept_idx;
  unsigned long long* out_n_kept;
  uint32_t* out_seg_off;
  uint32_t* out_seg_kept;
  const PardSegConst* ktab;        /* several ctx: the queues' constants, from k_ctx_prep */
  uint32_t* kept_words;            /* several ctx: look-back words over the ctxs' kept counts, zero at the start */
  uint32_t* kept_tmp;
  PardTicket answer;               /* the call's only kernel, and its caller waits: the status goes out from here */
};
int allow_local_smem();            /* once per device, by the planner's set-up */
int launch_ctx_prep(const LocalArgs& a, PardSegConst* ktab, uint32_t* ctx_start, PlanHeader* hdr, cudaStream_t stream);
int launch_plan_local(const LocalArgs& a, PlanHeader* hdr, bool raw, cudaStream_t stream);

/* Decision by a sequential walk of every queue (requests whose downstream path is known, arrival
 * order, the Nexus and Clipper++ rules): defined in pard_policy.cu, enqueued by pard_plan after
 * the sort and the queue boundaries.  The sorted elements are in buf_b when hdr->npass is odd,
 * else in buf_a; the other buffer (8 bytes per request) is free by then and serves as scratch. */
struct PolicyArgs {
  PlanHeader* hdr;
  unsigned long long* buf_a;
  unsigned long long* buf_b;
  uint32_t n, ibits, n_seg, mode;
  const PardSegConst* ktab;
  const uint32_t* seg_off;
  const uint4* req;
  const pard_arrival_t* arrivals;
  PipeTable pipes;
  uint32_t n_pipelines;
  pard_queue_state_t st;
  uint32_t* rounds;               /* [n_seg] batch rounds the walk has closed */
  uint32_t* tail;                 /* [n_seg] Nexus: requests of the last, partly filled window */
  uint32_t* tile_x;               /* [tiles of kDecTile] kept requests ahead of the tile's first one, in its queue */
  uint8_t* out_keep;
  long long* out_est;
  uint32_t* out_perm;
  uint32_t* out_kept_idx;
  const long long* path_sums;     /* [n_seg][kMaskPaths] Eq. 3 along every path a request can name, -1: no such path; or null */
  const uint32_t* kept_base;      /* [n_seg] output offset of every queue's survivors, known after the walk */
  uint32_t* seg_kept;
  uint32_t rounds_there;          /* the sort has written every request's rounds (k_sort_requests) */
};
int allow_walk_smem();             /* once per device, by the planner's set-up */
/* thresholds and walk: every queue's rounds and kept count (seg_kept) */
int launch_policy_walk(const PolicyArgs& a, int sms, cudaStream_t stream);
/* estimates, flags, order and survivors, once the output offsets are known */
int launch_policy_emit(const PolicyArgs& a, cudaStream_t stream);

}  // namespace pard_plan_detail

#endif  /* PARD_PLAN_INTERNAL_CUH_ */
