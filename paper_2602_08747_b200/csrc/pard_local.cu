/* One block plans one ctx from start to end.
 *
 * For calls whose requests come grouped by ascending ctx with no ctx above 8,192 requests -- one
 * module's queue planned every few milliseconds, or thousands of decision epochs in one call -- a
 * block does the whole job for "its" ctx without leaving shared memory:
 *   1. reads the ctx's requests once into registers; deadline range, input checks, and whether the
 *      deadlines ever step back;
 *   2. gets the constants of the ctx's queues (Eq. 3);
 *   3. sorts (stage | deadline offset | index) in shared memory -- by the stage alone when the
 *      deadlines are in order already (arrival order, one objective), for up to 16 stages a
 *      counting sort in registers;
 *   4. finds the batch-window tables (see pard_plan.cu) in the sorted elements: an element whose
 *      window differs from its neighbour's knows the P of the windows between them;
 *   5. the tables give every queue's kept count, a look-back over the ctxs before gives the place of
 *      the ctx's survivors in the output;
 *   6. decides every request on its own and writes the outputs.
 * 16 bytes are read and 13 + 4f written per request and nothing else touches global memory.
 * Queues with more windows than the block's tables hold are decided by the segmented prefix-min
 * scan over the elements instead.
 * Bound by instructions (half of the issue slots, integer ones at half rate) and the chain of steps between barriers, two
 * blocks per multiprocessor covering for each other: of 297 us for 4,096 contexts of 8,192 requests (1.0 GB: 155 us at the
 * copy bandwidth) 86 go to the requests, 74 to the counting sort, 30 to the tables, 87 to the outputs and 20 to the
 * survivors.  Every request's window and position on its own, 32 in a row to a warp: 345; two segmented scans instead of
 * tables took 762, three radix passes without a look at the order 865. */
#include <cstddef>

#include "pard_plan_internal.cuh"

using namespace pard_plan_detail;

namespace {

constexpr int kLocThreads = 512;
constexpr int kLocWarps = kLocThreads / 32;
constexpr int kLocItems = kLocalTile / kLocThreads;      /* rounds of 32 consecutive requests per warp */
static_assert(kLocItems == 16 && kLocItems * kLocThreads == kLocalTile, "16 items per thread");
constexpr uint32_t kTabEntries = 2048;                   /* window-table entries of one ctx */
constexpr uint32_t kNoWindow = 0xffffu;                  /* window of a request with deadline < A */
constexpr uint32_t kNoCtx = 0xffffffffu;

struct Tables {                                          /* 4. to 6., in the room of the sort's counters */
  uint32_t P[kTabEntries];                               /* requests of the queue in earlier windows */
  int32_t E[kTabEntries];                                /* min of u_t - t over them */
  uint32_t Kp[kTabEntries];                              /* raw positions: kept requests among them */
  uint16_t win[kLocalTile];                              /* windows of the sorted elements */
};

/* The usual ctx after its sort: nothing served high budget first, offsets and A within 31 bits, at most
 * 32 stages.  The elements fall apart into arrays, queue after queue; position p stands at p + lead, lead = the ctx's first
 * request modulo 8, so that a thread's groups of eight are those of the output. */
constexpr int kLocGroup = 8;
constexpr int32_t kFewWindows = 4;                       /* of a group, by eight comparisons each; more: request after request */
constexpr uint32_t kLocOneByOne = 1024;                  /* see finish_split */
struct Split {
  uint32_t off[kLocalTile + kLocGroup];                  /* deadline offsets */
  uint16_t idx[kLocalTile + kLocGroup];                  /* index inside the ctx */
  uint32_t P[kTabEntries];
  int2 QU[kTabEntries];                                  /* of a window: min(E, 1) - 1, or Kp for raw positions; u */
  uint16_t kept[kLocalTile];                             /* survivors, queue after queue */
};

/* Requests that come in order, on their way into the Split form: beside its off and idx. */
struct Ordered {
  uint32_t off[kLocalTile + kLocGroup];                  /* Split's */
  uint16_t idx[kLocalTile + kLocGroup];
  uint32_t D[kLocalTile];                                /* low words of the deadlines */
  uint8_t code[kLocalTile];                              /* four times the stage */
  uint16_t place[16][kLocThreads];                       /* [stage][thread]: first place of the thread's requests */
};

struct LocalSmem {
  unsigned long long keys[kLocalTile];
  union {
    struct {
      uint32_t slot[kLocWarps][kBins];                   /* running counts, then first place of every (warp, digit) */
      uint32_t match[kLocWarps][kBins];                  /* lanes currently holding the digit */
    };
    Tables tab;
    unsigned char room[sizeof(Ordered) - sizeof(unsigned long long) * kLocalTile];
  };
  PardSegConst K[PARD_MAX_STAGES];
  uint32_t stage_first[PARD_MAX_STAGES + 2];
  uint32_t stage_kept[PARD_MAX_STAGES];
  uint32_t kept_base[PARD_MAX_STAGES];
  uint32_t hb_kept[PARD_MAX_STAGES];                     /* high budget first: length of the kept prefix */
  uint32_t win_off[PARD_MAX_STAGES], win_cnt[PARD_MAX_STAGES];
  uint32_t scan[kLocWarps];
  uint32_t few[8][kLocWarps];
  unsigned long long red_min[kLocWarps], red_max[kLocWarps];
  int32_t wm[kLocWarps];
  uint32_t wh[kLocWarps];
  uint32_t ctx, first, cnt, flags, use_scan, kept, base, abort;
};

static_assert(sizeof(Ordered) <= offsetof(LocalSmem, K) && sizeof(Split) <= offsetof(LocalSmem, K), "inside keys and counters");

/* smallest of the warp's values, by the words */
__device__ __forceinline__ unsigned long long warp_min(unsigned long long x) {
  const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(x >> 32));
  return (unsigned long long)hi << 32 | __reduce_min_sync(0xffffffffu, (uint32_t)(x >> 32) == hi ? (uint32_t)x : 0xffffffffu);
}

/* a thread's sorted element, decoded */
struct Elem {
  uint32_t stage, idx, r;
  long long X;                                           /* deadline - A */
};

struct Format {                                          /* of the ctx's elements: stage | deadline offset | index */
  uint32_t ibits, dbits, imask;
  unsigned long long dmask;
};

__device__ __forceinline__ Elem decode(unsigned long long e, uint32_t pos, const LocalSmem& Sm, const Format& f) {
  Elem x;
  x.stage = (uint32_t)(e >> (f.ibits + f.dbits));
  x.idx = (uint32_t)e & f.imask;
  x.r = pos - Sm.stage_first[x.stage];
  x.X = slack_of((e >> f.ibits) & f.dmask, Sm.K[x.stage]);
  return x;
}

/* window of a request of a queue that has a table */
__device__ __forceinline__ uint32_t window_of(long long X, const PardSegConst& K) {
  if (X < 0) return kNoWindow;
  if (((unsigned long long)X >> 32) == 0 && K.d_magic) return div_magic32((uint32_t)X, K.d_magic);
  return (uint32_t)((unsigned long long)X / (unsigned long long)K.d);
}

/* 16-bit values of a thread's items, two to a register */
__device__ __forceinline__ void put16(uint32_t (&v)[kLocItems / 2], int i, uint32_t x) {
  v[i / 2] = (i & 1) ? (v[i / 2] & 0xffffu) | (x << 16) : x;
}
__device__ __forceinline__ uint32_t get16(const uint32_t (&v)[kLocItems / 2], int i) {
  return (i & 1) ? v[i / 2] >> 16 : v[i / 2] & 0xffffu;
}

/* One stable pass over 8 bits: ranks first -- the lanes that hold the same digit find each other
 * through a shared word (atomic OR), the warp's running count gives the rank inside the warp --,
 * then the counts of all warps become places, then the elements move.  Every warp's counters are
 * zero at the start and again at the end. */
__device__ __forceinline__ void pass_byte(unsigned long long (&key)[kLocItems], uint32_t shift, int items, LocalSmem& Sm, uint32_t tid,
                                          bool reload) {
  const uint32_t lane = tid & 31, warp = tid >> 5, lanebit = 1u << lane;
  uint32_t* slot = Sm.slot[warp];
  uint32_t* match = Sm.match[warp];
  uint32_t rank[kLocItems / 2];
#pragma unroll
  for (int i = 0; i < kLocItems; ++i) {
    if (i >= items) break;                               /* uniform */
    const uint32_t d = (uint32_t)(key[i] >> shift) & 255u;
    atomicOr(&match[d], lanebit);
    __syncwarp();
    const uint32_t grp = match[d], below = grp & (lanebit - 1), first = slot[d];
    __syncwarp();
    if (below == 0) {                                    /* lowest lane of the group */
      slot[d] = first + __popc(grp);
      match[d] = 0;
    }
    put16(rank, i, first + __popc(below));
    __syncwarp();
  }
  __syncthreads();
  uint32_t count = 0, x = 0;
  if (tid < kBins) {                                     /* thread d owns digit d */
#pragma unroll
    for (int w = 0; w < kLocWarps; ++w) count += Sm.slot[w][tid];
    x = count;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    if (lane == 31) Sm.scan[warp] = x;
  }
  __syncthreads();
  if (tid < kBins) {
    uint32_t place = x - count;
#pragma unroll
    for (int w = 0; w < kBins / 32; ++w)
      if (w < (int)warp) place += Sm.scan[w];
#pragma unroll
    for (int w = 0; w < kLocWarps; ++w) {
      const uint32_t t = Sm.slot[w][tid];
      Sm.slot[w][tid] = place;
      place += t;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kLocItems; ++i) {
    if (i >= items) break;
    Sm.keys[slot[(uint32_t)(key[i] >> shift) & 255u] + get16(rank, i)] = key[i];
  }
  __syncthreads();
  if (reload) {
    const uint32_t wfirst = warp * 32 * (uint32_t)items;
#pragma unroll
    for (int i = 0; i < kLocItems; ++i)
      if (i < items) key[i] = Sm.keys[wfirst + i * 32 + lane];
    for (uint32_t b = lane; b < kBins; b += 32) slot[b] = 0;
    __syncwarp();
  }
}

/* the codes of a thread's PER consecutive requests: 16, or 4 in contexts of up to 2,048 requests, so that every warp has
 * some (one of 141: 26.2 -> 22.5 us) */
template <int PER>
__device__ __forceinline__ uint4 load_codes(const Ordered& T, uint32_t tid) {
  if (PER == 16) return *reinterpret_cast<const uint4*>(&T.code[tid * 16]);
  return make_uint4(*reinterpret_cast<const uint32_t*>(&T.code[tid * 4]), 0u, 0u, 0u);
}

/* A stable counting sort by stage of requests that come in order: a thread owns 16 (in small contexts 4) consecutive
 * requests and counts its stages in half bytes of a register (of two, from nine stages on), which also yields every
 * request's rank among them (returned, four bits each); the counts, two to a word, are scanned over the block.  Bound by
 * instructions: with whole bytes 17 per request where this takes 7.  (By ballots, row after row, with ranks and deadlines
 * kept in registers: no fewer, and spilled.)  Leaves the queues' first positions in Sm.stage_first and the
 * thread's places in T.place. */
template <int HALVES, int PER>
__device__ __forceinline__ uint2 order_few(LocalSmem& Sm, Ordered& T, uint32_t cnt, uint32_t S) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t n[HALVES], ranks[2] = {0, 0};                 /* n: stages 0 to 7, 8 to 15; of the first 15 requests */
#pragma unroll
  for (int h = 0; h < HALVES; ++h) n[h] = 0;
  const uint32_t mine = cnt > tid * PER ? min(cnt - tid * PER, (uint32_t)PER) : 0u;
  uint32_t last[HALVES];                                 /* the sixteenth, apart: a count of 16 takes five bits */
#pragma unroll
  for (int h = 0; h < HALVES; ++h) last[h] = 0;
  if (mine) {
    const uint4 s = load_codes<PER>(T, tid);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      if (i >= (int)mine) break;
      const uint32_t w = i < 4 ? s.x : i < 8 ? s.y : i < 12 ? s.z : s.w;
      const uint32_t k4 = (w >> (8 * (i & 3))) & 63u;     /* four times the stage */
      const uint32_t sh = HALVES == 2 ? k4 & 31u : k4, inc = 1u << sh;
      const bool up = HALVES == 2 && k4 >= 32;
      ranks[i / 8] |= (((up ? n[HALVES - 1] : n[0]) >> sh) & 15u) << (4 * (i & 7));
      uint32_t* to = i < 15 ? n : last;
      if (HALVES == 1) to[0] += inc;
      else { to[0] += up ? 0u : inc; to[HALVES - 1] += up ? inc : 0u; }
    }
  }
  /* stages 8h + q and 8h + q + 4 in c[4h + q]; counts of at most 8,192 in 16 bits */
  uint32_t c[4 * HALVES], own[4 * HALVES];
#pragma unroll
  for (int h = 0; h < HALVES; ++h)
#pragma unroll
    for (int q = 0; q < 4; ++q) own[4 * h + q] = c[4 * h + q] = ((n[h] >> (4 * q)) & 0x000f000fu) + ((last[h] >> (4 * q)) & 0x000f000fu);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
#pragma unroll
    for (int q = 0; q < 4 * HALVES; ++q) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, c[q], o);
      if (lane >= (uint32_t)o) c[q] += y;
    }
  if (lane == 31)
#pragma unroll
    for (int q = 0; q < 4 * HALVES; ++q) Sm.few[q][warp] = c[q];
  __syncthreads();
  uint32_t run = 0;                                      /* first position of the stage at hand */
  uint32_t total[4 * HALVES];
#pragma unroll
  for (int q = 0; q < 4 * HALVES; ++q) {
    const uint32_t w = lane < (uint32_t)kLocWarps ? Sm.few[q][lane] : 0u;
    total[q] = __reduce_add_sync(0xffffffffu, w);
    c[q] += __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u) - own[q];     /* before this thread */
  }
#pragma unroll
  for (int k = 0; k < 8 * HALVES; ++k) {
    const int q = 4 * (k / 8) + (k & 3), sh = (k & 4) ? 16 : 0;
    T.place[k][tid] = (uint16_t)(run + ((c[q] >> sh) & 0xffffu));
    if (tid == 0 && k < (int)S) Sm.stage_first[k] = run;
    run += (total[q] >> sh) & 0xffffu;
  }
  if (tid == 0) Sm.stage_first[S] = cnt;
  __syncthreads();
  return make_uint2(ranks[0], ranks[1]);
}

/* the thread's own requests to their places */
template <int PER>
__device__ __forceinline__ void place_few(Ordered& T, uint32_t cnt, uint2 ranks, uint32_t lead, uint32_t dmin) {
  const uint32_t tid = threadIdx.x, p0 = tid * PER;
  if (p0 >= cnt) return;
  const bool whole = p0 + PER <= cnt;
  const uint4 s = load_codes<PER>(T, tid);
#pragma unroll
  for (int q = 0; q < PER / 4; ++q) {
    const uint4 x = *reinterpret_cast<const uint4*>(&T.D[p0 + 4 * q]);
    const uint32_t w = q == 0 ? s.x : q == 1 ? s.y : q == 2 ? s.z : s.w;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t pos = p0 + 4 * q + u, low = u == 0 ? x.x : u == 1 ? x.y : u == 2 ? x.z : x.w;
      const uint32_t at = lead + (&T.place[0][tid])[((w >> (8 * u)) & 63u) * (kLocThreads / 4)] + (((q < 2 ? ranks.x : ranks.y) >> (4 * ((4 * q + u) & 7))) & 15u);
      if (whole || pos < cnt) {
        T.off[at] = low - dmin;
        T.idx[at] = (uint16_t)pos;
      }
    }
  }
}

/* E and, for raw positions, Kp of one queue's table, by one warp; returns the queue's kept count,
 * which follows from the complete table: n - 1 + min(E, 1), or the running Kp. */
template <bool RAW>
__device__ uint32_t table_prefix(Tables& t, uint32_t off, uint32_t cnt, uint32_t cap, uint32_t lane) {
  uint32_t* P = t.P + off;
  const uint32_t P0 = P[0];
  int32_t e_carry = P0 > 0 ? -(int32_t)(P0 - 1) : kWinInf;       /* the requests with deadline < A: u = 0 */
  uint32_t k_carry = 0;
  if (lane == 0) { t.E[off] = e_carry; if (RAW) t.Kp[off] = 0; }
  for (uint32_t b0 = 0; b0 + 1 < cnt; b0 += 32) {                /* windows b0.. -> entries b0+1.. */
    const uint32_t b = b0 + lane;
    int32_t val = kWinInf;
    uint32_t kept = 0;
    if (b + 1 < cnt) {
      const uint32_t p = P[b], q = P[b + 1];
      if (q > p) {
        const uint32_t u = win_u(b, cap);
        val = (int32_t)u - (int32_t)(q - 1);
        if (RAW) { const uint32_t top = u < q ? u : q; kept = top > p ? top - p : 0; }
      }
    }
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t v2 = __shfl_up_sync(0xffffffffu, val, o);
      if (lane >= (uint32_t)o) val = min(val, v2);
      if (RAW) {
        const uint32_t k2 = __shfl_up_sync(0xffffffffu, kept, o);
        if (lane >= (uint32_t)o) kept += k2;
      }
    }
    const int32_t e_inc = min(e_carry, val);
    const uint32_t k_inc = k_carry + kept;
    if (b + 1 < cnt) { t.E[off + b + 1] = e_inc; if (RAW) t.Kp[off + b + 1] = k_inc; }
    e_carry = __shfl_sync(0xffffffffu, e_inc, 31);
    if (RAW) k_carry = __shfl_sync(0xffffffffu, k_inc, 31);
  }
  const uint32_t n_q = P[cnt - 1];
  return n_q == 0 ? 0u : (RAW ? k_carry : (uint32_t)((int32_t)n_q - 1 + min(e_carry, 1)));
}

/* Places of the survivors of the ctx's queues inside the ctx, the queues' kept counts to the caller, the
 * ctx's count to the blocks behind.  One warp. */
__device__ __forceinline__ void publish_kept(const LocalArgs& a, LocalSmem& Sm, uint32_t c, uint32_t lane) {
  const uint32_t S = (uint32_t)a.st.stage_stride;
  uint32_t run = 0;
  for (uint32_t k0 = 0; k0 < S; k0 += 32) {
    const uint32_t k = k0 + lane;
    const uint32_t v = k < S ? Sm.stage_kept[k] : 0u;
    uint32_t y = v;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= (uint32_t)o) y += z;
    }
    if (k < S) {
      Sm.kept_base[k] = run + y - v;
      if (a.out_seg_kept) a.out_seg_kept[(size_t)c * S + k] = v;
    }
    run += __shfl_sync(0xffffffffu, y, 31);
  }
  if (lane == 0) {
    Sm.kept = run;
    if (a.ctx_start) st_relaxed(a.kept_words + c, run | (c == 0 ? kLbIncl : kLbAgg));
  }
}

/* Kept requests of all ctxs before this one: ctxs are taken in ticket order, so a block only waits
 * for blocks that run already; 32 ctxs per round trip, bounded.  Called as late as possible: the
 * blocks in flight are mostly at the same point, and a block that asks right after publishing its own
 * count waits for the slowest of those before it (92 us of 468 at 4,096 ctxs). */
__device__ __forceinline__ bool look_back(PlanHeader* hdr, uint32_t* words, uint32_t c, uint32_t mine, uint32_t lane, uint32_t* before) {
  uint32_t sum = 0, spins = 0;
  int64_t t = (int64_t)c - 1;
  while (t >= 0) {
    const uint32_t v = t - (int64_t)lane >= 0 ? ld_relaxed(words + (t - lane)) : (uint32_t)kLbIncl;
    const uint32_t unset = __ballot_sync(0xffffffffu, (v >> 30) == 0), incl = __ballot_sync(0xffffffffu, (v & kLbIncl) != 0);
    const uint32_t stop = incl ? (uint32_t)__ffs(incl) : 32u;        /* lanes 0 .. stop-1 count */
    const uint32_t ready = unset ? (uint32_t)__ffs(unset) - 1 : 32u;
    const uint32_t use = min(stop, ready);
    sum += __reduce_add_sync(0xffffffffu, lane < use ? v & kLbMask : 0u);
    if (use == stop && incl) break;
    t -= use;
    if (use < 32) {
      if (++spins > kSpinLimit || ld_relaxed(&hdr->aborted)) return false;
      __nanosleep(40);
    }
  }
  if (lane == 0 && c > 0) st_relaxed(words + c, ((sum + mine) & kLbMask) | kLbIncl);
  *before = sum;
  return true;
}

/* The ctx's place in the list of survivors (one warp; the others wait).  False: a wait ran out, here or
 * in another block. */
__device__ __forceinline__ bool place_survivors(PlanHeader* __restrict__ hdr, const LocalArgs& a, LocalSmem& Sm, uint32_t c) {
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  if (tid < 32) {
    uint32_t before = 0;
    if (a.ctx_start && !look_back(hdr, a.kept_words, c, Sm.kept, lane, &before) && lane == 0) Sm.abort = 1;
    if (lane == 0) {
      Sm.base = before;
      if (c + 1 == a.n_ctx && a.out_n_kept) *a.out_n_kept = before + Sm.kept;
    }
  }
  __syncthreads();
  if (Sm.abort && tid == 0 && !ld_relaxed(&hdr->aborted)) {          /* the wait ran out (not: another block gave up) */
    hdr->aborted = 1;
    __threadfence();
    atomicExch(&hdr->status, (uint32_t)(-PARD_ETIMEOUT));
  }
  return Sm.abort == 0;
}

/* A_rel as this file keeps it.  A queue booked further ahead than its ctx's latest deadline, however far,
 * counts as booked one microsecond behind it: all its requests are late either way, and nothing but that
 * is read off A_rel then.  (One queue in five booked 36 minutes ahead, as a backlog carried from epoch to
 * epoch leaves them, kept four contexts of five out of the Split form: 4,096 epochs of 8,192 requests
 * 678 us, with this 358.) */
__device__ __forceinline__ int64_t booked_within(int64_t A_rel, unsigned long long span) {
  return A_rel > (int64_t)span ? (int64_t)span + 1 : A_rel;      /* span < 2^60 */
}

/* Whether the constants allow the Split form; by all threads. */
__device__ __forceinline__ bool split_fits(const LocalArgs& a, const LocalSmem& Sm, unsigned long long span) {
  const uint32_t S = (uint32_t)a.st.stage_stride, k = threadIdx.x;
  bool ok = S <= 32 && !a.st.d_priority && !a.force_scan && span < (1ull << 31) - 1;
  if (k < S) {
    const PardSegConst& K = Sm.K[k];
    const bool none = Sm.stage_first[k] == Sm.stage_first[k + 1];
    ok = ok && (none || (!(K.narrow & kSegNoStage) && K.d_magic != 0 && K.A_rel > -(1ll << 31)));
  }
  return __syncthreads_and(ok) != 0;
}

/* 4. to 6. in the Split form.  A thread takes groups of eight positions.  Windows only rise along a queue, so a group
 * whose neighbour ahead and whose last request are in one window is done with two divisions; along a window the
 * admitted position rises by one per request up to u, c = min(r + q, u) with q = min(E, 1) - 1 (at the window's first
 * request too: E is at most the u before less the requests ahead), so its survivors are the window's first ones and a
 * group's estimates are at most two when a batch round takes eight, for raw positions (c = r) too.  (Every request on its
 * own, 32 in a row to a warp: 218 instructions per request for 4,096 contexts of 8,192, 172 like this with the sort below;
 * calls 362 -> 321 us, raw positions 360 -> 318, rounds of one request 385 -> 334.)
 * The tables' P begin as zeros, written by all threads: a queue whose first request lies many windows on, as after a
 * pause or with rounds of a few requests, has its first windows done.  (By the thread of that request, eight comparisons
 * for each: 2,000 contexts of 1,000 requests in rounds of one 122 us, every request on its own 109, like this 94.)
 * Every request goes on its own where groups would leave most warps idle: up to kLocOneByOne requests, and up to twice as
 * many where a group meets more than a window on average (3,000 contexts of 800 in rounds of one, two objectives:
 * groups 227 us, like this 214; 2,000 of 1,500 173 and 166, by default rounds 161 as groups, 163 one by one) or there is one
 * ctx (less code to fetch when its caller's other work has taken the L2: 2,000 requests 39.9 -> 36.0 us; 4,000 would take
 * 33.7 instead of 30.8 with the code at hand).  False: more windows than the tables hold, nothing has been written. */
template <bool RAW>
__device__ __forceinline__ bool finish_split(PlanHeader* __restrict__ hdr, const LocalArgs& a, LocalSmem& Sm, uint32_t c, uint32_t first, uint32_t cnt) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t S = (uint32_t)a.st.stage_stride, lead = first % kLocGroup;
  Split& T = *reinterpret_cast<Split*>(Sm.keys);
  if (warp == 0) {                                       /* extents: windows up to every queue's last request */
    uint32_t w = 0;
    if (lane < S) {
      const uint32_t lo = Sm.stage_first[lane], hi = Sm.stage_first[lane + 1];
      const PardSegConst& K = Sm.K[lane];
      if (hi > lo) {
        const long long X = (long long)T.off[lead + hi - 1] - K.A_rel;
        w = X < 0 ? 1u : min(div_magic32((uint32_t)X, K.d_magic), kTabEntries) + 2u;
      }
    }
    uint32_t x = w;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t p = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += p;
    }
    if (lane < S) {
      Sm.win_off[lane] = x - w;
      Sm.win_cnt[lane] = w;
    }
    if (lane == 31) Sm.use_scan = x > kTabEntries ? 1u : 0u;
  } else {                                               /* no request ahead of a window: what holds up to a queue's first one */
    for (uint32_t e = tid - 32; e < kTabEntries / 4; e += kLocThreads - 32) reinterpret_cast<uint4*>(T.P)[e] = make_uint4(0u, 0u, 0u, 0u);
  }
  __syncthreads();
  if (Sm.use_scan) return false;
  if (tid < S && Sm.win_cnt[tid]) T.P[Sm.win_off[tid] + Sm.win_cnt[tid] - 1] = Sm.stage_first[tid + 1] - Sm.stage_first[tid];   /* the end marker */
  /* (The loops below move on by a request at least and look no further than a queue's table, so that they end whatever
   * the arrays hold.) */
  /* the queue of position p, the last that begins at or before it */
  auto queue_at = [&](uint32_t p) {
    uint32_t k = 0, z = S;
    while (z - k > 1) {
      const uint32_t mid = (k + z) / 2;
      if (Sm.stage_first[mid] <= p) k = mid; else z = mid;
    }
    return k;
  };
  const uint32_t end = lead + cnt, groups = cnt ? (end + kLocGroup - 1) / kLocGroup : 0u;   /* (an empty ctx: none) */
  const bool one_by_one = cnt <= kLocOneByOne || (cnt <= 2 * kLocOneByOne && (a.n_ctx == 1 || Sm.win_off[S - 1] + Sm.win_cnt[S - 1] > groups));
  if (one_by_one)
    for (uint32_t p = tid; p < cnt; p += kLocThreads) {
      const uint32_t k = queue_at(p), r = p - Sm.stage_first[k];
      const int32_t off = (int32_t)T.off[lead + p], A = (int32_t)Sm.K[k].A_rel;
      const unsigned long long magic = Sm.K[k].d_magic;
      const int32_t b = off < A ? -1 : (int32_t)div_magic32((uint32_t)off - (uint32_t)A, magic);
      int32_t e = b;                                     /* (up to a queue's first request: no request ahead) */
      if (r) {
        const int32_t before = (int32_t)T.off[lead + p - 1];
        e = before < A ? -1 : (int32_t)div_magic32((uint32_t)before - (uint32_t)A, magic);
      }
      while (e < b) T.P[Sm.win_off[k] + (uint32_t)++e] = r;
    }
  else
  for (uint32_t g = tid; g < groups; g += kLocThreads) {
    const uint32_t x0 = g * kLocGroup;
    uint32_t x = max(x0, lead);                          /* span after span of requests of one queue: mostly one */
    const uint32_t xe = min(x0 + kLocGroup, end);
    while (x < xe) {
      const uint32_t k = queue_at(x - lead), lo = Sm.stage_first[k], stop = max(min(xe, lead + Sm.stage_first[k + 1]), x + 1), r = x - lead - lo;
      const int32_t A = (int32_t)Sm.K[k].A_rel;
      const unsigned long long magic = Sm.K[k].d_magic;
      uint32_t* P = T.P + Sm.win_off[k];
      auto window = [&](uint32_t at) {                   /* -1: deadline before A */
        const int32_t off = (int32_t)T.off[at];
        return off < A ? -1 : (int32_t)div_magic32((uint32_t)off - (uint32_t)A, magic);
      };
      const int32_t ahead = window(r ? x - 1 : x), last = window(stop - 1);
      if (last - ahead > kFewWindows) {                  /* windows begin here: their P, the requests before them */
        int32_t e = ahead;
        for (uint32_t y = x; y < stop; ++y)
          for (const int32_t b = window(y); e < b;) P[++e] = y - lead - lo;
      } else if (ahead < last) {
        const uint32_t d = (uint32_t)Sm.K[k].d;
        uint32_t X[kLocGroup];                           /* deadline - A, expired: 0 (window 0 begins at the first that is not) */
        uint32_t expired = 0;
        const uint4 u = *reinterpret_cast<const uint4*>(&T.off[x0]), v = *reinterpret_cast<const uint4*>(&T.off[x0 + 4]);
        const uint32_t off[kLocGroup] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < kLocGroup; ++i) {
          const bool in = x0 + i >= x && x0 + i < stop;
          const bool late = (int32_t)off[i] < A;
          X[i] = !in ? 0xffffffffu : late ? 0u : off[i] - (uint32_t)A;
          expired += in && late ? 1u : 0u;
        }
        for (int32_t e = ahead + 1; e <= last; ++e) {
          const uint32_t from = (uint32_t)e * d;         /* <= the last request's deadline - A */
          uint32_t below = 0;
#pragma unroll
          for (int i = 0; i < kLocGroup; ++i) below += X[i] < from ? 1u : 0u;
          P[e] = r + (e ? below : expired);
        }
      }
      x = stop;
    }
  }
  __syncthreads();
  /* E (Kp), u and every queue's kept count */
  for (uint32_t k = warp; k < S; k += kLocWarps) {
    uint32_t kept = 0;
    const uint32_t at = Sm.win_off[k], wins = Sm.win_cnt[k], cap = Sm.K[k].cap;
    if (wins) {
      const uint32_t P0 = T.P[at];
      int32_t e_carry = P0 > 0 ? -(int32_t)(P0 - 1) : kWinInf;       /* the requests with deadline < A: u = 0 */
      uint32_t k_carry = 0;
      for (uint32_t b0 = 0; b0 + 1 < wins; b0 += 32) {               /* windows b0.. */
        const uint32_t b = b0 + lane;
        int32_t val = kWinInf;
        uint32_t more = 0, u = 0;
        if (b + 1 < wins) {
          const uint32_t p = T.P[at + b], q = T.P[at + b + 1];
          u = win_u(b, cap);
          if (q > p) {
            val = (int32_t)u - (int32_t)(q - 1);
            const uint32_t top = u < q ? u : q;
            more = top > p ? top - p : 0;
          }
        }
        const uint32_t own_more = more;
        for (int o = 1; o < 32; o <<= 1) {
          if (RAW) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, more, o);
            if (lane >= (uint32_t)o) more += y;
          } else {
            const int32_t y = __shfl_up_sync(0xffffffffu, val, o);
            if (lane >= (uint32_t)o) val = min(val, y);
          }
        }
        /* of the windows before this lane's */
        int32_t before = __shfl_up_sync(0xffffffffu, val, 1);
        before = min(e_carry, lane ? before : kWinInf);
        if (b + 1 < wins) T.QU[at + b] = make_int2(RAW ? (int32_t)(k_carry + more - own_more) : min(before, 1) - 1, (int32_t)u);
        if (RAW) k_carry += __shfl_sync(0xffffffffu, more, 31);
        else e_carry = min(e_carry, __shfl_sync(0xffffffffu, val, 31));
      }
      const uint32_t n_q = T.P[at + wins - 1];
      kept = RAW ? k_carry : (uint32_t)((int32_t)n_q - 1 + min(e_carry, 1));
    }
    if (lane == 0) {
      Sm.stage_kept[k] = kept;
      if (a.out_seg_off) a.out_seg_off[(size_t)c * S + k] = first + Sm.stage_first[k];
    }
  }
  if (tid == 0 && c + 1 == a.n_ctx && a.out_seg_off) a.out_seg_off[(size_t)a.n_ctx * S] = a.n;
  __syncthreads();
  if (warp == 0) publish_kept(a, Sm, c, lane);
  __syncthreads();
  if (one_by_one)
    for (uint32_t p = tid; p < cnt; p += kLocThreads) {
      const uint32_t k = queue_at(p), r = p - Sm.stage_first[k], local = T.idx[lead + p];
      const PardSegConst& K = Sm.K[k];
      const int32_t off = (int32_t)T.off[lead + p], A = (int32_t)K.A_rel;
      uint32_t cpos = RAW ? r : 0u, ahead = 0, u = 0;    /* batch-slot position; kept requests ahead in the queue */
      if (off >= A) {
        const uint32_t at = Sm.win_off[k] + div_magic32((uint32_t)off - (uint32_t)A, K.d_magic);
        const int2 w = T.QU[at];
        u = (uint32_t)w.y;
        if (RAW) {
          const uint32_t top = r < u ? r : u, P = T.P[at];
          ahead = (uint32_t)w.x + (top > P ? top - P : 0);
        } else {
          cpos = ahead = min((uint32_t)((int32_t)r + w.x), u);
        }
      }
      const bool keep = cpos < u;
      const uint32_t round = K.cap_magic ? div_magic32(cpos, K.cap_magic) : cpos;
      if (keep) T.kept[Sm.kept_base[k] + ahead] = (uint16_t)local;
      const size_t at = (size_t)first + p;
      if (a.out_keep) a.out_keep[at] = keep ? 1 : 0;
      if (a.out_est) a.out_est[at] = K.A + (long long)((unsigned long long)round * (uint32_t)K.d);
      if (a.out_perm) a.out_perm[at] = first + local;
    }
  else
  for (uint32_t g = tid; g < groups; g += kLocThreads) {
    const uint32_t x0 = g * kLocGroup, xa = max(x0, lead), xe = min(x0 + kLocGroup, end);
    const size_t out = (size_t)(first - lead) + x0;
    const uint4 ix = *reinterpret_cast<const uint4*>(&T.idx[x0]);
    const uint32_t pair[4] = {ix.x, ix.y, ix.z, ix.w};
    uint32_t keepbits = 0, list = 0, k = 0, r_less = 0, rest = 0;  /* position in the queue less that in the group; the queue's end in the group */
    long long est[kLocGroup];
#pragma unroll
    for (int q = 0; q < kLocGroup; ++q) est[q] = 0;
    for (uint32_t i = xa - x0; i < xe - x0;) {           /* span after span of one queue and window: mostly one */
      if (i >= rest) {                                   /* a queue begins, or the group does */
        k = queue_at(x0 + i - lead);
        r_less = x0 - lead - Sm.stage_first[k];
        rest = min(lead + Sm.stage_first[k + 1], xe) - x0;
      }
      const PardSegConst& K = Sm.K[k];
      const uint32_t r = r_less + i, cap = K.cap;
      const int32_t off = (int32_t)T.off[x0 + i], first_off = (int32_t)K.A_rel;
      const int32_t b = off < first_off ? -1 : (int32_t)div_magic32((uint32_t)off - (uint32_t)first_off, K.d_magic);
      const uint32_t at = Sm.win_off[k] + (uint32_t)b;
      const uint32_t stop = max(min(T.P[at + 1] - r_less, rest), i + 1);
      int2 w = make_int2(0, 0);
      if (b >= 0) w = T.QU[at];
      uint32_t c0 = 0, left = 0, into = 0;               /* batch-slot position, kept ones of the span from here on, their place among the queue's */
      if (RAW) {
        c0 = r;
        if (b >= 0 && r < (uint32_t)w.y) {
          left = (uint32_t)w.y - r;
          into = (uint32_t)w.x + r - T.P[at];
        }
      } else if (b >= 0) {
        c0 = into = min((uint32_t)((int32_t)r + w.x), (uint32_t)w.y);
        left = (uint32_t)w.y - c0;
      }
      const long long A = K.A;
      const uint32_t d = (uint32_t)K.d;                  /* d fits 32 bits: it has a magic number */
      const unsigned long long magic = K.cap_magic;
      if (cap >= kLocGroup) {
        const uint32_t round = div_magic32(c0, magic), fresh = cap - (c0 - round * cap);     /* requests up to the next round */
        const uint32_t next = RAW || fresh <= left ? i + fresh : (uint32_t)kLocGroup;
        const long long e0 = A + (long long)((unsigned long long)round * d), e1 = e0 + d;
#pragma unroll
        for (int q = 0; q < kLocGroup; ++q) {            /* (what lies behind the span is made good by the next one) */
          if (q >= (int)i) est[q] = e0;
          if (q >= (int)next) est[q] = e1;
        }
      } else {                                           /* small rounds */
#pragma unroll
        for (int q = 0; q < kLocGroup; ++q)
          if (q >= (int)i) {
            const uint32_t c = RAW ? c0 + (q - i) : min(c0 + (q - i), c0 + left);
            est[q] = A + (long long)((unsigned long long)(cap > 1 ? div_magic32(c, magic) : c) * d);
          }
      }
      const uint32_t n_kept = min(stop - i, left);
      if (!keepbits) list = Sm.kept_base[k] + into;
      keepbits |= ((1u << n_kept) - 1) << i;
      i = stop;
    }
    /* the thread's survivors follow one another, across queues too */
#pragma unroll
    for (int q = 0; q < kLocGroup; ++q)
      if ((keepbits >> q) & 1u) T.kept[list++] = (uint16_t)((q & 1) ? pair[q / 2] >> 16 : pair[q / 2] & 0xffffu);
    if (xe - xa == kLocGroup) {
      if (a.out_keep) *reinterpret_cast<uint2*>(a.out_keep + out) = make_uint2(((keepbits & 15u) * 0x00204081u) & 0x01010101u, ((keepbits >> 4) * 0x00204081u) & 0x01010101u);
      if (a.out_est) {
        store4(a.out_est + out, est[0], est[1], est[2], est[3]);
        store4(a.out_est + out + 4, est[4], est[5], est[6], est[7]);
      }
      if (a.out_perm) {
        auto two = [&](uint32_t v) { return (first + (v & 0xffffu)) | (unsigned long long)(first + (v >> 16)) << 32; };
        store4(a.out_perm + out, two(pair[0]), two(pair[1]), two(pair[2]), two(pair[3]));
      }
    } else {
#pragma unroll
      for (int q = 0; q < kLocGroup; ++q)
        if (x0 + q >= xa && x0 + q < xe) {
          if (a.out_keep) a.out_keep[out + q] = (keepbits >> q) & 1u;
          if (a.out_est) a.out_est[out + q] = est[q];
          if (a.out_perm) a.out_perm[out + q] = first + ((q & 1) ? pair[q / 2] >> 16 : pair[q / 2] & 0xffffu);
        }
    }
  }
  if (!place_survivors(hdr, a, Sm, c)) return true;      /* (its barrier also completes the list) */
  if (a.out_kept_idx)
    for (uint32_t i = tid; i < Sm.kept; i += kLocThreads) a.out_kept_idx[Sm.base + i] = first + T.kept[i];
  return true;
}

/* 4. to 6. for every other ctx, from the sorted elements as they are. */
template <bool RAW>
__device__ __noinline__ void finish_ctx(PlanHeader* __restrict__ hdr, const LocalArgs& a, LocalSmem& Sm, const Format& f, uint32_t c,
                                        uint32_t first, uint32_t cnt, int items) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t S = (uint32_t)a.st.stage_stride, wfirst = warp * (32 * (uint32_t)items), kshift = f.ibits + f.dbits;
  const uint32_t n_good = Sm.stage_first[S];             /* requests that passed the checks; the others follow them */

  /* 4. window tables.  Their extents: a queue has windows up to its last element's. */
  if (warp == 0) {
    uint32_t run = 0;
    for (uint32_t k0 = 0; k0 < S; k0 += 32) {
      const uint32_t k = k0 + lane;
      uint32_t w = 0;
      if (k < S) {
        const uint32_t lo = Sm.stage_first[k], hi = Sm.stage_first[k + 1];
        const PardSegConst& K = Sm.K[k];
        if (a.out_seg_off) a.out_seg_off[(size_t)c * S + k] = first + lo;
        Sm.stage_kept[k] = 0;
        Sm.hb_kept[k] = hi - lo;
        if (hi > lo && (K.narrow & kSegNoStage)) set_status(hdr, PARD_EDATA);   /* requests queued at a stage the pipeline lacks */
        if (hi > lo && !(K.narrow & (kSegNoStage | kSegHighFirst))) {
          const long long X = slack_of((Sm.keys[hi - 1] >> f.ibits) & f.dmask, K);
          const unsigned long long nb = X < 0 ? 0ull : (unsigned long long)X / (unsigned long long)K.d + 1;
          if (nb >= kTabEntries) Sm.use_scan = 1;
          else w = (uint32_t)nb + 1;
        }
      }
      uint32_t x = w;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x += y;
      }
      if (k < S) { Sm.win_off[k] = run + x - w; Sm.win_cnt[k] = w; }
      run += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0 && (run > kTabEntries || a.force_scan)) Sm.use_scan = 1;
    if (c + 1 == a.n_ctx && lane == 0 && a.out_seg_off) a.out_seg_off[(size_t)a.n_ctx * S] = a.n;
  }
  __syncthreads();
  /* a queue served high budget first keeps a prefix: its length is the first position r with r >= u_r */
  if (a.st.d_priority) {
#pragma unroll 1
    for (int i = 0; i < items; ++i) {
      const uint32_t pos = wfirst + i * 32 + lane;
      if (pos >= n_good) break;
      const Elem x = decode(Sm.keys[pos], pos, Sm, f);
      const PardSegConst& K = Sm.K[x.stage];
      if ((K.narrow & (kSegHighFirst | kSegNoStage)) == kSegHighFirst && x.r >= threshold_u(x.X, K)) atomicMin(&Sm.hb_kept[x.stage], x.r);
    }
    __syncthreads();
  }
  const bool tables = !Sm.use_scan;
  if (tables) {
#pragma unroll 1
    for (int i = 0; i < items; ++i) {
      const uint32_t pos = wfirst + i * 32 + lane;
      const bool in = pos < n_good;
      Elem x = {};
      uint32_t b = kNoWindow;
      bool has = false;
      if (in) {
        x = decode(Sm.keys[pos], pos, Sm, f);
        has = Sm.win_cnt[x.stage] != 0;
        if (has) b = window_of(x.X, Sm.K[x.stage]);
      }
      if (in) Sm.tab.win[pos] = (uint16_t)b;
      uint32_t pb = __shfl_up_sync(0xffffffffu, b, 1);   /* the neighbour's window, when it is of the same queue */
      if (lane == 0 && in && has && x.r > 0) pb = window_of(decode(Sm.keys[pos - 1], pos - 1, Sm, f).X, Sm.K[x.stage]);
      if (has) {
        const uint32_t off = Sm.win_off[x.stage];
        const uint32_t from = x.r == 0 || pb == kNoWindow ? 0u : pb + 1;
        if (b != kNoWindow)
          for (uint32_t e = from; e <= b; ++e) Sm.tab.P[off + e] = x.r;
        if (pos + 1 == Sm.stage_first[x.stage + 1]) Sm.tab.P[off + Sm.win_cnt[x.stage] - 1] = x.r + 1;
      }
    }
    __syncthreads();
    for (uint32_t k = warp; k < S; k += kLocWarps) {
      uint32_t kept = 0;
      if (Sm.win_cnt[k]) kept = table_prefix<RAW>(Sm.tab, Sm.win_off[k], Sm.win_cnt[k], Sm.K[k].cap, lane);
      else if ((Sm.K[k].narrow & (kSegHighFirst | kSegNoStage)) == kSegHighFirst) kept = Sm.hb_kept[k];
      if (lane == 0) Sm.stage_kept[k] = kept;
    }
    __syncthreads();
  }

  if (tables) {
    if (warp == 0) publish_kept(a, Sm, c, lane);
    if (!place_survivors(hdr, a, Sm, c)) return;
    const uint32_t base = Sm.base;
    /* 6. every request on its own */
#pragma unroll 2
    for (int i = 0; i < items; ++i) {
      const uint32_t pos = wfirst + i * 32 + lane;
      if (pos >= cnt) break;
      const unsigned long long e = Sm.keys[pos];
      const uint32_t idx = (uint32_t)e & f.imask;
      uint32_t keep = 0;
      long long est = 0;
      if (pos < n_good) {
        const uint32_t stage = (uint32_t)(e >> kshift), r = pos - Sm.stage_first[stage];
        const PardSegConst& K = Sm.K[stage];
        uint32_t cpos = RAW ? r : 0u, ahead = 0, u = 0;  /* batch-slot position; kept requests ahead in the queue */
        const uint32_t b = Sm.tab.win[pos];
        if (b != kNoWindow) {
          const uint32_t at = Sm.win_off[stage] + b, P = Sm.tab.P[at];
          u = win_u(b, K.cap);
          if (RAW) {
            const uint32_t top = r < u ? r : u;
            ahead = Sm.tab.Kp[at] + (top > P ? top - P : 0);
          } else {
            int32_t m = Sm.tab.E[at];                    /* min over t < r of (u_t - t); values above 1 cannot lower the position */
            if (r > P) m = min(m, (int32_t)u - (int32_t)(r - 1));
            cpos = ahead = r == 0 ? 0u : r - 1 + (uint32_t)min(m, 1);
          }
        } else if ((K.narrow & (kSegHighFirst | kSegNoStage)) == kSegHighFirst) {
          u = threshold_u(slack_of((e >> f.ibits) & f.dmask, K), K);
          ahead = min(r, Sm.hb_kept[stage]);
          cpos = RAW ? r : ahead;
        }
        keep = cpos < u ? 1u : 0u;
        const uint32_t round = K.cap_magic ? div_magic32(cpos, K.cap_magic) : cpos;
        est = K.A + (long long)((unsigned long long)round * (unsigned long long)K.d);
        if (keep && a.out_kept_idx) a.out_kept_idx[base + Sm.kept_base[stage] + ahead] = idx;
      }
      const uint32_t g = first + pos;
      if (a.out_keep) a.out_keep[g] = (uint8_t)keep;
      if (a.out_est) a.out_est[g] = est;
      if (a.out_perm) a.out_perm[g] = idx;
    }
    return;
  }

  /* Too many windows: the segmented scan over the elements, first what every warp's add up to, then
   * positions and decisions; the survivors' list is packed afterwards. */
  SegVal run = seg_identity<RAW>();
  for (int pass = 0; pass < 2; ++pass) {
    SegVal carry = seg_identity<RAW>();
    if (pass == 1)
      for (uint32_t w = 0; w < warp; ++w) {
        SegVal t; t.m = Sm.wm[w]; t.head = Sm.wh[w];
        carry = seg_combine<RAW>(carry, t);
      }
#pragma unroll 1
    for (int i = 0; i < items; ++i) {
      const uint32_t pos = wfirst + i * 32 + lane;
      const bool in = pos < n_good;
      Elem x = {};
      SegVal v = seg_identity<RAW>();
      uint32_t u = 0;
      if (in) {
        x = decode(Sm.keys[pos], pos, Sm, f);
        const PardSegConst& K = Sm.K[x.stage];
        u = (K.narrow & kSegNoStage) ? 0u : threshold_u(x.X, K);
        v.head = x.r == 0 ? 1u : 0u;
        v.m = RAW ? (x.r < u ? 1 : 0) : (int32_t)u - (int32_t)x.r;
      }
      const SegVal inc = warp_scan<RAW>(v, lane);
      SegVal exc, all;
      exc.m = __shfl_up_sync(0xffffffffu, inc.m, 1);
      exc.head = __shfl_up_sync(0xffffffffu, inc.head, 1);
      if (lane == 0) exc = seg_identity<RAW>();
      all.m = __shfl_sync(0xffffffffu, inc.m, 31);
      all.head = __shfl_sync(0xffffffffu, inc.head, 31);
      if (pass == 0) { run = seg_combine<RAW>(run, all); continue; }
      const SegVal pre = seg_combine<RAW>(carry, exc);   /* over the earlier requests of the same queue */
      carry = seg_combine<RAW>(carry, all);
      if (pos >= cnt) continue;
      uint32_t keep = 0;
      long long est = 0;
      if (in) {
        const PardSegConst& K = Sm.K[x.stage];
        uint32_t cpos, ahead;
        if (RAW) {
          cpos = x.r;
          ahead = x.r == 0 ? 0u : (uint32_t)pre.m;
        } else {
          const long long cc = (long long)x.r - 1 + pre.m;
          cpos = x.r == 0 ? 0u : (cc < (long long)x.r ? (uint32_t)cc : x.r);
          if (K.narrow & kSegHighFirst) cpos = min(x.r, Sm.hb_kept[x.stage]);
          ahead = cpos;
        }
        const uint32_t round = K.cap_magic ? div_magic32(cpos, K.cap_magic) : cpos;
        est = K.A + (long long)((unsigned long long)round * (unsigned long long)K.d);
        keep = cpos < u ? 1u : 0u;
        if (keep && a.kept_tmp) a.kept_tmp[first + Sm.stage_first[x.stage] + ahead] = x.idx;
        if (pos + 1 == Sm.stage_first[x.stage + 1]) Sm.stage_kept[x.stage] = ahead + keep;     /* the queue's last request */
      }
      const uint32_t g = first + pos;
      if (a.out_keep) a.out_keep[g] = (uint8_t)keep;
      if (a.out_est) a.out_est[g] = est;
      if (a.out_perm) a.out_perm[g] = (uint32_t)Sm.keys[pos] & f.imask;
    }
    if (pass == 0) {
      if (lane == 0) { Sm.wm[warp] = run.m; Sm.wh[warp] = run.head; }
      __syncthreads();
    }
  }
  __threadfence_block();
  __syncthreads();
  if (warp == 0) publish_kept(a, Sm, c, lane);
  if (!place_survivors(hdr, a, Sm, c)) return;
  if (a.out_kept_idx && a.kept_tmp)
    for (uint32_t k = 0; k < S; ++k) {
      const uint32_t nk = Sm.stage_kept[k], from = first + Sm.stage_first[k], to = Sm.base + Sm.kept_base[k];
      for (uint32_t i = tid; i < nk; i += kLocThreads) a.out_kept_idx[to + i] = a.kept_tmp[from + i];
    }
}

template <bool RAW, bool SINGLE>
__device__ __forceinline__ void plan_ctx(PlanHeader* __restrict__ hdr, const LocalArgs& a, LocalSmem& Sm) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t S = (uint32_t)a.st.stage_stride;
  /* SINGLE: the call's one ctx; the last warps work out its constants, a chain of dependent loads, while the others read
   * the requests (3,001 requests of three stages 36.0 -> 33.5 us a call, 8,000 50.5 -> 47.5). */
  constexpr uint32_t kReaders = SINGLE ? kLocWarps - 4 : kLocWarps;
  if (SINGLE) {                                          /* the only kernel of the call: the header starts here */
    if (tid < sizeof(PlanHeader) / 4) reinterpret_cast<uint32_t*>(hdr)[tid] = 0;
    if (tid == 0) { Sm.ctx = 0; Sm.first = 0; Sm.cnt = a.n; }
  } else if (tid == 0) {
    /* The promised grouping is broken: found by k_ctx_prep, or (`unsorted`) by a block of this kernel, so
     * that one thread has to look for the whole block.  (It takes its ticket meanwhile; that nobody will
     * plan that ctx then does not matter, the waits behind it end with `aborted`.) */
    const uint32_t broken = ld_relaxed(&hdr->unsorted) | ld_relaxed(&hdr->ctx_too_big), t = atomicAdd(&hdr->ticket[0], 1u);
    Sm.ctx = kNoCtx;
    if (broken) {
      if (blockIdx.x == 0) { set_status(hdr, PARD_EDATA); hdr->aborted = 1; }
    } else {
      Sm.ctx = t;
      Sm.first = a.ctx_start[t];
      Sm.cnt = a.ctx_start[t + 1] - Sm.first;
      /* As many requests behind this ctx on their way into L2 for the block that takes the next one: 4,096 x 8,192
       * requests 391 -> 361 us (two contexts on 362, eight 398; by each thread's own prefetches 470 -> 506). */
      l2_ahead(reinterpret_cast<const unsigned long long*>(a.req), 2ull * Sm.first, 2ull * Sm.cnt, 2 * Sm.cnt, 2ull * a.n);
    }
  }
  if (tid == 0) { Sm.flags = a.st.d_priority ? 4u : 0u; Sm.use_scan = 0; Sm.abort = 0; }
  __syncthreads();
  if (Sm.ctx == kNoCtx) return;
  const uint32_t c = Sm.ctx, first = Sm.first, cnt = Sm.cnt;
  /* every warp owns `items` rounds of 32 consecutive requests: as few as the ctx needs */
  const int items = (int)((cnt + kLocThreads - 1) / kLocThreads);
  const uint32_t wfirst = warp * (32 * (uint32_t)items);

  /* 1. the ctx's requests: deadline range, input checks, order.  As long as a warp finds its requests
   * in order (and the deadlines share their high word: no 71-minute boundary inside the ctx) it only
   * looks at low words, and leaves them and the stages in shared memory. */
  Ordered& O = *reinterpret_cast<Ordered*>(Sm.keys);
  const bool few = S <= 16 && !a.st.d_priority;          /* (queues served high budget first want descending deadlines) */
  unsigned long long lmin = ~0ull, lmax = 0;
  uint32_t seen = few ? 0u : 4u;                         /* 1: a request of another ctx, 2: out of range, 4: not in order */
  const uint32_t ritems = SINGLE ? (cnt + 32 * kReaders - 1) / (32 * kReaders) : (uint32_t)items, rfirst = warp * 32 * ritems;   /* rounds per warp in this step */
  if (rfirst < cnt && warp < kReaders) {
    const uint4* req = a.req + first;
    const uint4 p = __ldg(&req[rfirst > 0 ? rfirst - 1 : 0]);
    const uint32_t wend = min(cnt, rfirst + 32 * ritems);
    const uint32_t high = p.y, x_first = __ldg(&req[rfirst]).x, x_last = __ldg(&req[wend - 1]).x;
    uint32_t last = p.x;                                 /* low words of the row before this one, first the request before the warp's */
    constexpr int kUn = 4;                               /* requests in flight per thread */
    bool ordered = few;                                  /* (uniform) */
#pragma unroll 1
    for (uint32_t p0 = rfirst + lane; p0 - lane < wend; p0 += 32 * kUn) {
      uint4 r[kUn];
      const bool full = p0 - lane + 32 * kUn <= wend;    /* uniform */
      if (full) {
#pragma unroll
        for (int u = 0; u < kUn; ++u) r[u] = __ldg(&req[p0 + u * 32]);
      } else {
#pragma unroll
        for (int u = 0; u < kUn; ++u) {
          r[u] = make_uint4(0xffffffffu, high, c, 0u);   /* behind every request */
          if (p0 + u * 32 < wend) r[u] = __ldg(&req[p0 + u * 32]);
        }
      }
      if (ordered) {
        uint32_t other = 0, top = 0;
        bool back = false;
        const uint32_t behind = __shfl_sync(0xffffffffu, last, 31);
#pragma unroll
        for (int u = 0; u < kUn; ++u) {
          const uint32_t px = __shfl_sync(0xffffffffu, lane == 31 ? last : r[u].x, (lane - 1) & 31);
          last = r[u].x;
          back |= r[u].x < px;
          other |= (r[u].z ^ c) | (r[u].y ^ high);
          top = max(top, r[u].w & 0xffffu);
          if (full || p0 + u * 32 < wend) {
            O.D[p0 + u * 32] = r[u].x;
            O.code[p0 + u * 32] = (uint8_t)(4 * (r[u].w & 15u));
          }
        }
        if (__all_sync(0xffffffffu, !back && other == 0 && top < S && high < (uint32_t)(PARD_TIME_LIMIT_US >> 32))) continue;
        ordered = false;
        if (p0 - lane > rfirst) {                        /* the rows so far were in order */
          lmin = ((unsigned long long)high << 32) | x_first;
          lmax = ((unsigned long long)high << 32) | behind;
        }
      }
#pragma unroll
      for (int u = 0; u < kUn; ++u) {
        const unsigned long long D = ((unsigned long long)r[u].y << 32) | r[u].x;
        if (p0 + u * 32 < wend) {
          if (r[u].z == c && (r[u].w & 0xffffu) < S && D < (unsigned long long)PARD_TIME_LIMIT_US) {
            lmin = D < lmin ? D : lmin;
            lmax = D > lmax ? D : lmax;
          } else {
            seen |= r[u].z != c ? 3u : 2u;
          }
        }
      }
    }
    if (ordered) {                                       /* the warp's range is that of its first and its last request */
      lmin = ((unsigned long long)high << 32) | x_first;
      lmax = ((unsigned long long)high << 32) | x_last;
    } else {
      seen |= 4u;
    }
  }
  if (SINGLE && warp >= kReaders) {
    __shared__ CtxScratch s_scratch;
    if (ctx_constants<true, 1>(a.pipes, a.n_pipelines, a.st, c, 0, 0, Sm.K, s_scratch, nullptr, 32 * kReaders)) set_status(hdr, PARD_EDATA);
  }
  lmin = warp_min(lmin);
  lmax = ~warp_min(~lmax);
  seen = __reduce_or_sync(0xffffffffu, seen);
  if (lane == 0) {
    Sm.red_min[warp] = lmin;
    Sm.red_max[warp] = lmax;
    if (seen) atomicOr(&Sm.flags, seen);
  }
  __syncthreads();
  const uint32_t flags = Sm.flags;
  if (flags & 1u) {                                      /* not grouped by ctx after all (or, with one ctx, a request of another) */
    if (tid == 0) { hdr->unsorted = 1; set_status(hdr, PARD_EDATA); hdr->aborted = 1; }
    return;
  }
  const unsigned long long dmin = warp_min(Sm.red_min[lane % kLocWarps]), dmax = ~warp_min(~Sm.red_max[lane % kLocWarps]);
  const bool flagged = flags & 2u;
  const unsigned long long span = dmin <= dmax ? dmax - dmin : 0ull;
  const bool in_order = cnt > 0 && !(flags & 6u) && (span >> 31) == 0;
  Format f;
  f.ibits = a.ibits;
  f.dbits = span ? 64u - (uint32_t)__clzll((long long)span) : 0u;
  f.imask = (1u << a.ibits) - 1;
  f.dmask = f.dbits >= 64 ? ~0ull : ((1ull << f.dbits) - 1);
  /* stage field of the elements: requests that failed the checks carry the value S there, so
   * that they sort behind the ctx's queues; they are reported, never decided */
  const uint32_t sb = 32u - __clz(flagged ? S : S - 1);  /* bit width of the largest value; __clz(0) = 32 */
  if (flagged && tid == 0) set_status(hdr, PARD_EDATA);

  /* 2. constants of the ctx's queues: worked out beside the first step when the call is this one block; else taken
   * from the table filled for all queues at once (a chain of dependent loads that every block
   * would otherwise wait for); completed with what hangs on the ctx's deadline range */
  for (uint32_t k = tid; k < S; k += kLocThreads) {
    PardSegConst K = SINGLE ? Sm.K[k] : a.ktab[(size_t)c * S + k];
    K.A_rel = (K.narrow & kSegHighFirst) ? (int64_t)dmax - K.A : booked_within(K.A - (int64_t)dmin, span);
    Sm.K[k] = K;
  }

  /* 3. elements, sorted */
  const uint32_t lead = first % kLocGroup;
  if (in_order) {
    const bool small = cnt <= 4 * kLocThreads;
    const uint2 ranks = small ? (S <= 8 ? order_few<1, 4>(Sm, O, cnt, S) : order_few<2, 4>(Sm, O, cnt, S))
                              : (S <= 8 ? order_few<1, 16>(Sm, O, cnt, S) : order_few<2, 16>(Sm, O, cnt, S));
    if (split_fits(a, Sm, span)) {
      if (small) place_few<4>(O, cnt, ranks, lead, (uint32_t)dmin);
      else place_few<16>(O, cnt, ranks, lead, (uint32_t)dmin);
      __syncthreads();
      if (finish_split<RAW>(hdr, a, Sm, c, first, cnt)) return;
    }
  }
  if (sb + f.dbits + f.ibits > 64) {         /* the element does not fit 64 bits */
    if (tid == 0) { hdr->wide = 1; set_status(hdr, PARD_ERANGE); hdr->aborted = 1; }
    return;
  }
  {
    unsigned long long key[kLocItems];
#pragma unroll
    for (int i = 0; i < kLocItems; ++i) {
      if (i >= items) break;
      const uint32_t pos = wfirst + i * 32 + lane;
      key[i] = ~0ull;                                    /* padding sorts last */
      if (pos < cnt) {
        const uint4 r = __ldg(&a.req[first + pos]);
        const unsigned long long D = ((unsigned long long)r.y << 32) | r.x;
        const uint32_t stage = r.w & 0xffffu, j = first + pos;
        if (stage < S && D < (unsigned long long)PARD_TIME_LIMIT_US) {
          const bool high_first = a.st.d_priority && a.st.d_priority[(size_t)c * S + stage] != 0;
          key[i] = ((((unsigned long long)stage << f.dbits) | ((high_first ? dmax - D : D - dmin) & f.dmask)) << f.ibits) | j;
        } else {
          key[i] = (((unsigned long long)S << f.dbits) << f.ibits) | j;
        }
      }
    }
    __syncthreads();                                     /* the room of the counters has been in use */
    for (uint32_t i = tid; i < 2 * kLocWarps * kBins; i += kLocThreads) (&Sm.slot[0][0])[i] = 0;
    __syncthreads();
    const uint32_t skip = (flags & 4u) ? 0u : f.dbits, passes = (f.dbits - skip + sb + 7) / 8;
    for (uint32_t p = 0; p < passes; ++p) pass_byte(key, f.ibits + skip + 8 * p, items, Sm, tid, p + 1 < passes);
    if (passes == 0) {
#pragma unroll
      for (int i = 0; i < kLocItems; ++i)
        if (i < items) Sm.keys[wfirst + i * 32 + lane] = key[i];
      __syncthreads();
    }
  }

  /* queue boundaries: where the stage changes between neighbours */
  const uint32_t kshift = f.ibits + f.dbits;
#pragma unroll 1
  for (int i = 0; i < items; ++i) {
    const uint32_t pos = wfirst + i * 32 + lane;
    if (pos >= cnt) break;
    const uint32_t k1 = (uint32_t)(Sm.keys[pos] >> kshift);
    const uint32_t k0 = pos ? (uint32_t)(Sm.keys[pos - 1] >> kshift) + 1 : 0u;
    for (uint32_t k = k0; k <= k1; ++k) Sm.stage_first[k] = pos;
    if (pos + 1 == cnt)
      for (uint32_t k = k1 + 1; k <= S; ++k) Sm.stage_first[k] = cnt;
  }
  if (cnt == 0)
    for (uint32_t k = tid; k <= S; k += kLocThreads) Sm.stage_first[k] = 0;
  __syncthreads();
  if (Sm.stage_first[S] == cnt && split_fits(a, Sm, span)) {
    /* the elements apart, in place */
    Split& T = *reinterpret_cast<Split*>(Sm.keys);
    unsigned long long e[kLocItems];
#pragma unroll
    for (int i = 0; i < kLocItems; ++i)
      if (i < items) e[i] = Sm.keys[wfirst + i * 32 + lane];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kLocItems; ++i) {
      if (i >= items) break;
      const uint32_t pos = wfirst + i * 32 + lane;
      if (pos < cnt) {
        T.off[lead + pos] = (uint32_t)((e[i] >> f.ibits) & f.dmask);
        T.idx[lead + pos] = (uint16_t)(((uint32_t)e[i] & f.imask) - first);
      }
    }
    __syncthreads();
    if (finish_split<RAW>(hdr, a, Sm, c, first, cnt)) return;
#pragma unroll
    for (int i = 0; i < kLocItems; ++i)                  /* too many windows: as they were */
      if (i < items) Sm.keys[wfirst + i * 32 + lane] = e[i];
    __syncthreads();
  }
  finish_ctx<RAW>(hdr, a, Sm, f, c, first, cnt, items);
}

template <bool RAW, bool SINGLE>
__global__ void __launch_bounds__(kLocThreads, SINGLE ? 1 : 2)
k_plan_local(PlanHeader* __restrict__ hdr, const __grid_constant__ LocalArgs a) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  plan_ctx<RAW, SINGLE>(hdr, a, *reinterpret_cast<LocalSmem*>(smem_raw));
  if (a.answer.word) {
    __syncthreads();
    if (threadIdx.x == 0) pard_report(&hdr->status, a.answer.word, a.answer.ticket);
  }
}

/* What the blocks of a grouped call need beforehand: the constants of all queues (a block per ctx)
 * and where every ctx begins (a warp per ctx, in further blocks of the same launch): the first request
 * whose ctx is >= c, by a 32-ary search.  Whether the requests do come in ctx order is settled by
 * k_plan_local, where every block checks that its range holds requests of its ctx only; that test is
 * complete as long as the boundaries never step back and the ranges cover all requests, which is
 * checked here. */
__global__ void __launch_bounds__(kConstThreads)
k_ctx_prep(const __grid_constant__ LocalArgs a, PardSegConst* __restrict__ ktab, uint32_t* __restrict__ ctx_start, PlanHeader* hdr) {
  pdl_wait();
  __shared__ CtxScratch scratch;
  if (blockIdx.x < a.n_ctx) {
    if (ctx_constants<true>(a.pipes, a.n_pipelines, a.st, blockIdx.x, 0, 0, ktab + (size_t)blockIdx.x * a.st.stage_stride, scratch))
      set_status(hdr, PARD_EDATA);
    return;
  }
  const uint32_t c = (blockIdx.x - a.n_ctx) * (kConstThreads / 32) + (threadIdx.x >> 5);
  if (c <= a.n_ctx) ctx_range_search(a.req, a.n, a.n_ctx, c, ctx_start, hdr, kLocalTile);
}

}  // namespace

namespace pard_plan_detail {

int allow_local_smem() {
  PARD_CUDA_OK(cudaFuncSetAttribute(k_plan_local<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LocalSmem)));
  PARD_CUDA_OK(cudaFuncSetAttribute(k_plan_local<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LocalSmem)));
  PARD_CUDA_OK(cudaFuncSetAttribute(k_plan_local<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LocalSmem)));
  PARD_CUDA_OK(cudaFuncSetAttribute(k_plan_local<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LocalSmem)));
  return PARD_OK;
}

int launch_ctx_prep(const LocalArgs& a, PardSegConst* ktab, uint32_t* ctx_start, PlanHeader* hdr, cudaStream_t stream) {
  const uint32_t per = kConstThreads / 32;
  PARD_CUDA_OK(launch_pdl(k_ctx_prep, a.n_ctx + (a.n_ctx + 1 + per - 1) / per, kConstThreads, 0, stream, a, ktab, ctx_start, hdr));
  return PARD_OK;
}

int launch_plan_local(const LocalArgs& a, PlanHeader* hdr, bool raw, cudaStream_t stream) {
  auto kernel = a.ctx_start ? (raw ? k_plan_local<true, false> : k_plan_local<false, false>)
                            : (raw ? k_plan_local<true, true> : k_plan_local<false, true>);
  PARD_CUDA_OK(launch_pdl(kernel, a.ctx_start ? a.n_ctx : 1u, kLocThreads, sizeof(LocalSmem), stream, hdr, a));
  return PARD_OK;
}

}  // namespace pard_plan_detail
