/* Requests grouped by ctx that come in order: no sort.  Part of pard_plan.cu (included there).
 *
 * Queues filled in arrival order with one objective per ctx hold their requests in budget order already:
 * grouped by ctx, deadlines never stepping back along a ctx.  Then a request's place in its queue is the
 * number of earlier requests of its stage, and since the thresholds u only rise along a queue the admitted
 * count at any point follows from two figures of what lies before it: how many requests, and the minimum of
 * u_t - t over them.  Both combine over consecutive spans, so the plan takes two reads of the requests and
 * nothing else:
 *   k_dir_begin   the queues' constants; the pieces, runs of tiles of one ctx; the scratch cleared
 *   k_dir_count   (count, minimum) of every queue, per piece; checks the order; also finds what k_prepass would, so
 *                 that nothing is read twice when the order is not there
 *   k_dir_scan    their running values over the pieces of every ctx, queue boundaries, kept counts, offsets
 *   k_dir_emit    every tile's requests ordered by stage in shared memory, decided, written to their place
 * What the path does not take -- deadlines that step back, requests not grouped, input errors, constants
 * beyond 32 bits -- is found out by k_dir_count (direct_off); the kernels of the general path, launched behind
 * these in any case, then do the work, and return at once otherwise.  Whether a deadline stepped back goes to
 * them too (pair_steps_back): without one their passes take the stage bits alone. */

constexpr int kDirThreads = 256;
constexpr int kDirWarps = kDirThreads / 32;
constexpr int kDirRows = 7;                       /* rows of 32 requests per warp and tile */
constexpr uint32_t kDirTile = kDirThreads * kDirRows;   /* requests a block of k_dir_emit orders at a time (a multiple of 128) */
constexpr int kDirStages = 16;                    /* most stages: lane j of a warp keeps the figures of stage j */
constexpr uint32_t kDirMaxTiles = 4;              /* tiles per piece, at most (places in a piece take 16 bits) */
constexpr int32_t kDirInf = 0x7fffffff;           /* no request: positions below 2^30 taken off it leave more than 1 */

struct DirectArgs {
  const uint4* req;
  uint32_t n, n_ctx, S, sbits, ibits;
  const PardSegConst* ktab;
  uint32_t* ctx_start;                            /* [n_ctx + 1] */
  uint32_t* const_bad;                            /* [n_ctx] 1: an input of the constants out of range */
  uint32_t piece, n_pieces;                       /* requests per piece, a multiple of the tile; pieces (some may be empty) */
  uint32_t stall;                                 /* testing aid: k_dir_emit's first block never asks for its first tile */
  uint4* piece_info;                              /* [n_pieces] ctx, first request, end, 0 */
  uint2* piece_rows;                              /* [n_pieces][kDirStages] count, minimum; from k_dir_scan on: of all earlier pieces of the ctx */
};

constexpr uint32_t kDirOff = 1u, kDirSteps = 2u;  /* bits of PlanHeader::direct_off; the second: a step back has been seen, nobody needs to look for more */

/* {count, minimum} of a span followed by another */
__device__ __forceinline__ uint2 dir_then(uint2 a, uint2 b) { return make_uint2(a.x + b.x, (uint32_t)min((int32_t)a.y, (int32_t)b.y - (int32_t)a.x)); }

/* The pieces of ctx c, requests [first, end), by one warp.  A ctx has as many numbers as it may need pieces,
 * ceil(len / piece) <= end / piece - first / piece + 1, from first / piece + c on. */
__device__ __forceinline__ void dir_pieces(const DirectArgs& a, uint32_t c, uint32_t first, uint32_t end, uint32_t lane) {
  const uint32_t p0 = first / a.piece + c, p1 = min(end / a.piece + c + 1, a.n_pieces);
  for (uint32_t p = p0 + lane; p < p1; p += 32) {
    const unsigned long long b = first + (unsigned long long)(p - p0) * a.piece;
    a.piece_info[p] = b < end ? make_uint4(c, (uint32_t)b, (uint32_t)min((unsigned long long)end, b + a.piece), 0u) : make_uint4(c, 0u, 0u, 0u);
  }
}

/* blocks [0, n_ctx): constants; the next ones: where every ctx begins and ends, and its pieces; the rest clear the scratch.
 * (The constants are a chain of dependent loads: in the first blocks of k_dir_count, under its traffic, they come
 * 10 us later.) */
__global__ void __launch_bounds__(kDirThreads)
k_dir_begin(const __grid_constant__ DirectArgs a, const __grid_constant__ ConstArgs ca, uint4* __restrict__ zero, unsigned long long n16,
            uint32_t range_blocks) {
  pdl_wait();
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  if (blockIdx.x < a.n_ctx) {
    __shared__ CtxScratch scratch;
    const uint32_t c = blockIdx.x;
    const bool bad = __syncthreads_or(ctx_constants<true>(ca.pipes, ca.n_pipelines, ca.st, c, 0, 0, ca.ktab + (size_t)c * a.S, scratch, sums_of(ca, c)));
    if (tid == 0) a.const_bad[c] = bad ? 1u : 0u;
    return;
  }
  const uint32_t block = blockIdx.x - a.n_ctx;
  if (block < range_blocks) {
    const uint32_t c = block * kDirWarps + (tid >> 5);
    if (c >= a.n_ctx) return;
    uint32_t lo[2] = {0, 0}, hi[2] = {a.n, a.n};   /* first request whose ctx is >= c, >= c + 1 */
    while (lo[0] < hi[0] || lo[1] < hi[1]) {
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (lo[q] < hi[q]) {                      /* uniform across the warp */
          const uint32_t p = lo[q] + (uint32_t)(((unsigned long long)(lane + 1) * (hi[q] - lo[q])) / 33u);   /* lo <= p < hi */
          const uint32_t k = __popc(__ballot_sync(0xffffffffu, __ldg(&a.req[p]).z < c + q));
          const uint32_t below = __shfl_sync(0xffffffffu, p, k ? k - 1 : 0), at = __shfl_sync(0xffffffffu, p, k < 32 ? k : 31);
          if (k) lo[q] = below + 1;
          if (k < 32) hi[q] = at;
        }
    }
    if (lane == 0) {
      a.ctx_start[c] = lo[0];
      if (c + 1 == a.n_ctx) a.ctx_start[c + 1] = lo[1];
    }
    dir_pieces(a, c, lo[0], lo[1], lane);
    return;
  }
  const unsigned long long step = (unsigned long long)(gridDim.x - a.n_ctx - range_blocks) * kDirThreads;
  for (unsigned long long i = (unsigned long long)(block - range_blocks) * kDirThreads + tid; i < n16; i += step) zero[i] = make_uint4(0u, 0u, 0u, 0u);
}

/* A queue's constants against the piece's first deadline: A in 32 bits, d, its reciprocal, cap. */
struct DirConst {
  int32_t A;
  uint32_t d, cap;
  unsigned long long magic;
};
/* False: the queue's constants do not allow it.  Offsets stay below 2^31 - 1, so that an A later than all of
 * them can be cut off there. */
__device__ __forceinline__ bool dir_const(const PardSegConst& K, unsigned long long D0, DirConst& out) {
  const long long A = K.A - (long long)D0;
  out.A = A > 0x7fffffffll ? 0x7fffffff : (int32_t)A;
  out.d = (uint32_t)K.d;
  out.cap = K.cap;
  out.magic = K.d_magic;
  return K.d_magic != 0 && A >= -0x80000000ll;
}
/* u of a request, and the first offset from which it is larger */
__device__ __forceinline__ uint32_t dir_u(uint32_t off, const DirConst& K, int32_t* next) {
  if ((int32_t)off < K.A) {
    *next = K.A;
    return 0;
  }
  const uint32_t b = div_magic32(off - (uint32_t)K.A, K.magic);
  const long long at = K.A + (long long)(((unsigned long long)b + 1) * K.d);
  *next = at > 0x7fffffffll ? 0x7fffffff : (int32_t)at;
  const unsigned long long u = ((unsigned long long)b + 1) * K.cap;
  return u > kUClamp ? kUClamp : (uint32_t)u;
}
__device__ __noinline__ uint32_t dir_u_far(uint32_t off, const DirConst& K, int32_t* next) { return dir_u(off, K, next); }
/* the lanes of a row whose stage is this lane's number: from the ballots of the stages' bits */
template <int BITS>
__device__ __forceinline__ uint32_t dir_mine(uint32_t st, uint32_t valid, uint32_t lane) {
  uint32_t m = valid;
#pragma unroll
  for (int b = 0; b < BITS; ++b) m &= __ballot_sync(0xffffffffu, (st >> b) & 1u) ^ (((lane >> b) & 1u) - 1u);
  return (lane & (kDirStages - 1)) >> BITS ? 0u : m;
}

struct DirScanOut {
  uint32_t *seg_off, *out_seg_off, *seg_kept, *kept_base, *chunk_base, *out_seg_kept;
  unsigned long long* out_n_kept;
};
/* Running values over the pieces of a ctx, a block per ctx and a warp per stage; the queues' boundaries and kept
 * counts; in the last block the output offsets of all queues' survivors. */
constexpr int kDirScanThreads = 32 * kDirStages;
__global__ void __launch_bounds__(kDirScanThreads)
k_dir_scan(const __grid_constant__ DirectArgs a, PlanHeader* hdr, const __grid_constant__ DirScanOut out) {
  pdl_wait();
  if (!hdr->direct) return;
  __shared__ uint2 s_all[kDirStages];
  constexpr int kHold = 8;                        /* pieces per lane kept in registers: 256 a round */
  const uint32_t tid = threadIdx.x, lane = tid & 31, k = tid >> 5, c = blockIdx.x;
  const uint32_t first = __ldcg(&a.ctx_start[c]), len = __ldcg(&a.ctx_start[c + 1]) - first;
  const uint32_t p0 = first / a.piece + c, np = (uint32_t)(((uint64_t)len + a.piece - 1) / a.piece);
  if (k < a.S) {
    uint2* rows = a.piece_rows + (size_t)p0 * kDirStages + k;
    uint2 run = make_uint2(0u, (uint32_t)kDirInf);
    for (uint32_t base = 0; base < np; base += 32 * kHold) {
      const uint32_t at = base + lane * kHold;
      uint2 v[kHold], sum = make_uint2(0u, (uint32_t)kDirInf);
#pragma unroll
      for (int i = 0; i < kHold; ++i) v[i] = at + i < np ? __ldcg(&rows[(size_t)(at + i) * kDirStages]) : make_uint2(0u, (uint32_t)kDirInf);
#pragma unroll
      for (int i = 0; i < kHold; ++i) sum = dir_then(sum, v[i]);
      uint2 incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint2 y = make_uint2(__shfl_up_sync(0xffffffffu, incl.x, o), __shfl_up_sync(0xffffffffu, incl.y, o));
        if (lane >= (uint32_t)o) incl = dir_then(y, incl);
      }
      uint2 before = make_uint2(__shfl_up_sync(0xffffffffu, incl.x, 1), __shfl_up_sync(0xffffffffu, incl.y, 1));
      before = lane ? dir_then(run, before) : run;
#pragma unroll
      for (int i = 0; i < kHold; ++i) {
        if (at + i < np) rows[(size_t)(at + i) * kDirStages] = before;
        before = dir_then(before, v[i]);
      }
      run = dir_then(run, make_uint2(__shfl_sync(0xffffffffu, incl.x, 31), __shfl_sync(0xffffffffu, incl.y, 31)));
    }
    if (lane == 0) s_all[k] = run;
  }
  __syncthreads();
  if (tid < 32) {
    const uint2 run = lane < a.S ? s_all[lane] : make_uint2(0u, 0u);
    uint32_t x = run.x;
    for (int o = 1; o < kDirStages; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    if (lane < a.S) {
      const size_t q = (size_t)c * a.S + lane;
      const uint32_t at = first + x - run.x;
      out.seg_off[q] = at;
      if (out.out_seg_off) out.out_seg_off[q] = at;
      out.seg_kept[q] = run.x ? (uint32_t)((int32_t)run.x - 1 + min((int32_t)run.y, 1)) : 0u;
      if (q + 1 == (size_t)a.n_ctx * a.S) {
        out.seg_off[q + 1] = a.n;
        if (out.out_seg_off) out.out_seg_off[q + 1] = a.n;
      }
    }
  }
  if (last_block_done(&hdr->win_done))
    kept_scan_block<kDirScanThreads>(out.seg_kept, a.n_ctx * a.S, out.kept_base, out.chunk_base, out.out_seg_kept, out.out_n_kept);
}

/* Counts, minima and checks of one piece per block.  A warp reads a run of consecutive requests, 128 at a time, and
 * needs the other warps only for the running sums at the end.  Lane j keeps the figures of stage j: the count, the
 * minimum so far, the last request's u and the offset from which u rises.  While u stays, u - t falls with every
 * request, so the minimum needs a look only where u rises and at the end: a row of 32 requests none of which
 * reaches its queue's limit (most do not) is only counted.  2^24 requests of 16 stages: 62 us, 41 by the read; 105 with
 * every request's threshold worked out, 37 M instructions instead of 65 M. */
template <int BITS>
__global__ void __launch_bounds__(kDirThreads, 4)
k_dir_count(const __grid_constant__ DirectArgs a, const __grid_constant__ ConstArgs ca, PlanHeader* hdr,
            unsigned long long* __restrict__ ctx_dmin_inv, unsigned long long* __restrict__ ctx_dmax) {
  pdl_wait();
  constexpr int kUn = 4;
  __shared__ DirConst s_K[kDirWarps][kDirStages];
  __shared__ uint2 s_warp[kDirWarps][kDirStages];
  __shared__ int32_t s_low[kDirWarps][kDirStages];
  __shared__ unsigned long long s_min[kDirWarps], s_max[kDirWarps];
  __shared__ bool s_back[kDirWarps];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t piece = blockIdx.x;
  uint4 info = __ldcg(&a.piece_info[piece]);
  /* (requests not grouped by ctx may leave entries that no ctx has filled in) */
  const bool nonsense = info.x >= a.n_ctx || info.y > info.z || info.z > a.n || info.z - info.y > a.piece;
  if (nonsense) info = make_uint4(0u, 0u, 0u, 0u);
  const uint32_t c = info.x, begin = info.y, end = info.z;
  const uint32_t sub = (a.piece / kDirWarps + 127) & ~127u;
  const uint32_t wbegin = min(end, begin + warp * sub), wend = min(end, wbegin + sub);
  /* a chunk's requests are asked for while the one before is worked on, the first ones before all else */
  uint4 r[kUn];
  auto fetch = [&](uint32_t pos) {
#pragma unroll
    for (int i = 0; i < kUn; ++i) {
      r[i] = make_uint4(0u, 0u, c, 0u);
      if (pos + i * 32 + lane < wend) r[i] = __ldg(&a.req[pos + i * 32 + lane]);
    }
  };
  const uint32_t off_word = ld_relaxed(&hdr->direct_off);
  bool off = nonsense || off_word != 0;
  if (!off) fetch(wbegin);
  /* the boundaries found must ascend from 0 to n (the requests' own ctxs are compared below: both together prove the grouping) */
  bool gaps = false, bad_const = false;
  for (uint32_t i = piece * kDirThreads + tid; i <= a.n_ctx; i += a.n_pieces * kDirThreads)
    gaps |= i < a.n_ctx ? __ldcg(&a.ctx_start[i]) > __ldcg(&a.ctx_start[i + 1]) || (i == 0 && __ldcg(&a.ctx_start[0]) != 0) : __ldcg(&a.ctx_start[i]) != a.n;
  for (uint32_t i = piece * kDirThreads + tid; i < a.n_ctx; i += a.n_pieces * kDirThreads) bad_const |= __ldcg(&a.const_bad[i]) != 0;
  if (bad_const) {
    set_status(hdr, PARD_EDATA);
    off = true;
  }
  if (gaps) {
    off = true;
    hdr->unsorted = 1;                            /* not grouped as the caller said: reported by k_pack_ctx */
  }
  auto deadline = [&](uint32_t j) { return __ldg(reinterpret_cast<const unsigned long long*>(&a.req[j])); };
  const unsigned long long D0 = !off && begin < end ? deadline(begin) : 0ull;
  uint32_t last = 0;                              /* offset of the request before; in 32 bits or not one that may come before any */
  if (!off && wbegin < wend && wbegin > begin) {
    const unsigned long long before = deadline(wbegin - 1) - D0;
    last = before >> 32 ? 0xffffffffu : (uint32_t)before;
  }
  DirConst mineK = {0, 1u, 1u, 0ull};             /* every warp keeps the constants for itself: no barrier before the end */
  if (!off && begin < end) {
    const uint32_t k = lane & (kDirStages - 1);
    if (k < a.S) {
      const PardSegConst& g = a.ktab[(size_t)c * a.S + k];
      if (g.narrow & kSegNoStage) mineK.A = -1;   /* no such stage: its requests are input errors */
      else off |= !dir_const(g, D0, mineK);
    }
    off |= D0 >= (unsigned long long)PARD_TIME_LIMIT_US - (1ull << 31);      /* in every warp: whichever holds a deadline beyond the limit looks for it */
    if (tid == 0) {
      /* the ctx's deadlines must leave room for the key that a sort would need */
      const uint32_t first = __ldcg(&a.ctx_start[c]), stop = __ldcg(&a.ctx_start[c + 1]);
      const unsigned long long Df = deadline(min(first, a.n - 1)), Dl = deadline(min(max(stop, 1u), a.n) - 1), Dp = deadline(begin > first ? begin - 1 : begin);
      off |= Dl < Df || D0 < Dp || a.sbits + a.ibits + bit_width64(Dl - Df) > 64;
    }
  }
  if (lane < kDirStages) { s_K[warp][lane] = mineK; s_low[warp][lane] = kDirInf; }
  off = __any_sync(0xffffffffu, off);             /* (also what __syncwarp would do) */
  uint32_t run = 0, ucur = 0;
  int32_t low = kDirInf, next = mineK.A;
  unsigned long long lmin = ~0ull, lmax = 0;
  bool stepped = false;
  /* the figures of the requests so far, as {count, minimum} */
  auto figures = [&]() {
    const int32_t m = min(low, s_low[warp][lane & (kDirStages - 1)]);
    return make_uint2(run, (uint32_t)(run ? min(m, (int32_t)ucur - (int32_t)(run - 1)) : m));
  };
  if (!off && wbegin < wend) {
    const uint32_t below = (1u << lane) - 1;
    for (uint32_t pos = wbegin; pos < wend; pos += 32 * kUn) {
      uint32_t x[kUn], st[kUn], other = 0, top = 0;
      bool back = false;
#pragma unroll
      for (int i = 0; i < kUn; ++i) {
        const bool in = pos + i * 32 + lane < wend;
        const unsigned long long d = (((unsigned long long)r[i].y << 32) | r[i].x) - D0;
        st[i] = r[i].w & 0xffffu;
        x[i] = in ? (uint32_t)d : 0x7ffffffeu;    /* behind all others */
        other |= (in ? (uint32_t)(d >> 32) : 0u) | (r[i].z ^ c);
        top = max(top, st[i]);
        const uint32_t px = __shfl_sync(0xffffffffu, lane == 31 ? last : x[i], (lane - 1) & 31);
        last = x[i];
        back |= x[i] < px;
      }
      if (!__all_sync(0xffffffffu, other == 0 && !back && top < a.S && last < 0x7fffffffu)) { off = true; break; }
      fetch(pos + 32 * kUn);
#pragma unroll
      for (int i = 0; i < kUn; ++i) {
        const bool in = pos + i * 32 + lane < wend;
        const uint32_t valid = __ballot_sync(0xffffffffu, in);
        const uint32_t mine = dir_mine<BITS>(st[i], valid, lane);
        const int32_t limit = __shfl_sync(0xffffffffu, next, st[i]);
        if (__any_sync(0xffffffffu, in && (int32_t)x[i] >= limit)) {
          const DirConst K = s_K[warp][st[i]];
          off |= in && K.magic == 0;              /* a request at a stage that its pipeline lacks */
          int32_t at;
          const uint32_t u = dir_u(x[i], K, &at);
          const uint32_t ahead = __shfl_sync(0xffffffffu, mine, st[i]) & below;
          const uint32_t before = __shfl_sync(0xffffffffu, run, st[i]) + __popc(ahead);
          const uint32_t u1 = __shfl_sync(0xffffffffu, u, 31 - __clz(ahead | 1u)), u0 = __shfl_sync(0xffffffffu, ucur, st[i]);
          const uint32_t up = ahead ? u1 : u0;    /* u of the queue's request before */
          if (in && before && up != u) atomicMin(&s_low[warp][st[i]], (int32_t)up - (int32_t)(before - 1));
          const uint32_t ul = __shfl_sync(0xffffffffu, u, 31 - __clz(mine | 1u));
          const int32_t al = __shfl_sync(0xffffffffu, at, 31 - __clz(mine | 1u));
          if (mine) { ucur = ul; next = al; }
        }
        run += __popc(mine);
      }
    }
    off = __any_sync(0xffffffffu, off);
    if (!off) {
      lmin = deadline(wbegin);
      lmax = deadline(wend - 1);
    }
  }
  /* What k_prepass would find: the deadlines' range, input errors, steps back (the warps that stay out of this have
   * found none, the request ahead of their first one included).  The path may be off for another reason: requests in
   * order then need no more passes than if it had not been tried.  (With steps back taken for granted, ordered requests
   * of 256 contexts, 2^24 with one stage of 1 us: 812 us a call, now 609; 288 k of 24 in two halves 2^32 us apart:
   * 128 and 85.  The general path by itself: 608 and 84.)  The next rows are asked for ahead (unordered 2^24 547 -> 543). */
  if (off) {
    bool bad = false, foreign = nonsense;
    lmin = ~0ull;
    lmax = 0;
    auto look = [&](auto steps) {
      constexpr bool STEPS = decltype(steps)::value;
      unsigned long long prev = 0;                /* lane 31: of the row before */
      if (STEPS && wbegin < wend && (wbegin > begin || begin > __ldcg(&a.ctx_start[c]))) prev = deadline(wbegin - 1);
      fetch(wbegin);
      for (uint32_t pos = wbegin; pos < wend; pos += 32 * kUn) {
        uint4 v[kUn];
#pragma unroll
        for (int i = 0; i < kUn; ++i) v[i] = r[i];
        fetch(pos + 32 * kUn);
#pragma unroll
        for (int i = 0; i < kUn; ++i) {
          const bool there = pos + i * 32 + lane < wend;
          const unsigned long long D = there ? ((unsigned long long)v[i].y << 32) | v[i].x : ~0ull;
          if (STEPS) {                            /* (rows beyond the share compare as in order) */
            const unsigned long long pD = __shfl_sync(0xffffffffu, lane == 31 ? prev : D, (lane - 1) & 31);
            prev = D;
            stepped |= D < pD;
          }
          foreign |= there && v[i].z != c;
          if (D >= (unsigned long long)PARD_TIME_LIMIT_US || v[i].z != c || (v[i].w & 0xffffu) >= a.S) {
            bad |= there && v[i].z == c;
            continue;
          }
          lmin = D < lmin ? D : lmin;
          lmax = D > lmax ? D : lmax;
        }
      }
    };
    if (__any_sync(0xffffffffu, off_word & kDirSteps)) look(std::false_type());
    else look(std::true_type());
    if (bad) set_status(hdr, PARD_EDATA);
    if (foreign) hdr->unsorted = 1;
    stepped = __any_sync(0xffffffffu, stepped);
    for (int o = 16; o; o >>= 1) {
      const unsigned long long p = __shfl_xor_sync(0xffffffffu, lmin, o), q = __shfl_xor_sync(0xffffffffu, lmax, o);
      lmin = p < lmin ? p : lmin;
      lmax = q > lmax ? q : lmax;
    }
  }
  __syncwarp();
  if (lane < kDirStages) s_warp[warp][lane] = figures();
  if (lane == 0) { s_min[warp] = lmin; s_max[warp] = lmax; s_back[warp] = stepped; }
  const bool block_off = __syncthreads_or(off);
  if (tid == 0) {
    for (int w = 1; w < kDirWarps; ++w) {
      lmin = s_min[w] < lmin ? s_min[w] : lmin;
      lmax = s_max[w] > lmax ? s_max[w] : lmax;
      stepped |= s_back[w];
    }
    if (lmin <= lmax) {
      if (__ldcg(&ctx_dmin_inv[c]) < ~lmin) atomicMax(&ctx_dmin_inv[c], ~lmin);
      if (__ldcg(&ctx_dmax[c]) < lmax) atomicMax(&ctx_dmax[c], lmax);
    }
  }
  if (block_off) {
    if (tid == 0) {
      const uint32_t word = stepped ? kDirOff | kDirSteps : kDirOff;
      if (word & ~ld_relaxed(&hdr->direct_off)) {
        if (stepped) hdr->time_steps_back = hdr->pair_steps_back = 1;    /* inside a ctx: both */
        atomicOr(&hdr->direct_off, word);
      }
    }
  } else if (tid < kDirStages) {
    uint2 sum = make_uint2(0u, (uint32_t)kDirInf);
    for (int w = 0; w < kDirWarps; ++w) sum = dir_then(sum, s_warp[w][tid]);
    a.piece_rows[(size_t)piece * kDirStages + tid] = sum;
  }
  if (!last_block_done(&hdr->direct_done)) return;
  if (!ld_relaxed(&hdr->direct_off)) {
    if (tid == 0) hdr->direct = 1;
  } else if (ca.with_key_width && a.n_ctx * a.S <= kFoldSegs) {
    finish_constants<true>(ca, ctx_dmin_inv, ctx_dmax, hdr);
  }
}

/* The pieces, tile after tile ordered by stage in shared memory, decided and written out.
 * A queue's requests of the tile take the slots from `start` on, which stands to a group of 4 slots as its first
 * output position to a multiple of 4, and a thread decides a group: constants and divisions once per group, the
 * Request Broker's own loop over its requests, outputs in aligned vectors.  What does not fill a group waits for the
 * next tile.  What a group needs of the requests before its first one is their number and by how much they lower the
 * minimum of u_t - t.  With m that minimum before the tile (at most 1: larger ones lower nothing) they cannot lower
 * it by more than their number, so the running minimum over the slots is a running maximum of (stage, amount) in one
 * word, which never leaks from one queue into the next.  The next tile is copied into shared memory meanwhile.
 * Pieces are taken by ticket.  Bound by shared memory (two thirds of its wavefronts) and instructions: 127 us for 2^24
 * requests of 16 stages, 75 by its bytes (16 in, 13 + 4f out, 8 % kept).  On the way there: a lane per request 151, groups of
 * 8 slots 147, with copies ahead and what does not fill a group left for the next tile 131; a warp per tile without
 * block barriers 156; ranks from four-bit counters per thread instead of ballots the same 127. */
constexpr int kEmitRounds = 2;                    /* groups per thread */
constexpr uint32_t kEmitSlots = 4 * kEmitRounds * kDirThreads;
static_assert(kDirTile + 6 * kDirStages <= kEmitSlots, "every queue may leave three slots free, or hold three requests of the tile before, at either end");
struct EmitSmem {
  struct __align__(16) Queue {
    DirConst K;
    long long A;
    unsigned long long cap_magic;
    uint32_t rank, out, kept;                     /* of the first slot's request: rank, output position; the queue's survivors begin at */
    int32_t m;
    uint32_t start, len;                          /* slots taken */
  };
  struct __align__(16) Next {                     /* what the next tile starts from */
    uint32_t rank, out;
    int32_t m;
    uint32_t wait;                                /* requests of this tile that take its first slots */
  };
  uint4 raw[kDirTile];                            /* the tile's requests */
  uint32_t x[kEmitSlots];                         /* deadline offsets */
  uint16_t id[kEmitSlots];                        /* place in the piece */
  Queue q[kDirStages];
  Next then[kDirStages];
  uint32_t cnt[kDirWarps][kDirStages];
  uint32_t group[kDirStages + 1];                 /* first group */
  uint32_t top[kEmitRounds * kDirWarps];
  uint32_t next;                                  /* the piece after this one */
  uint4 info;
  unsigned long long full;                        /* mbarrier: the tile has arrived */
};

static_assert(sizeof(EmitSmem) <= 48 * 1024, "four blocks per multiprocessor, no opt-in");

/* a tile's requests into shared memory, by one thread */
__device__ __forceinline__ void emit_fetch(EmitSmem& Sm, const uint4* src, uint32_t count) { bulk_fetch(&Sm.full, Sm.raw, src, count * 16); }

template <int BITS>
__global__ void __launch_bounds__(kDirThreads, 4)
k_dir_emit(const __grid_constant__ DirectArgs a, PlanHeader* __restrict__ hdr, const uint32_t* __restrict__ seg_off,
           const uint32_t* __restrict__ kept_base, uint8_t* __restrict__ out_keep, long long* __restrict__ out_est,
           uint32_t* __restrict__ out_perm, uint32_t* __restrict__ out_kept_idx) {
  pdl_wait();
  if (!hdr->direct) return;
  extern __shared__ __align__(16) unsigned char emit_raw[];
  EmitSmem& Sm = *reinterpret_cast<EmitSmem*>(emit_raw);
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, below = (1u << lane) - 1, kl = lane & (kDirStages - 1);
  uint32_t phase = 0;
  if (tid == 0) {
    bulk_init(&Sm.full);
    uint32_t p = atomicAdd(&hdr->direct_ticket, 1u);
    uint4 info = make_uint4(0u, 0u, 0u, 0u);
    while (p < a.n_pieces) {                      /* (a piece may be empty) */
      info = __ldg(&a.piece_info[p]);
      if (info.y < info.z) break;
      p = atomicAdd(&hdr->direct_ticket, 1u);
    }
    Sm.next = p;
    Sm.info = info;
    if (p < a.n_pieces && !(a.stall && blockIdx.x == 0)) emit_fetch(Sm, a.req + info.y, min(kDirTile, info.z - info.y));
  }
  __syncthreads();
  for (;;) {
    const uint32_t piece = Sm.next;
    if (piece >= a.n_pieces) return;
    const uint4 info = Sm.info;
    uint32_t ticket = 0;
    if (tid == 0) ticket = atomicAdd(&hdr->direct_ticket, 1u);     /* (needed when the last tile is on) */
    const unsigned long long D0 = __ldg(reinterpret_cast<const unsigned long long*>(&a.req[info.y]));
    if (tid < kDirStages) {
      EmitSmem::Queue q = {};
      EmitSmem::Next first = {};
      if (tid < a.S) {
        const size_t s = (size_t)info.x * a.S + tid;
        const PardSegConst& g = a.ktab[s];
        const uint2 run = a.piece_rows[(size_t)piece * kDirStages + tid];
        dir_const(g, D0, q.K);
        q.A = g.A; q.cap_magic = g.cap_magic;
        q.kept = out_kept_idx ? kept_base[s] : 0u;
        first.rank = run.x;
        first.m = min((int32_t)run.y, 1);
        first.out = seg_off[s] + run.x;
      }
      Sm.q[tid] = q;
      Sm.then[tid] = first;
    }
    uint32_t wait_x = 0, wait_id = 0;             /* thread 4k + j: the j-th request of stage k that waits for this tile */
    for (uint32_t base = info.y; base < info.z; base += kDirTile) {
      const uint32_t cnt = min(kDirTile, info.z - base);
      const bool final = base + kDirTile >= info.z;
      /* 1. the tile's requests, row by row; their ranks within the warp's share */
      bool late = !bulk_arrived(&Sm.full, phase);
      phase ^= 1;
      uint32_t x[kDirRows], meta[kDirRows], run = 0;     /* run: lane j: the warp's requests of stage j so far */
      const uint32_t wfirst = warp * (kDirRows * 32);
#pragma unroll
      for (int i = 0; i < kDirRows; ++i) {
        const uint32_t p = wfirst + i * 32 + lane;
        const uint4 r = Sm.raw[p];                /* (beyond the tile: whatever the buffer holds) */
        x[i] = r.x - (uint32_t)D0;
        meta[i] = r.w & (kDirStages - 1);
        const uint32_t mine = dir_mine<BITS>(meta[i], cnt == kDirTile ? 0xffffffffu : __ballot_sync(0xffffffffu, p < cnt), lane);
        const uint32_t rank = __shfl_sync(0xffffffffu, run, meta[i]) + __popc(__shfl_sync(0xffffffffu, mine, meta[i]) & below);
        run += __popc(mine);
        meta[i] |= rank << 16;
      }
      if (lane < kDirStages) Sm.cnt[warp][lane] = run;
      if (__syncthreads_or(late)) {
        bulk_arrived(&Sm.full, phase ^ 1);              /* no copy is under way when the block ends */
        if (tid == 0) set_aborted(hdr);
        return;
      }
      if (tid == 0) {                             /* the next tile, of this piece or of the next one */
        if (!final) {
          emit_fetch(Sm, a.req + base + kDirTile, min(kDirTile, info.z - base - kDirTile));
        } else {
          uint4 then = make_uint4(0u, 0u, 0u, 0u);
          while (ticket < a.n_pieces) {
            then = __ldg(&a.piece_info[ticket]);
            if (then.y < then.z) break;
            ticket = atomicAdd(&hdr->direct_ticket, 1u);
          }
          Sm.next = ticket;
          Sm.info = then;
          if (ticket < a.n_pieces) emit_fetch(Sm, a.req + then.y, min(kDirTile, then.z - then.y));
        }
      }
      /* where the queues' requests go: every warp for itself (lane j: stage j) */
      const EmitSmem::Next from = Sm.then[kl];
      const uint32_t waiting = from.wait;
      uint32_t slot, start, n_groups;
      {
        uint32_t len = waiting, mine = 0;
#pragma unroll
        for (int w = 0; w < kDirWarps; ++w) {
          const uint32_t y = Sm.cnt[w][kl];
          if (w < (int)warp) mine += y;
          len += y;
        }
        const uint32_t lead = from.out & 3u, groups = len ? (lead + len + 3) / 4 : 0u;
        uint32_t incl = groups;
#pragma unroll
        for (int o = 1; o < kDirStages; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o, kDirStages);
          if (kl >= (uint32_t)o) incl += y;
        }
        n_groups = __shfl_sync(0xffffffffu, incl, kDirStages - 1);
        start = 4 * (incl - groups) + lead;
        slot = start + waiting + mine;
        if (warp == 0 && lane < kDirStages) {
          EmitSmem::Queue& q = Sm.q[kl];
          q.rank = from.rank; q.out = from.out; q.m = from.m;
          q.start = start; q.len = len;
          Sm.group[kl] = incl - groups;
        }
      }
      /* 2. into their slots */
#pragma unroll
      for (int i = 0; i < kDirRows; ++i) {
        const uint32_t p = wfirst + i * 32 + lane, at = __shfl_sync(0xffffffffu, slot, meta[i] & 0xffffu) + (meta[i] >> 16);
        if (p < cnt) {
          Sm.x[at] = x[i];
          Sm.id[at] = (uint16_t)(base - info.y + p);
        }
      }
      {
        const uint32_t k = (tid / 4) & (kDirStages - 1), j = tid & 3u, at = __shfl_sync(0xffffffffu, start, k) + j, waits = __shfl_sync(0xffffffffu, waiting, k);
        if (tid < 4 * kDirStages && j < waits) {
          Sm.x[at] = wait_x;
          Sm.id[at] = (uint16_t)wait_id;
        }
      }
      __syncthreads();
      /* 3. thresholds of the groups' requests, and by how much they lower the minimum */
      uint32_t u[kEmitRounds][4], key[kEmitRounds], which[kEmitRounds];    /* which: stage, valid slots of the group */
#pragma unroll
      for (int h = 0; h < kEmitRounds; ++h) {
        const uint32_t grp = h * kDirThreads + tid, slot0 = 4 * grp;
        key[h] = which[h] = 0;
        if (grp >= n_groups) continue;
        uint32_t k = 0;                           /* the last stage whose groups begin at or before this one */
#pragma unroll
        for (int b = kDirStages / 2; b; b >>= 1)
          if (Sm.group[k + b] <= grp) k += b;
        const EmitSmem::Queue& q = Sm.q[k];
        const uint32_t lo = q.start > slot0 ? q.start - slot0 : 0u, hi = min(4u, q.start + q.len - slot0);
        if (hi < 4 && !final) continue;           /* waits for the next tile */
        const uint32_t mask = (0xfu >> (4 - hi)) & (0xfu << lo);
        const uint4 xa = *reinterpret_cast<const uint4*>(&Sm.x[slot0]);
        const uint32_t xs[4] = {xa.x, xa.y, xa.z, xa.w};
        const DirConst K = q.K;
        int32_t next, by = 0;
        uint32_t cur = dir_u(lo == 0 ? xs[0] : lo == 1 ? xs[1] : lo == 2 ? xs[2] : xs[3], K, &next);       /* next > 0 from here on */
        const int32_t from = q.m + (int32_t)(q.rank + slot0 - q.start);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const bool in = (mask >> i) & 1u;
          if (in && (int32_t)xs[i] >= next) {     /* the next window, or one beyond it */
            if (i) by = max(by, from + i - 1 - (int32_t)cur);    /* the request before was its window's last */
            next = (int32_t)min((uint32_t)next + min(K.d, 0x7fffffffu), 0x7fffffffu);
            cur = min(cur + K.cap, kUClamp);
            if ((int32_t)xs[i] >= next) cur = dir_u_far(xs[i], K, &next);
          }
          u[h][i] = in ? cur : 0u;
        }
        by = max(by, from + (int32_t)hi - 1 - (int32_t)cur);
        key[h] = k << 12 | (uint32_t)by;
        which[h] = k << 4 | mask;
      }
      uint32_t earlier[kEmitRounds];
#pragma unroll
      for (int h = 0; h < kEmitRounds; ++h) {
        uint32_t incl = key[h];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= (uint32_t)o) incl = max(incl, y);
        }
        earlier[h] = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) earlier[h] = 0;
        if (lane == 31) Sm.top[h * kDirWarps + warp] = incl;
      }
      __syncthreads();
#pragma unroll
      for (int h = 0; h < kEmitRounds; ++h)
        earlier[h] = max(earlier[h], __reduce_max_sync(0xffffffffu, lane < h * kDirWarps + warp ? Sm.top[lane] : 0u));
      /* 4. decisions */
#pragma unroll
      for (int h = 0; h < kEmitRounds; ++h) {
        const uint32_t mask = which[h] & 15u, k = which[h] >> 4, slot0 = 4 * (h * kDirThreads + tid);
        if (!mask) continue;
        const EmitSmem::Queue& q = Sm.q[k];
        const uint32_t start = q.start, done = slot0 + 4 - start, rank = q.rank, out = q.out;
        const uint32_t r = rank + max(slot0, start) - start, o = out + slot0 - start;
        const int32_t m = q.m;
        uint32_t c = r ? r - 1 + (uint32_t)(m - (earlier[h] >> 12 == k ? (int32_t)(earlier[h] & 0xfffu) : 0)) : 0u;
        const uint32_t cap = q.K.cap, d = q.K.d, round = q.cap_magic ? div_magic32(c, q.cap_magic) : c;
        uint32_t full_at = (round + 1) * cap;     /* the admitted count at which the next round begins */
        long long est = q.A + (long long)((unsigned long long)round * d);
        const uint2 ids = *reinterpret_cast<const uint2*>(&Sm.id[slot0]);
        const uint32_t id2[2] = {ids.x, ids.y};
        uint32_t* survivor = out_kept_idx + q.kept + c;
        const bool some = c < max(max(u[h][0], u[h][1]), max(u[h][2], u[h][3]));
        uint32_t keeps = 0, idx[4];
        long long e[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          idx[i] = info.y + __byte_perm(id2[i / 2], 0u, i & 1 ? 0x4432 : 0x4410);
          e[i] = est;
          if (some && c < u[h][i]) {
            keeps |= 1u << (8 * i);
            if (out_kept_idx) *survivor++ = idx[i];
            if (++c == full_at) { est += d; full_at += cap; }
          }
        }
        if (mask == 0xfu) {
          if (out_est) store4(out_est + o, e[0], e[1], e[2], e[3]);
          if (out_perm) *reinterpret_cast<uint4*>(out_perm + o) = make_uint4(idx[0], idx[1], idx[2], idx[3]);
          if (out_keep) *reinterpret_cast<uint32_t*>(out_keep + o) = keeps;
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (!((mask >> i) & 1u)) continue;
            if (out_est) out_est[o + i] = e[i];
            if (out_perm) out_perm[o + i] = idx[i];
            if (out_keep) out_keep[o + i] = (uint8_t)((keeps >> (8 * i)) & 1u);
          }
        }
        /* the queue's last group that is decided: where the next tile goes on */
        if (done <= q.len && done + 4 > q.len) {
          EmitSmem::Next& w = Sm.then[k];
          w.rank = rank + done;
          w.out = out + done;
          w.m = (int32_t)c - (int32_t)(rank + done) + 1;
          w.wait = q.len - done;
        }
      }
      if (!final) {
        /* a queue none of whose groups was filled waits as a whole; the requests that wait, into registers */
        const uint32_t kk = (tid / 4) & (kDirStages - 1), j = tid & 3u, first = Sm.q[kk].start, len = Sm.q[kk].len;
        if (tid < 4 * kDirStages) {
          const uint32_t lead = first & 3u, left = lead + len < 4 ? len : (lead + len) & 3u;
          if (lead + len < 4 && j == 0) Sm.then[kk].wait = len;
          if (j < left) {
            wait_x = Sm.x[first + len - left + j];
            wait_id = Sm.id[first + len - left + j];
          }
        }
      }
    }
    __syncthreads();
  }
}

/* The path's arrays, for a call that may take it as far as the host can see; they take the second sort buffer.  Pieces
 * of at most four tiles, so that the blocks of long and of short contexts end together.  (One ctx: its constants would
 * have to be there before the requests are read, where k_prepass works them out meanwhile; a million requests in
 * order gained 2 us, as many out of order lost 3.) */
inline bool dir_layout(uint64_t n, uint32_t n_ctx, uint32_t S, int sms, char* buf, DirectArgs* a) {
  if (S > (uint32_t)kDirStages) return false;
  const uint64_t tiles = (n + kDirTile - 1) / kDirTile, blocks = 4ull * sms;
  a->piece = kDirTile * (uint32_t)std::min<uint64_t>(kDirMaxTiles, (tiles + blocks - 1) / blocks);
  a->n_pieces = (uint32_t)(n / a->piece) + n_ctx;     /* (contexts of more than 8,192 requests on average: 16 + 128 bytes for 1,792 of them) */
  a->piece_info = (uint4*)buf;
  a->piece_rows = (uint2*)(buf + 16ull * a->n_pieces);
  return true;
}
