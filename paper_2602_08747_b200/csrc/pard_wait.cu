/* Batch-wait estimate w = F^{-1}(lambda) of the State Planner (paper Sec. 4.2,
 * Batch wait estimation): for every (ctx, stage, downstream path) slot, M
 * samples of the batch wait aggregated over the path's stages, and the sample
 * of rank floor(lambda * M).
 *
 * A block takes every G-th slot of one ctx.  The recorded waits of one stage at a time are copied
 * into shared memory, asynchronously and one row ahead (across slots too), and the draws gather
 * from there; a thread keeps the sums of its samples in registers.  The rank-th smallest sum: a
 * histogram over the top 11 of the bits that occur, a scan of it, then the few sums of the one bin
 * that holds the rank are compared with each other (or, if they are many, split again).
 * Bound by the integer pipes (multiplications and logic both near 60 % of their cycles, issue slots
 * at 68 %): of some 35 instructions per draw two thirds are splitmix64.  M = 10,000 on the
 * 4,500 slots of 256 pipelines (262 M draws): 635 us with a block of its own for every slot of the
 * stride -- most of them padding, each paying five dependent loads to find its path --, the sums
 * in shared memory and four rounds of selection over all of them; 430 us like this. */
#include <algorithm>
#include <mutex>

#include "pard_plan_internal.cuh"

using namespace pard_plan_detail;

namespace {

constexpr uint32_t kSampleBits = 24;             /* recorded waits lie in [0, 2^24) us */
constexpr uint32_t kSelBits = 11, kSelBins = 1u << kSelBits;

struct WaitHeader {
  uint32_t status;                               /* 0, or the positive value of a pard_status */
  uint32_t pad[63];
};
static_assert(sizeof(WaitHeader) == 256, "header is 256 bytes");

struct WaitArgs {
  uint32_t n_pipelines;
  const int32_t* pipeline_of_ctx;
  uint32_t S, R, M, G, rank;
  const int32_t* samples;
  unsigned long long seed;
  long long* w_out;
  WaitHeader* hdr;
};

/* High word of splitmix64 (Steele, Lea, Flood 2014): the finaliser applied to counter + gamma, given
 * as two words that already hold the sum.  The counters of one slot are neighbours: unless their low
 * words wrap around inside the slot (SAME_HI is false then) the high word is the same for all draws,
 * and so is its part of the first product, `fixed`. */
constexpr unsigned long long kMixA = 0xBF58476D1CE4E5B9ull, kMixB = 0x94D049BB133111EBull;
__device__ __forceinline__ unsigned long long splitmix_fixed(uint32_t hi) {
  return (unsigned long long)((hi ^ (hi >> 30)) * (uint32_t)kMixA) << 32;
}
/* the rest, from the low word after the first shift */
__device__ __forceinline__ uint32_t splitmix_rest(uint32_t l, unsigned long long fixed) {
  unsigned long long z = (unsigned long long)l * (uint32_t)kMixA + fixed;
  z += (unsigned long long)(l * (uint32_t)(kMixA >> 32)) << 32;
  z = (z ^ (z >> 27)) * kMixB;
  const uint32_t h = (uint32_t)(z >> 32);
  return h ^ (h >> 31);
}
__device__ __forceinline__ uint32_t splitmix_hi(uint32_t lo, uint32_t hi, unsigned long long fixed) {
  return splitmix_rest(lo ^ __funnelshift_r(lo, hi, 30), fixed);
}

__device__ __forceinline__ void copy_async_16(uint32_t smem, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem), "l"(g) : "memory");
}
__device__ __forceinline__ void copy_async_4(uint32_t smem, const void* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem), "l"(g) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

/* one row of M recorded waits into shared memory; 16 bytes at a time where rows start on such a boundary */
template <int THREADS>
__device__ __forceinline__ void copy_row(uint32_t* dst, const int32_t* row, uint32_t M) {
  const uint32_t s = (uint32_t)__cvta_generic_to_shared(dst);
  if (((uintptr_t)row & 15) == 0) {
    for (uint32_t q = threadIdx.x; q < M / 4; q += THREADS) copy_async_16(s + 16 * q, row + 4 * q);
    for (uint32_t m = (M & ~3u) + threadIdx.x; m < M; m += THREADS) copy_async_4(s + 4 * m, row + m);
  } else {
    for (uint32_t m = threadIdx.x; m < M; m += THREADS) copy_async_4(s + 4 * m, row + m);
  }
}

/* THREADS * PER >= M.  DOUBLE: two row buffers, the next row is copied while this one is drawn from. */
template <int THREADS, int PER, bool DOUBLE>
__global__ void __launch_bounds__(THREADS, THREADS >= 1024 ? 1 : 1024 / THREADS)
k_estimate_w(const __grid_constant__ PipeTable pipes, const WaitArgs a) {
  pdl_wait();
  constexpr int WARPS = THREADS / 32, kGroup = 4;
  static_assert(PER % kGroup == 0, "whole groups");
  extern __shared__ __align__(16) uint32_t s_rows[];         /* one or two rows, each padded to 16 bytes */
  __shared__ uint32_t s_hist[kSelBins];
  __shared__ int32_t s_path[2][PARD_MAX_STAGES];
  __shared__ uint32_t s_len[2], s_warp[WARPS], s_bin, s_left, s_count;
  __shared__ uint32_t s_cand[THREADS];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t c = blockIdx.x / a.G, g = blockIdx.x % a.G, M = a.M;
  const int32_t pi = a.pipeline_of_ctx ? a.pipeline_of_ctx[c] : 0;
  if (pi < 0 || (uint32_t)pi >= a.n_pipelines) {
    if (tid == 0) atomicMax(&a.hdr->status, (uint32_t)(-PARD_EDATA));
    return;
  }
  const PardPipeDev* P = a.n_pipelines <= (uint32_t)kFewPipelines ? pipes.few[pi] : pipes.many[pi];
  const uint32_t n_slots = (uint32_t)P->n_slots;             /* slots beyond it are padding: left untouched */
  if (n_slots > a.R || (uint32_t)P->n_stages > a.S) {
    if (tid == 0) atomicMax(&a.hdr->status, (uint32_t)(-PARD_EDATA));
    return;
  }
  if (g >= n_slots) return;
  const int32_t* __restrict__ path_off = P->path_off;
  const int32_t* __restrict__ path_stage = P->path_stage;
  const int32_t* ctx_samples = a.samples + (size_t)c * a.S * M;
  const uint32_t row_words = (M + 3) & ~3u;
  auto load_path = [&](uint32_t slot, uint32_t to) {         /* by one warp */
    const int32_t p0 = path_off[slot];
    const uint32_t len = (uint32_t)(path_off[slot + 1] - p0);
    for (uint32_t k = lane; k < len; k += 32) s_path[to][k] = path_stage[p0 + k];
    if (lane == 0) s_len[to] = len;
  };
  if (warp == 0) load_path(g, 0);
  __syncthreads();
  if (DOUBLE) copy_row<THREADS>(s_rows, ctx_samples + (size_t)s_path[0][0] * M, M);
  uint32_t pb = 0, buf = 0;
#pragma unroll 1
  for (uint32_t slot = g; slot < n_slots; slot += a.G, pb ^= 1) {
    const uint32_t len = s_len[pb];
    const bool more = slot + a.G < n_slots;
    if (more && warp == 0) load_path(slot + a.G, pb ^ 1);    /* read behind the next barrier */

    /* ---- the M samples: one recorded wait per stage of the path, picked at random ---- */
    uint32_t sum[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) sum[i] = 0;
    uint32_t seen = 0;
    const unsigned long long x0 = a.seed + 0x9E3779B97F4A7C15ull + ((unsigned long long)c * a.R + slot) * M * 64ull;
    const bool same_hi = (uint32_t)x0 <= ~0u - (THREADS * PER + 1u) * 64u;       /* uniform */
    /* nearly always the two top bits of the low words are the same too, all that the first shift takes from them: one shift
     * per stage instead of one per draw (the kernel, 4,500 slots: 435.5 -> 429.5 us) */
    const bool same_top = same_hi && ((uint32_t)x0 >> 30) == (((uint32_t)x0 + (THREADS * PER + 1u) * 64u) >> 30);
    unsigned long long x = x0 + tid * 64ull;
#pragma unroll 1
    for (uint32_t j = 0; j < len; ++j, ++x) {
      if (!DOUBLE) {
        __syncthreads();
        copy_row<THREADS>(s_rows, ctx_samples + (size_t)s_path[pb][j] * M, M);
      }
      copy_async_wait();
      __syncthreads();
      if (DOUBLE) {
        uint32_t* next = s_rows + (buf ^ 1) * row_words;
        if (j + 1 < len) copy_row<THREADS>(next, ctx_samples + (size_t)s_path[pb][j + 1] * M, M);
        else if (more) copy_row<THREADS>(next, ctx_samples + (size_t)s_path[pb ^ 1][0] * M, M);
      }
      const uint32_t* row = s_rows + (DOUBLE ? buf * row_words : 0u);
      const uint32_t lo = (uint32_t)x, hi = (uint32_t)(x >> 32);
      const unsigned long long fixed = splitmix_fixed(hi);
      const uint32_t shifted = __funnelshift_r(lo, hi, 30);
      auto draw = [&](int i) {
        const uint32_t step = (uint32_t)i * THREADS * 64u;
        if (same_hi) return row[__umulhi(splitmix_hi(lo + step, hi, fixed), M)];
        const uint32_t h = hi + (lo + step < lo ? 1u : 0u);
        return row[__umulhi(splitmix_hi(lo + step, h, splitmix_fixed(h)), M)];
      };
#pragma unroll
      for (int i0 = 0; i0 < PER; i0 += kGroup) {
        if (i0 * THREADS >= (int)M) break;                   /* uniform */
        if (same_top && (i0 + kGroup) * THREADS <= (int)M) {  /* every lane has all of the group's samples */
#pragma unroll
          for (int i = i0; i < i0 + kGroup; ++i) {
            const uint32_t v = row[__umulhi(splitmix_rest((lo + (uint32_t)i * THREADS * 64u) ^ shifted, fixed), M)];
            seen |= v;
            sum[i] += v;                                     /* < 64 * 2^24 = 2^30 when no value is bad */
          }
        } else {
#pragma unroll
          for (int i = i0; i < i0 + kGroup; ++i) {
            const uint32_t v = draw(i);
            if (tid + i * THREADS < M) seen |= v;
            sum[i] += v;
          }
        }
      }
      if (DOUBLE) buf ^= 1;
    }

    /* ---- the sum of rank a.rank ---- */
    uint32_t top = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i)
      if (tid + i * THREADS < M) top |= sum[i];
    top = __reduce_or_sync(0xffffffffu, top);
    if (lane == 0) s_warp[warp] = top;
    if (__syncthreads_or((int)(seen >> kSampleBits))) {
      if (tid == 0) atomicMax(&a.hdr->status, (uint32_t)(-PARD_EDATA));
      copy_async_wait();
      return;
    }
    for (int w = 0; w < WARPS; ++w) top |= s_warp[w];
    int hi = 32 - __clz((int)top);                           /* bits not settled yet: [0, hi) */
    uint32_t prefix = 0, left = a.rank;                      /* settled bits of the answer; its rank among the sums that share them */
    uint32_t answer = 0;
#pragma unroll 1
    for (;;) {
      const int shift = hi > (int)kSelBits ? hi - (int)kSelBits : 0;
      for (uint32_t b = tid; b < kSelBins; b += THREADS) s_hist[b] = 0;
      if (tid == 0) s_count = 0;
      __syncthreads();
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        if ((uint32_t)i * THREADS >= M) break;
        if (tid + i * THREADS < M && ((sum[i] ^ prefix) >> hi) == 0) atomicAdd(&s_hist[(sum[i] >> shift) & (kSelBins - 1)], 1u);
      }
      __syncthreads();
      /* which bin holds the rank: a thread owns kSelBins / THREADS bins in a row */
      constexpr int kOwn = kSelBins / THREADS;
      uint32_t mine = 0;
#pragma unroll
      for (int b = 0; b < kOwn; ++b) mine += s_hist[tid * kOwn + b];
      uint32_t incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= (uint32_t)o) incl += y;
      }
      if (lane == 31) s_warp[warp] = incl;
      __syncthreads();
      const uint32_t w = lane < (uint32_t)WARPS ? s_warp[lane] : 0u;
      uint32_t before = incl - mine + __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
      if (left >= before && left < before + mine) {          /* exactly one thread */
#pragma unroll
        for (int b = 0; b < kOwn; ++b) {
          const uint32_t k = s_hist[tid * kOwn + b];
          if (left >= before && left < before + k) { s_bin = tid * kOwn + b; s_left = left - before; s_count = k; }
          before += k;
        }
      }
      __syncthreads();
      const uint32_t count = s_count;
      prefix |= s_bin << shift;
      left = s_left;
      hi = shift;
      __syncthreads();
      if (hi == 0) { answer = prefix; break; }
      if (count > (uint32_t)THREADS) continue;               /* many in one bin: split it */
      /* few: list them, every one counts those before it */
      if (tid == 0) s_count = 0;
      __syncthreads();
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        if ((uint32_t)i * THREADS >= M) break;
        if (tid + i * THREADS < M && ((sum[i] ^ prefix) >> hi) == 0) s_cand[atomicAdd(&s_count, 1u)] = sum[i];
      }
      __syncthreads();
      if (tid < count) {
        const uint32_t v = s_cand[tid];
        uint32_t less = 0, same = 0;
        for (uint32_t k = 0; k < count; ++k) {
          less += s_cand[k] < v ? 1u : 0u;
          same += s_cand[k] == v ? 1u : 0u;
        }
        if (left >= less && left < less + same) s_bin = v;   /* equal values write the same */
      }
      __syncthreads();
      answer = s_bin;
      break;
    }
    if (tid == 0) a.w_out[(size_t)c * a.R + slot] = (long long)answer;
  }
}

/* Threads and samples per thread by M: the smallest block whose threads keep all sums in 20
 * registers each (more, smaller blocks hide each other's barriers); beyond 20,480 samples 32
 * registers and a single row buffer (two rows would not fit). */
struct WaitShape {
  void (*kernel)(const PipeTable, const WaitArgs);
  int threads, rows;
};
constexpr int kShapes = 5;
const WaitShape kShape[kShapes] = {{k_estimate_w<128, 20, true>, 128, 2},  {k_estimate_w<256, 20, true>, 256, 2},
                                   {k_estimate_w<512, 20, true>, 512, 2},  {k_estimate_w<1024, 20, true>, 1024, 2},
                                   {k_estimate_w<1024, 32, false>, 1024, 1}};
inline int shape_of(uint32_t M) { return M <= 2560 ? 0 : M <= 5120 ? 1 : M <= 10240 ? 2 : M <= 20480 ? 3 : 4; }

std::mutex g_attr_mutex;
int g_attr_bytes[kShapes][64];                   /* per shape and device: dynamic shared memory already allowed */

int allow_wait_smem(int dev, int shape, int bytes) {
  if (bytes <= 32 * 1024) return PARD_OK;        /* static and dynamic shared memory together stay below 48 KB */
  std::lock_guard<std::mutex> lock(g_attr_mutex);
  if (dev >= 0 && dev < 64 && g_attr_bytes[shape][dev] >= bytes) return PARD_OK;
  PARD_CUDA_OK(cudaFuncSetAttribute(kShape[shape].kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  if (dev >= 0 && dev < 64) g_attr_bytes[shape][dev] = bytes;
  return PARD_OK;
}

}  // namespace

extern "C" int pard_estimate_w_workspace_bytes(uint32_t n_pipelines, uint64_t* bytes) {
  if (!bytes || n_pipelines < 1) return PARD_EINVAL;
  *bytes = sizeof(WaitHeader) + ((8ull * n_pipelines + 255) & ~255ull);
  return PARD_OK;
}

extern "C" int pard_estimate_w(const pard_pipeline_t* const* pipelines, uint32_t n_pipelines,
                               const int32_t* d_pipeline_of_ctx, uint32_t n_ctx, int32_t stage_stride,
                               int32_t slot_stride, const int32_t* d_wait_samples, uint32_t n_samples,
                               uint32_t lambda_num, uint32_t lambda_den, uint64_t seed, uint32_t mode,
                               int64_t* d_w_us, void* d_workspace, uint64_t workspace_bytes,
                               void* cuda_stream) {
  if (!pipelines || n_pipelines < 1 || !d_wait_samples || !d_w_us || n_ctx < 1) return PARD_EINVAL;
  if (stage_stride < 1 || slot_stride < 1 || lambda_den == 0 || lambda_num > lambda_den) return PARD_EINVAL;
  if (mode & ~PARD_MODE_NOWAIT) return PARD_EINVAL;
  if (n_pipelines > 1 && !d_pipeline_of_ctx) return PARD_EINVAL;
  if (n_pipelines > 65536) return PARD_ERANGE;
  if (stage_stride > PARD_MAX_STAGES || slot_stride > PARD_MAX_PATH_SLOTS ||
      (uint64_t)n_ctx * (uint64_t)stage_stride > PARD_MAX_SEGMENTS ||
      (uint64_t)n_ctx * (uint64_t)slot_stride >= (1ull << 31) || n_samples < 1 ||
      n_samples > PARD_MAX_WAIT_SAMPLES)
    return PARD_ERANGE;
  int dev = -1;
  PARD_CUDA_OK(cudaGetDevice(&dev));
  for (uint32_t i = 0; i < n_pipelines; ++i) {
    const pard_pipeline_t* p = pipelines[i];
    if (!p || !p->d_blob || p->device != dev) return PARD_EINVAL;
    if (p->n_stages > stage_stride || p->n_slots > slot_stride) return PARD_EINVAL;
  }
  if (!d_workspace || ((uintptr_t)d_workspace & 255)) return PARD_EINVAL;
  uint64_t need = 0;
  pard_estimate_w_workspace_bytes(n_pipelines, &need);
  if (workspace_bytes < need) return PARD_EWORKSPACE;

  cudaStream_t stream = (cudaStream_t)cuda_stream;
  WaitHeader* hdr = (WaitHeader*)d_workspace;
  const int shape = shape_of(n_samples);
  const int smem = (int)(4u * ((n_samples + 3) & ~3u)) * kShape[shape].rows;
  int rc = allow_wait_smem(dev, shape, smem);
  if (rc != PARD_OK) return rc;
  PipeTable table;
  rc = pard_pipe_table(pipelines, n_pipelines, (char*)d_workspace + sizeof(WaitHeader), stream, &table);
  if (rc != PARD_OK) return rc;
  PARD_CUDA_OK(pard_clear_status(hdr, stream));
  WaitArgs a = {};
  a.n_pipelines = n_pipelines; a.pipeline_of_ctx = d_pipeline_of_ctx;
  a.S = (uint32_t)stage_stride; a.R = (uint32_t)slot_stride; a.M = n_samples;
  a.samples = d_wait_samples; a.seed = (unsigned long long)seed; a.w_out = (long long*)d_w_us; a.hdr = hdr;
  const uint64_t rank = (uint64_t)lambda_num * n_samples / lambda_den;
  a.rank = (uint32_t)std::min<uint64_t>(rank, n_samples - 1);
  /* blocks per ctx: about thirty rounds of resident blocks in all, so that uneven paths even out;
   * with few contexts a block per slot */
  int sms = 148;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint64_t blocks = 32ull * (uint64_t)sms * (1024 / kShape[shape].threads);
  a.G = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)slot_stride, (blocks + n_ctx - 1) / n_ctx));
  PARD_CUDA_OK(launch_pdl(kShape[shape].kernel, n_ctx * a.G, kShape[shape].threads, (size_t)smem, stream, table, a));
  if (mode & PARD_MODE_NOWAIT) return PARD_OK;
  return pard_wait_status(&hdr->status, stream);
}
