/* How a waiting call learns its status.
 *
 * Copying the status word to the host and synchronising the stream costs 12.5 us for a call whose
 * kernels take 25: a copy into pageable memory is staged and waited for on its own.  Instead the
 * device writes the word straight into pinned host memory -- the last kernel of the call, or a
 * kernel of one thread behind it -- and the host polls it: 4 to 5 us from the end of the last
 * kernel.  The words come from one page, allocated when the first pipeline is loaded: a thread
 * takes one of 64 on its first waiting call and gives it back when it ends; a thread that finds
 * none takes the copy.  A word carries the ticket of the call it answers, so that a late answer
 * to an abandoned call is never taken for the next one's. */
#include <atomic>
#include <mutex>

#include "pard_internal.h"

namespace {

constexpr int kSlots = 64;
struct alignas(64) Slot {
  unsigned long long word;                       /* ticket << 32 | status */
  unsigned long long count;                      /* a number that goes with it */
  unsigned long long pad[6];
};
std::mutex g_mu;
std::atomic<Slot*> g_page{nullptr};
std::atomic<char*> g_staging{nullptr};           /* kStagingBytes for each of the first kStagingSlots slots */
constexpr int kStagingSlots = 8;
std::atomic<uint64_t> g_taken{0};
uint32_t g_ticket[kSlots];                       /* of the slot's owner */

struct Owned {
  int slot = -1;
  ~Owned() {
    if (slot >= 0) g_taken.fetch_and(~(1ull << slot), std::memory_order_release);
  }
};
thread_local Owned t_owned;

int own_slot() {
  if (t_owned.slot >= 0 || !g_page.load(std::memory_order_acquire)) return t_owned.slot;
  uint64_t taken = g_taken.load(std::memory_order_relaxed);
  while (~taken) {
    const int k = __builtin_ctzll(~taken);
    if (g_taken.compare_exchange_weak(taken, taken | (1ull << k), std::memory_order_acquire)) return t_owned.slot = k;
  }
  return -1;
}

__global__ void k_report(const uint32_t* status, unsigned long long* word, uint32_t ticket, const unsigned long long* count) {
  pdl_wait();
  if (count) word[1] = __ldcg(count);
  pard_report(status, word, ticket);
}

__global__ void k_clear_status(uint32_t* hdr) {
  pdl_wait();
  hdr[threadIdx.x] = 0;
}

}  // namespace

cudaError_t pard_clear_status(void* hdr, cudaStream_t stream) {
  return launch_pdl(k_clear_status, 1, 64, 0, stream, (uint32_t*)hdr);
}

void pard_report_init() {
  if (g_page.load(std::memory_order_acquire)) return;
  std::lock_guard<std::mutex> lock(g_mu);
  if (g_page.load(std::memory_order_relaxed)) return;
  void* p = nullptr;
  if (cudaHostAlloc(&p, sizeof(Slot) * kSlots, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
    cudaGetLastError();                          /* the calls copy their status then */
    return;
  }
  for (int i = 0; i < kSlots; ++i) ((Slot*)p)[i].word = 0;
  void* s = nullptr;
  if (cudaHostAlloc(&s, (size_t)kStagingSlots * kStagingBytes, cudaHostAllocPortable) == cudaSuccess)
    g_staging.store((char*)s, std::memory_order_release);
  else
    cudaGetLastError();
  g_page.store((Slot*)p, std::memory_order_release);
}

PardTicket pard_report_ticket() {
  PardTicket t = {nullptr, 0};
  const int k = own_slot();
  if (k < 0) return t;
  t.word = &g_page.load(std::memory_order_acquire)[k].word;
  t.ticket = ++g_ticket[k] ? g_ticket[k] : ++g_ticket[k];      /* 0 is the page's initial value */
  return t;
}

int pard_report_wait(const PardTicket& t, const uint32_t* d_status, cudaStream_t stream, bool* answered) {
  if (answered) *answered = false;
  if (t.word) {
    for (uint32_t spins = 1;; ++spins) {
      const unsigned long long w = __atomic_load_n(t.word, __ATOMIC_ACQUIRE);
      if ((uint32_t)(w >> 32) == t.ticket) {
        if (answered) *answered = true;
        return (uint32_t)w ? -(int)(uint32_t)w : PARD_OK;
      }
#if defined(__x86_64__)
      __builtin_ia32_pause();
#endif
      if ((spins & 4095) == 0) {                 /* a stream that failed will not answer */
        const cudaError_t e = cudaStreamQuery(stream);
        if (e == cudaErrorNotReady) continue;
        if (e != cudaSuccess) return PARD_ECUDA;
        if ((uint32_t)(__atomic_load_n(t.word, __ATOMIC_ACQUIRE) >> 32) != t.ticket) break;
      }
    }
  }
  uint32_t h_status = 0;
  PARD_CUDA_OK(cudaMemcpyAsync(&h_status, d_status, 4, cudaMemcpyDeviceToHost, stream));
  PARD_CUDA_OK(cudaStreamSynchronize(stream));
  return h_status ? -(int)h_status : PARD_OK;
}

int pard_report_enqueue(const PardTicket& t, const uint32_t* d_status, const unsigned long long* d_count, cudaStream_t stream) {
  if (t.word) PARD_CUDA_OK(launch_pdl(k_report, 1, 1, 0, stream, d_status, t.word, t.ticket, d_count));
  return PARD_OK;
}

int pard_wait_status(const uint32_t* d_status, cudaStream_t stream) {
  const PardTicket t = pard_report_ticket();
  const int rc = pard_report_enqueue(t, d_status, nullptr, stream);
  return rc != PARD_OK ? rc : pard_report_wait(t, d_status, stream, nullptr);
}

char* pard_staging() {
  const int k = own_slot();
  char* s = g_staging.load(std::memory_order_acquire);
  return k >= 0 && k < kStagingSlots && s ? s + (size_t)k * kStagingBytes : nullptr;
}
