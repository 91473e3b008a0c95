// Device memory of calls that need a workspace only while they run (pw_heev,
// pw_zgemm_f64tc, their fixed forms, pw_zgemm_tc): a
// stream-ordered pool of the library's own per device.  Allocating and freeing
// them with cudaMalloc / cudaFree mapped and unmapped gigabytes on every call: 1.6
// of the 4.8 ms of a 1,458 x 1,458 x 43,819 split-FP16 product, 0.4 of the 1.3 ms
// of an order-54 eigensolve.
//
// The pool keeps at most PW_POOL_KEEP bytes between calls.  The driver gives back
// what is above that at a synchronisation, and a trim only what the host has seen
// released, so a call releases its workspaces before its last wait (pw_finish),
// never after it (after it, 9.8 GB of operands stayed on).  All of it goes back
// when an allocation of the library fails, when a serving run starts and on
// pw_release_memory (another allocator of the process cannot ask for it).  The
// driver orders the reuse of a block by another stream after its release, so
// concurrent calls on any streams and threads share it.
#include <mutex>

#include "pw_internal.cuh"

namespace {
constexpr uint64_t PW_POOL_KEEP = 2ull << 30;
constexpr int MAXDEV = 64;
std::mutex g_mu;
cudaMemPool_t g_pool[MAXDEV];
bool g_tried[MAXDEV];

// the current device's pool (nullptr if it cannot have one); created on first use
cudaMemPool_t pool(bool create) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAXDEV) return nullptr;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_tried[dev] && create) {
    g_tried[dev] = true;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    uint64_t keep = PW_POOL_KEEP;
    if (cudaMemPoolCreate(&p, &props) == cudaSuccess &&
        cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess)
      g_pool[dev] = p;
    else
      cudaGetLastError();
  }
  return g_pool[dev];
}
}  // namespace

void pw_pool_trim() {
  if (cudaMemPool_t p = pool(false))
    if (cudaMemPoolTrimTo(p, 0) != cudaSuccess) cudaGetLastError();
}

extern "C" pw_status pw_release_memory(void) {
  int dev = 0;
  PW_CUDA(cudaGetDevice(&dev));
  pw_pool_trim();
  return PW_OK;
}

cudaError_t pw_mem_alloc(const pw_mem &m, void **p, size_t bytes) {
  *p = nullptr;
  cudaMemPool_t pl = m.pooled ? pool(true) : nullptr;
  cudaError_t e = pl ? cudaMallocFromPoolAsync(p, bytes, pl, m.st) : cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    pw_pool_trim();
    e = pl ? cudaMallocFromPoolAsync(p, bytes, pl, m.st) : cudaMalloc(p, bytes);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
  }
  return e;
}

void pw_mem_free(const pw_mem &m, void *p) {
  if (!p) return;
  if (m.pooled && pool(false)) cudaFreeAsync(p, m.st);
  else cudaFree(p);
}

// A pinned word of the calling thread's, whose calls wait for what they copy into
// it: a copy to pageable memory would wait by itself, before the workspaces are
// released, and a call would wait twice (5 to 12 us more).
int *pw_host_word() {
  struct Word {
    int *p = nullptr;
    Word() {
      if (cudaHostAlloc((void **)&p, sizeof(int), cudaHostAllocPortable) != cudaSuccess) {
        cudaGetLastError();
        p = nullptr;
      }
    }
    ~Word() {
      if (p) cudaFreeHost(p);
    }
  };
  thread_local Word w;
  return w.p;
}
