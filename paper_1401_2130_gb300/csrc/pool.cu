// pool.cu -- device scratch and pinned staging kept between calls.
//
// Device scratch comes from one memory pool per device, apart from the
// process's default pool (whose settings are the application's).  A pool with
// the default release threshold gives its memory back to the system at every
// synchronisation, and mapping it again cost a call of host outputs 0.2 to 1.5
// ms (W = 4, L = 16, 1,000 configurations: 327 us alone, against 64 us among
// others that are not waited for).  This pool keeps at most kKeep bytes.
// Allocation and free stay stream-ordered, so threads and streams share it
// safely.
//
// Outputs for the host come back in one copy to a pinned buffer: each of the
// six pageable copies it replaces waits for the stream on its own.  At most
// kBuffers buffers of kStageBytes are kept; more concurrent calls allocate and
// free their own.
//
// Executable graphs are destroyed many at a time: cudaGraphExecDestroy waits
// until the device is idle, also for a graph that has ended (290 ms behind a
// kernel of 290 ms), and would make an asynchronous call wait for its stream.
// At most kRetired are kept; every kRetired-th call waits.
//
// Mails (take_mail) are kMails words of pinned memory.
//
// pc_shutdown gives everything back.
#include <map>
#include <mutex>
#include <new>
#include <vector>

#include "pool.cuh"

namespace pc {

namespace {

constexpr uint64_t kKeep = 1ull << 30;
constexpr size_t kStageBytes = 4u << 20;
constexpr size_t kBuffers = 8;

std::mutex g_mu;
std::map<int, cudaMemPool_t> g_pools;
char* g_stage[kBuffers];
size_t g_stages = 0;

constexpr unsigned kMails = 4096;
unsigned long long* g_mail = nullptr;
unsigned g_tag = 0;

constexpr size_t kRetired = 64;
struct Retired { cudaGraphExec_t ex; cudaEvent_t ev; };
Retired g_retired[kRetired];
size_t g_retireds = 0;

}  // namespace

cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t st) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  cudaMemPool_t pool = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_pools.find(dev);
    if (it == g_pools.end()) {
      cudaMemPoolProps props = {};
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      if ((e = cudaMemPoolCreate(&pool, &props)) != cudaSuccess) return e;
      uint64_t keep = kKeep;
      e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
      // memory freed on another stream is reused only once that stream has
      // passed the free: no stream is made to wait for another
      int no = 0;
      if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &no);
      if (e != cudaSuccess) { cudaMemPoolDestroy(pool); return e; }
      try {
        it = g_pools.emplace(dev, pool).first;
      } catch (const std::bad_alloc&) {
        cudaMemPoolDestroy(pool);
        return cudaErrorMemoryAllocation;
      }
    }
    pool = it->second;
  }
  return cudaMallocFromPoolAsync(p, bytes, pool, st);
}

HostStage::HostStage(size_t bytes) {
  if (bytes > kStageBytes) return;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (g_stages > 0) {
      p_ = g_stage[--g_stages];
      return;
    }
  }
  if (cudaMallocHost((void**)&p_, kStageBytes) != cudaSuccess) {
    cudaGetLastError();
    p_ = nullptr;
  }
}

HostStage::~HostStage() {
  if (!p_) return;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (g_stages < kBuffers) {
      g_stage[g_stages++] = p_;
      return;
    }
  }
  cudaFreeHost(p_);
}

bool Mail::answer(unsigned* v) const {
  if (!at) return false;
  const unsigned long long x = *(const volatile unsigned long long*)at;
  *v = (unsigned)x;
  return (unsigned)(x >> 32) == tag;
}

Mail take_mail() {
  Mail m;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_mail) {
    void* p = nullptr;
    if (cudaHostAlloc(&p, kMails * sizeof(unsigned long long), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
      cudaGetLastError();
      return m;
    }
    g_mail = (unsigned long long*)p;
    for (size_t i = 0; i < kMails; ++i) g_mail[i] = 0ull;
  }
  if (++g_tag == 0u) ++g_tag;
  m.tag = g_tag;
  m.at = g_mail + g_tag % kMails;
  return m;
}

void retire_graph(cudaGraphExec_t ex, cudaStream_t st) {
  cudaEvent_t ev = nullptr;
  if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess || cudaEventRecord(ev, st) != cudaSuccess) {
    cudaGetLastError();
    if (ev) cudaEventDestroy(ev);
    cudaGraphExecDestroy(ex);
    return;
  }
  Retired done[kRetired];
  size_t n = 0;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (g_retireds == kRetired) {
      size_t left = 0;
      for (size_t i = 0; i < kRetired; ++i) {
        if (i == 0 || cudaEventQuery(g_retired[i].ev) == cudaSuccess) done[n++] = g_retired[i];
        else g_retired[left++] = g_retired[i];
      }
      cudaGetLastError();  // "not ready"
      g_retireds = left;
    }
    g_retired[g_retireds++] = Retired{ex, ev};
  }
  for (size_t i = 0; i < n; ++i) {
    cudaGraphExecDestroy(done[i].ex);
    cudaEventDestroy(done[i].ev);
  }
}

void release_pools() {
  std::lock_guard<std::mutex> lk(g_mu);
  for (size_t i = 0; i < g_retireds; ++i) {
    cudaGraphExecDestroy(g_retired[i].ex);
    cudaEventDestroy(g_retired[i].ev);
  }
  g_retireds = 0;
  std::vector<int> devices;
  for (const auto& kv : g_pools) devices.push_back(kv.first);
  for (auto& kv : g_pools) cudaMemPoolDestroy(kv.second);
  g_pools.clear();
  while (g_stages > 0) cudaFreeHost(g_stage[--g_stages]);
  if (g_mail) {  // no kernel may still write into it
    int now = 0;
    cudaGetDevice(&now);
    for (int dev : devices) {
      cudaSetDevice(dev);
      cudaDeviceSynchronize();
    }
    cudaSetDevice(now);
    cudaFreeHost(g_mail);
  }
  g_mail = nullptr;
  cudaGetLastError();  // after cudaDeviceReset the handles are gone already
}

}  // namespace pc
