// Scratch memory of the single-call entries (sweep adjoint, deposit, gravity, spectra, noise
// refinement): stream-ordered allocations from a pool of this library, one per device.
//
// The device's default pool returns its memory to the system at every synchronisation of the
// host, so a caller that waits for each result paid for mapping and unmapping the scratch on
// every call: three adjoint sweeps at 96^3 with a wait after them 594 -> 184 us (137-150 us
// among other work), deposit + gravity + force at 128^3 591 -> 284 us, the spectra at 128^3
// 664 -> 186 us. This pool keeps up to kKeep bytes mapped. Its allocations are ordered on the
// caller's stream as before, so several threads and streams share it safely. The bound holds from
// the next host synchronisation on (that is when CUDA applies a pool's threshold). What the pool
// keeps is given back by sim_scratch_trim, when a handle is destroyed, before cuFFT plans are
// made, and when an allocation of this library fails. 512 MB is 0.2 % of the device and holds the largest scratch up to 188^3
// (20 n^3 floats, the x sweep's adjoint): above that the kernels take milliseconds and the
// mapping matters less.
#include <atomic>
#include <mutex>

#include "common.cuh"

namespace dh {

namespace {

constexpr unsigned long long kKeep = 512ull << 20;
constexpr int kMaxDev = 64;
std::mutex g_mu;
std::atomic<cudaMemPool_t> g_pool[kMaxDev];
bool g_tried[kMaxDev];

// Pool management is not stream work: allow it while another thread captures a graph.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// The current device's pool; null if there is none and (make false, or it cannot be made).
cudaMemPool_t pool_of_device(bool make) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
    cudaGetLastError();
    return nullptr;
  }
  if (cudaMemPool_t p = g_pool[dev].load(std::memory_order_acquire)) return p;
  if (!make) return nullptr;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_tried[dev]) {
    g_tried[dev] = true;
    RelaxedCapture relaxed;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    unsigned long long keep = kKeep;
    if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
      cudaGetLastError();
    } else if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
      cudaGetLastError();
      cudaMemPoolDestroy(p);
    } else {
      g_pool[dev].store(p, std::memory_order_release);
    }
  }
  return g_pool[dev].load(std::memory_order_acquire);
}

}  // namespace

cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t st) {
  // under capture the allocation belongs to the graph, as before
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  const bool plain = cudaStreamIsCapturing(st, &cs) != cudaSuccess;
  if (plain) cudaGetLastError();
  if (!plain && cs == cudaStreamCaptureStatusNone) {
    if (cudaMemPool_t pool = pool_of_device(true)) {
      if (cudaMallocFromPoolAsync(p, bytes, pool, st) == cudaSuccess) return cudaSuccess;
      cudaGetLastError();
      scratch_trim();
    }
  }
  return cudaMallocAsync(p, bytes, st);
}

void scratch_trim() {
  if (cudaMemPool_t pool = pool_of_device(false)) {
    RelaxedCapture relaxed;
    if (cudaMemPoolTrimTo(pool, 0) != cudaSuccess) cudaGetLastError();
  }
}

}  // namespace dh

extern "C" void sim_scratch_trim(void) { dh::scratch_trim(); }
