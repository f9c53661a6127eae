// Scratch of the stand-alone entry points: one buffer of a kind per device and stream, looked
// up by the stream's id (which, unlike its handle, is never used again). A look-up is on the
// path of calls of 10 us, bound by the host, and is made by the launches that need scratch
// alone: 0.1 us (capture state and id 33 ns each, the turn's lock 18); with a lock around the
// table and a look-up in every call the host took 0.2 to 0.5 us more a call.
#include "scratch.cuh"

#include <atomic>

#include "gemm.cuh"

namespace ddppo {

namespace {

constexpr int kStreams = 16, kDevices = 64;

struct Slot {
  std::atomic<unsigned long long> key{0};  // stream id + 1; 0: free
  std::mutex turn;
  void* buf[SCRATCH_KINDS] = {};
};
Slot g_slots[kDevices][kStreams];

// the stream's slot, a free one for a new stream, or null when there is none left
Slot* slot_of(int dev, unsigned long long id) {
  const unsigned long long key = id + 1;
  for (Slot& s : g_slots[dev]) {
    unsigned long long k = s.key.load(std::memory_order_acquire);
    if (k == key || (k == 0 && (s.key.compare_exchange_strong(k, key) || k == key))) return &s;
  }
  return nullptr;
}

bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  return st == cudaStreamCaptureStatusActive;
}

}  // namespace

Scratch::~Scratch() {
  if (owned_) (void)cudaFreeAsync(p_, s_);
}

int Scratch::take(ScratchKind kind, size_t bytes, size_t zeroed, cudaStream_t s) {
  int dev = 0;
  DDPPO_CHECK_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kDevices) {
    set_error("scratch: device ordinal out of range");
    return DDPPO_E_ARG;
  }
  if (p_) return DDPPO_OK;  // a second launch of the same call
  s_ = s;
  Slot* slot = nullptr;
  if (!capturing(s)) {
    unsigned long long id = 0;
    DDPPO_CHECK_CUDA(cudaStreamGetId(s, &id));
    slot = slot_of(dev, id);
  }
  if (slot) {
    turn_ = std::unique_lock<std::mutex>(slot->turn);
    p_ = slot->buf[kind];
    if (p_) return DDPPO_OK;
    DDPPO_CHECK_CUDA(cudaMalloc(&p_, bytes));
  } else {
    DDPPO_CHECK_CUDA(cudaMallocAsync(&p_, bytes, s));
    owned_ = true;
  }
  if (zeroed) {
    const cudaError_t e = cudaMemsetAsync((char*)p_ + bytes - zeroed, 0, zeroed, s);
    if (e != cudaSuccess && slot) (void)cudaFree(p_);
    DDPPO_CHECK_CUDA(e);
  }
  if (slot) slot->buf[kind] = p_;
  return DDPPO_OK;
}

int device_sms(int* sms) {
  static std::atomic<int> cache[kDevices];  // 0: not asked yet
  int dev = 0;
  DDPPO_CHECK_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kDevices) {
    set_error("device ordinal out of range");
    return DDPPO_E_ARG;
  }
  int n = cache[dev].load(std::memory_order_relaxed);
  if (!n) {
    DDPPO_CHECK_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
    cache[dev].store(n, std::memory_order_relaxed);
  }
  *sms = n;
  return DDPPO_OK;
}

int GemmWorkspace::sums(cudaStream_t s, float** p) const {
  if (!partial && scratch) {
    DDPPO_TRY(scratch->take(SCRATCH_SPLITK, kSplitkElems * sizeof(float), 0, s));
    *p = scratch->as<float>();
  } else {
    *p = partial;
  }
  return DDPPO_OK;
}

}  // namespace ddppo
