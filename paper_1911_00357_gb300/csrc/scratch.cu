// Scratch of the stand-alone entry points: one buffer of a kind per device and stream, looked
// up by the stream's id (which, unlike its handle, is never used again). Measured cost of a
// look-up: below the noise of a call (the smallest, 10 us, host-bound).
#include "scratch.cuh"

namespace ddppo {

namespace {

constexpr int kStreams = 16, kDevices = 64;

struct Slot {
  std::mutex turn;
  bool used = false;
  unsigned long long id = 0;
  void* buf[SCRATCH_KINDS] = {};
};
Slot g_slots[kDevices][kStreams];
std::mutex g_table;  // slots' used and id

// the stream's slot, a free one for a new stream, or null when there is none left
Slot* slot_of(int dev, unsigned long long id) {
  std::lock_guard<std::mutex> lock(g_table);
  for (Slot& s : g_slots[dev]) {
    if (s.used && s.id != id) continue;
    s.used = true;
    s.id = id;
    return &s;
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

}  // namespace ddppo
