// Device scratch of the stand-alone entry points (those that take no context).
//
// A call's launches write and read scratch on the caller's stream, so scratch belongs to a
// stream: two calls on one stream are ordered, two on different streams run together. Up to
// 16 streams of a device keep a buffer of each kind for the life of the process (64 MB of
// split-K sums; 78 MB for GroupNorm); streams beyond these, and every captured call, take
// stream-ordered memory for the call alone, which in a capture belongs to the graph: replays
// of two graphs share nothing. Two host threads on one stream take turns, a call at a time,
// for their launches would mix otherwise.
#pragma once

#include <mutex>

#include "common.cuh"

namespace ddppo {

constexpr size_t kSplitkElems = (size_t)16 << 20;  // floats of split-K sums
int device_sms(int* sms);                          // SMs of the current device

enum ScratchKind { SCRATCH_SPLITK = 0, SCRATCH_GN, SCRATCH_GCONV, SCRATCH_AMAX, SCRATCH_KINDS };

class Scratch {
 public:
  Scratch() = default;
  Scratch(const Scratch&) = delete;
  Scratch& operator=(const Scratch&) = delete;
  ~Scratch();
  // `bytes` (the same for every call of a kind) for this call's launches on s, held until the
  // object goes; the last `zeroed` of them are zero when the memory is new. One kind an object.
  int take(ScratchKind kind, size_t bytes, size_t zeroed, cudaStream_t s);
  template <typename T>
  T* as(size_t offset = 0) const { return reinterpret_cast<T*>((char*)p_ + offset); }

 private:
  void* p_ = nullptr;
  bool owned_ = false;  // stream-ordered memory of this call alone
  cudaStream_t s_ = nullptr;
  std::unique_lock<std::mutex> turn_;
};

}  // namespace ddppo
