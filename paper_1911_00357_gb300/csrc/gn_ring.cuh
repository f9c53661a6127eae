// Geometry of the GroupNorm backward's shared-memory ring (gn.cu), as plain host C++: which
// sizes its bulk copies cover. No CUDA header, so that a host compiler alone can check the
// rule over every size a network may have.
#pragma once

#include <cstddef>

namespace ddppo {

constexpr int kGnThreads = 256;  // consumer threads; 4 channels a thread
constexpr int kRingRows = 2;     // pixel rows a thread takes from one unit

// pixel rows the block covers in one pass at V channels a thread
constexpr int gn_rows_per_pass(int C, int V) { return C / V >= kGnThreads ? 1 : kGnThreads / (C / V); }
// pixels of one unit (an image's last unit holds what is left)
constexpr int ring_rows(int C) { return kRingRows * gn_rows_per_pass(C, 4); }

// A mask byte covers 4 channels, so a unit brings ring_rows C / 4 of them, an image HW C / 4,
// and unit u starts u ring_rows C / 4 bytes into its image. cp.async.bulk moves multiples of
// 16 bytes from 16-byte boundaries: both counts must be multiples of 16. (z and dy take 16
// bytes a thread and row, whatever C % 4 == 0.)
constexpr bool ring_mask_copies_ok(int HW, int C) {
  return (long long)HW * C % 64 == 0 && (long long)ring_rows(C) * C % 64 == 0;
}

}  // namespace ddppo
