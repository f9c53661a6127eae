// The step exchange of the LSTM cluster kernels (lstm_cluster.cu) as plain host C++, so that a
// host compiler alone can check the drain after an abort.
//
// Step s (1 <= s < T) is read from buffer s & 1, whose barrier completes one phase for every
// second step: steps 1, 3, 5, ... of one barrier are its phases 0, 1, 2, ..., steps 2, 4, 6, ...
// of the other. Every CTA of the cluster sends a block of step s + 1 to every CTA once it has
// received all of step s, so the last steps that two CTAs have sent differ by at most one.
#pragma once

namespace ddppo {

constexpr int step_bar(int s) { return s & 1; }
constexpr unsigned step_parity(int s) { return (unsigned)((s - 1) >> 1) & 1u; }

// sent[j]: the last step that CTA j sent. The CTAs whose block of step s never comes, or -1
// where there is nothing to wait for: no such step, or no CTA has sent it.
constexpr int step_missing(const int* sent, int ctas, int s, int T) {
  if (s < 1 || s >= T) return -1;
  int missing = 0;
  for (int j = 0; j < ctas; ++j) missing += sent[j] < s ? 1 : 0;
  return missing == ctas ? -1 : missing;
}

}  // namespace ddppo
