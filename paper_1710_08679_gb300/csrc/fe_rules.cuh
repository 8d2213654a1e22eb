// Rules that choose a kernel or a launch shape by the size of a call. Plain host code
// without CUDA types; the times beside each rule were measured on one GB300 (152 SMs).
#pragma once

#include <stdint.h>

namespace fe {

// Inner-loop vector passes with four cases per thread: from 140 such threads per SM on.
// With fewer the SMs are filled better by a thread per case. Step of the inner loop at level
// 0 with one / four cases per thread: 1,331 nodes, R = 4: 24.0 / 26.1 us, R = 64: 29.7 / 29.0;
// 4,913 nodes, R = 16: 28.6 / 29.1, R = 20: 33.9 / 31.5; 9,261 nodes, R = 8: 28.6 / 29.1,
// R = 12: 32.5 / 31.9.
inline bool four_case_passes(int64_t n_nodes, int R, int sms) {
  return R % 4 == 0 && n_nodes * R >= 560 * (int64_t)sms;
}

}  // namespace fe
