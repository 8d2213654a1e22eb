// Rules that choose a kernel or a launch shape by the size of a call. Plain host code
// without CUDA types; the times beside each rule were measured on one GB300 (152 SMs).
#pragma once

#include <stdint.h>

#include <algorithm>
#include <cmath>

namespace fe {

// FP32 direct product: two cases per thread (paired instructions) or one. Two halve the
// geometry and the arithmetic's instructions, at 168 registers a thread instead of 128: worth it
// on large meshes; on small ones, where a product is one or two rounds of warps, only for few
// cases. us in a graph with one / two: 3,072 elements, R = 4: 6.7 / 6.7, R = 24: 10.2 / 11.2;
// 7,986, R = 6: 9.6 / 9.1, R = 16: 13.5 / 15.5; 16,464, R = 8: 14.3 / 15.4, R = 32: 39.3 / 40.3;
// 31,104, R = 6: 22.4 / 20.9, R = 32: 67.8 / 67.0; 146,124, R = 32: 336 / 315.
inline bool direct_two_cases(int64_t n_elem, int R) { return R % 2 == 0 && (R <= 6 || n_elem >= 24000); }

// Rounds that `warps` warps of equal length take on the 4 * sms SM sub-partitions, each of
// which runs its warps through its FP64 unit one instruction after the other: the number on
// the fullest one. (Fewer warps than sub-partitions do not go one to each: some share one.)
inline double f64_rounds(int64_t warps, int sms) {
  const double n = (double)warps / (4.0 * sms);
  return n > 1.0 ? std::ceil(n) : 1.0 + 0.4 * std::max(0.0, n - 0.3);
}

// Lanes an element's R cases are spread over in the FP64 kernels whose threads loop over
// cases: `per_case` FP64 instructions' time for each case and `geometry` for the element. More
// lanes fill the sub-partitions evenly, fewer compute the geometry less often. `pow2`: the
// lanes' sums meet by shuffles, so their number is a power of two of at most 32.
inline int f64_case_split(int64_t n_elem, int R, int per_case, int geometry, int sms, bool pow2,
                          double* cost_out = nullptr) {
  int best = 1;
  double best_cost = 1e300;
  for (int k = R; k >= 1; --k) {   // cases per lane
    int split = (R + k - 1) / k;
    while (pow2 && (split & (split - 1)) != 0) ++split;
    if (pow2 && split > 32) continue;
    const double cost = f64_rounds((n_elem * split + 31) / 32, sms) * (k * per_case + geometry);
    if (cost < best_cost) {
      best_cost = cost;
      best = split;
    }
  }
  if (cost_out) *cost_out = best_cost;
  return best;
}

// FP64 direct product: lanes per element, 0 for the kernel with a lane per corner of every
// (element, case). The times of a case (480: 440 instructions and the waits on its loads),
// the geometry (70) and a corner (190) were fitted to 9 meshes of 750 to 146,124 elements, R = 1
// to 64, every split, launched behind the zero pass and in graphs: the choice takes 0.3 and
// 0.8 % longer than the fastest split on average. us in a graph with 1 / 2 / 4 / R lanes / corners:
// 3,072 elements, R = 12: 207 / 110 / 57 / 42 / 53; 16,464, R = 9: 172 / 155 / - / 152 / 192.
inline int f64_direct_split(int64_t n_elem, int R, int sms) {
  double cost = 0.0;
  const int split = f64_case_split(n_elem, R, 480, 70, sms, false, &cost);
  return f64_rounds((4 * n_elem * R + 31) / 32, sms) * 190 < cost ? 0 : split;
}

// Sensitivities: lanes per element (475 instructions a case; the choice takes 0.3 % longer
// than the fastest split on average over the same meshes and R).
inline int f64_adjoint_split(int64_t n_elem, int R, int sms) {
  return f64_case_split(n_elem, R, 500, 110, sms, true);
}

// Level-1 product from the sliced matrix: two blocks of a row in flight (64 registers, 1,024
// threads per SM) or one (48 registers, 1,280). Two cover more latency, one fits a few more
// threads: it is the faster one where it takes a round of threads less. us in a graph with
// one / two by w, the rounds of threads with two: w = 0.56 8.3 / 7.7; w = 1.17 25.0 / 28.6;
// w = 1.26 13.7 / 14.8; w = 1.36 16.4 / 16.2; w = 2.33 34.9 / 35.9; w = 2.44 21.8 / 23.3;
// w = 2.71 25.7 / 25.2; w = 4.66 56.1 / 52.8; w = 9.33 98.1 / 90.5.
inline bool level1_two_blocks(int64_t n_nodes, int R, int sms) {
  const double w = (double)(n_nodes * (R / 4)) / (1024.0 * sms);
  return !((w > 1.0 && w <= 1.3) || (w > 2.0 && w <= 2.5));
}

// Inner-loop vector passes with four cases per thread: from 140 such threads per SM on.
// With fewer the SMs are filled better by a thread per case. Step of the inner loop at level
// 0 with one / four cases per thread: 1,331 nodes, R = 4: 24.0 / 26.1 us, R = 64: 29.7 / 29.0;
// 4,913 nodes, R = 16: 28.6 / 29.1, R = 20: 33.9 / 31.5; 9,261 nodes, R = 8: 28.6 / 29.1,
// R = 12: 32.5 / 31.9.
inline bool four_case_passes(int64_t n_nodes, int R, int sms) {
  return R % 4 == 0 && n_nodes * R >= 560 * (int64_t)sms;
}

}  // namespace fe
