// Which way a size class of a batched solve goes: the time that the single-problem path
// takes for one iteration of each of its problems, to be compared with a sigma round of
// the class launch (one CTA per problem).
//
// Up to BATCH_WORKERS problems are in flight on the single-problem path, and they share the
// GPU and the driver: with w of them a problem takes 0.35 + 0.65 / w of its time alone.
// Measured on one GB300, batches of one class with every problem on that path, 6 to 10
// orbitals, FP64 and BF16x2: 3 problems 0.43 - 0.72 each (mean 0.59), 8 problems 0.27 - 0.46
// (0.40), 24 and 96 problems 0.24 - 0.47 (0.39).
//
// A mixed solve takes fewer and longer iterations than an FP64 one, and the CTAs' rounds
// are those of an FP64 one: its time per FP64 iteration was 0.63 - 0.88 (mean 0.72) of an
// iteration on FP32 vectors at 6 to 10 orbitals, one and two roots.
#pragma once

#include <algorithm>

namespace forte {

constexpr int BATCH_WORKERS = 8;

// iter_ms: one iteration of one problem on its own; nroots: the sigma builds in it.
inline double single_path_ms(double iter_ms, int nroots, bool mixed, int problems) {
  const int w = std::max(1, std::min(problems, BATCH_WORKERS));
  return iter_ms / nroots * (mixed ? 0.72 : 1.0) * (0.35 + 0.65 / w);
}

}  // namespace forte
