// Host rules that choose a GEMM's tiles, free of CUDA so that they can be
// checked without a device.
#pragma once
#include <cstdint>

namespace tadm {

// GLU GEMMs of CTA pairs: true for 192-wide tiles (96 gate and 96 up columns),
// false for 256-wide ones.  units: pair tiles of each width; clusters: how many
// clusters of each kernel are resident at once, which is also the launch's
// grid, so units / clusters are its rounds.  192 where its rounds take at most
// 0.85 of the 256-wide tiles' (a narrower tile re-reads the activations more
// often): the 256 x 2 x 21504 projection of a 27 B block step is 168 tiles on
// 76 clusters, whose third round is 16 tiles, or 224 in 2.95 rounds (the step
// of three layers 978 -> 945 us).
inline bool glu_tiles_192(int64_t units256, int clusters256, int64_t units192, int clusters192) {
  if (clusters256 <= 0 || clusters192 <= 0) return false;
  const int64_t r256 = (units256 + clusters256 - 1) / clusters256, r192 = (units192 + clusters192 - 1) / clusters192;
  return r192 * 192 * 100 <= r256 * 256 * 85;
}

}  // namespace tadm
