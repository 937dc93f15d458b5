// How a 3D sweep is cut into blocks (mu3_kernel, stream3_kernel); host code, no CUDA.
#pragma once

namespace lbch3 {

// Segments of `len` planes for `tiles` columns of nz planes on `sms` SMs, for the len that is
// predicted fastest. A block walks len + warm planes; two blocks fit an SM and together take about
// 1.1 times one alone (64^3, a step of both kernels: 15 x 10 segments 31.0 us, 15 x 16 25.5 us).
// Every number of segments is tried: with a few tiles only short segments fill the GPU (with 64 at
// most, a step of 16 x 14 x 4096 took 189 us, 51 us this way). Returns the number of blocks.
inline int plan_segments(int tiles, int nz, int warm, int sms, int* len_out) {
  double best = 0.0;
  int blocks = 0;
  for (int segs = 1; segs <= nz; ++segs) {
    const int len = (nz + segs - 1) / segs, used = (nz + len - 1) / len;
    const long long b = (long long)tiles * used, q = (b + sms - 1) / sms;
    const double t = (len + warm) * (1.1 * (double)(q / 2) + (double)(q % 2));
    if (b < (1LL << 31) && (blocks == 0 || t < best)) {
      best = t;
      *len_out = len;
      blocks = (int)b;
    }
  }
  return blocks;
}

}  // namespace lbch3
