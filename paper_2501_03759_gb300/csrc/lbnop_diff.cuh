// a - b - mean to the last bit of FP32 without FP64 arithmetic per value, which runs at a fiftieth
// of the FP32 rate. The kernel that uses it (head_bwd_kernel, 16 fields of 512^2) takes 16 us, bound
// by its arithmetic and reductions; FP64 differences alone would take about 35. With the mean cut to
// two FP32 values (48 bits) it took 13, with the check for overflow after every value 47.
#pragma once

#ifdef __CUDACC__
#define LBNOP_HD __host__ __device__ __forceinline__
#else
#define LBNOP_HD inline
#endif

namespace lbnop_diff {

// A double as three FP32 values: all of its 53 bits (down to the subnormals of FP32).
struct Mean3 {
  double d;
  float h, l, ll;
};
LBNOP_HD Mean3 split(double m) {
  Mean3 r;
  r.d = m;
  r.h = (float)m;
  const double rest = m - (double)r.h;
  r.l = (float)rest;
  r.ll = (float)(rest - (double)r.l);
  return r;
}

// Knuth's two-sum: s + e = a + b exactly.
LBNOP_HD void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// a - b - m where nothing overflows. The sums of the leading terms are exact, and what is rounded
// before the last addition lies 2^24 below a term that is itself at most a rounding error of its
// sum: the result is as near as the difference formed in FP64 and rounded once, also where a - b and
// m cancel.
LBNOP_HD float diff(float a, float b, const Mean3& m) {
  float d, e, s, f, g, h, u, v;
  two_sum(a, -b, d, e);
  two_sum(d, -m.h, s, f);
  two_sum(e, -m.l, g, h);
  two_sum(s, g, u, v);
  return u + (v + (f + (h - m.ll)));
}

// Four of them. Where FP32 overflows, FP64 decides what they are (finite, infinite or NaN).
LBNOP_HD void diff4(const float (&a)[4], const float (&b)[4], const Mean3& m, float (&r)[4]) {
  float bad = 0.0f;  // stays 0 while every result is finite
  for (int k = 0; k < 4; ++k) {
    r[k] = diff(a[k], b[k], m);
    bad += r[k] - r[k];
  }
  if (bad != 0.0f)
    for (int k = 0; k < 4; ++k) r[k] = (float)((double)a[k] - (double)b[k] - m.d);
}

}  // namespace lbnop_diff
