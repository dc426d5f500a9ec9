// Sums of double-float numbers (hi + lo of two floats) in three floats a + b + c, so that adding up a
// warp's lanes loses no bit that FP64 would keep: GB300 runs FP64 additions at 1/64 of its FP32 rate,
// and two floats alone round every addition at 2^-48. Plain C++: the host tests use it too.
#pragma once

#ifdef __CUDACC__
#define OVL_HD __host__ __device__ __forceinline__
#else
#define OVL_HD inline
#endif

namespace ovl {

struct ThreeWord {
  float a, b, c;   // |b| about 2^-24 of |a|, |c| 2^-48 (not normalised)
};

// s <- fl(s + x); the rounding error (Knuth's TwoSum)
OVL_HD float exact_add(float& s, float x) {
  const float t = s + x, v = t - s;
  const float e = (s - (t - v)) + (x - v);
  s = t;
  return e;
}

// exact but for the roundings of the third word, about 2^-71 of the first
OVL_HD ThreeWord operator+(ThreeWord x, ThreeWord y) {
  const float e = exact_add(x.a, y.a);
  const float f = exact_add(x.b, y.b);
  const float g = exact_add(x.b, e);
  x.c = (x.c + y.c) + (f + g);
  return x;
}

OVL_HD double to_double(ThreeWord x) { return (double)x.a + ((double)x.b + (double)x.c); }

}  // namespace ovl
