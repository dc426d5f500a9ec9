// Packed double-float arithmetic: two double-float numbers per operation, one for site i
// and one for site i + V/2, on the two lanes of the FP32x2 instructions.
//
// sm_103a issues one FP32x2 operation (add, sub, mul, fma on a register pair) in the slot of
// one scalar operation; the FP32 pipes do the same number of lane operations per clock
// either way (38.3 T/s measured for both forms), so the packed form halves the issue slots
// of the error-free transformations and leaves the other half to loads and addresses. Pairing a site with
// the one half the lattice further in t makes every operand of the Wilson kernel a natural
// pair: the neighbours of a pair are a pair again, with its lanes exchanged when a hop in t
// leaves its half of the lattice.
#pragma once
#include "common.cuh"
#include "threeword.h"

namespace ovl {

typedef unsigned long long f2;   // two floats: low word lane 0 (site i), high word lane 1 (site i + V/2)

__device__ __forceinline__ f2 pk(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void upk(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 bc(float a) { return pk(a, a); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// fl(a b) that stays a product: ptxas contracts a mul.rn.f32x2 whose only use is an add or sub
// into a fused multiply-add (for the packed form also with an explicit rounding and with
// contraction off; measured: 40% of the sums of products differ), which breaks the error-free
// transformations. A fused multiply-add of -0, which it cannot see to be -0, is the same
// product at the same cost.
static __constant__ f2 c_minus_zero = 0x8000000080000000ull;
__device__ __forceinline__ f2 prod2(f2 a, f2 b) { return fma2(a, b, c_minus_zero); }
__device__ __forceinline__ f2 neg2(f2 a) { return sub2(0ull, a); }
__device__ __forceinline__ f2 swap2(f2 a) { return (a >> 32) | (a << 32); }

// two double-floats h + l
struct dd2 {
  f2 h, l;
};
__device__ __forceinline__ dd2 dd2_zero() { return {0ull, 0ull}; }
__device__ __forceinline__ dd2 dd2_neg(dd2 a) { return {neg2(a.h), neg2(a.l)}; }
__device__ __forceinline__ dd2 dd2_bc(double x) {
  const float h = (float)x;
  return {bc(h), bc((float)(x - (double)h))};
}
__device__ __forceinline__ dd2 dd2_from(double a, double b) {
  const float ha = (float)a, hb = (float)b;
  return {pk(ha, hb), pk((float)(a - (double)ha), (float)(b - (double)hb))};
}
__device__ __forceinline__ void dd2_to(dd2 v, double& a, double& b) {
  float h0, h1, l0, l1;
  upk(v.h, h0, h1);
  upk(v.l, l0, l1);
  a = (double)h0 + (double)l0;
  b = (double)h1 + (double)l1;
}

// a + b: TwoSum of the high words (nv = -(s - a)), low words and rounding error added, and
// renormalised (FastTwoSum): the sum of common.cuh on both lanes
__device__ __forceinline__ dd2 dd2_add(dd2 a, dd2 b) {
  const f2 s = add2(a.h, b.h);
  const f2 nv = sub2(a.h, s);
  const f2 t = add2(s, nv);
  const f2 e0 = add2(sub2(a.h, t), add2(b.h, nv));
  const f2 e = add2(e0, add2(a.l, b.l));
  const f2 h = add2(s, e);
  return {h, sub2(e, sub2(h, s))};
}
// the same without the renormalisation ("lazy"), of a + g b with g = +-1 on both lanes
__device__ __forceinline__ dd2 dd2_lazy(dd2 a, dd2 b, f2 g) {
  const f2 s = fma2(b.h, g, a.h);
  const f2 nv = sub2(a.h, s);
  const f2 t = add2(s, nv);
  const f2 e = add2(sub2(a.h, t), fma2(b.h, g, nv));
  return {s, fma2(b.l, g, add2(a.l, e))};
}
__device__ __forceinline__ dd2 dd2_lazy(dd2 a, dd2 b) {
  const f2 s = add2(a.h, b.h);
  const f2 nv = sub2(a.h, s);
  const f2 t = add2(s, nv);
  const f2 e = add2(sub2(a.h, t), add2(b.h, nv));
  return {s, add2(add2(a.l, b.l), e)};
}
// h + l renormalised (FastTwoSum; |h| > |l|)
__device__ __forceinline__ dd2 dd2_norm(dd2 a) {
  const f2 h = add2(a.h, a.l);
  return {h, sub2(a.l, sub2(h, a.h))};
}
// a factor that many products share: high word, its negative, low word
struct fac2 {
  f2 h, n, l;
};
__device__ __forceinline__ fac2 fac2_of(dd2 v) { return {v.h, neg2(v.h), v.l}; }
__device__ __forceinline__ fac2 fac2_bc(double x) { return fac2_of(dd2_bc(x)); }
__device__ __forceinline__ fac2 fac2_minus(float2 f) { return {bc(-f.x), bc(f.x), bc(-f.y)}; }   // -(f.x + f.y)
__device__ __forceinline__ dd2 dd2_mul(fac2 a, dd2 b) {
  const f2 p = prod2(a.h, b.h);
  f2 e = fma2(a.h, b.h, prod2(a.n, b.h));   // the exact rounding error of p
  e = fma2(a.h, b.l, e);
  e = fma2(a.l, b.h, e);
  const f2 h = add2(p, e);
  return {h, sub2(e, sub2(h, p))};
}

// Compensated dot product (Dot2 of Ogita, Rump and Oishi, 2005) with the sum s and the
// errors c apart, one term x y with x = (xh, xl) and y given as (y, -y, yl). With np = -fl(x y),
// s1 = s - np and v = s1 - s (nv = -v), the TwoSum error of s + fl(x y) is
// (s - (s1 - v)) + (fl(x y) - v) and the product's own error is x y - fl(x y): the last two
// together are x y - v, one fused multiply-add, so that a term costs ten operations.
struct dot2p {
  f2 s, c;
};
__device__ __forceinline__ dot2p dot2p_first(f2 xh, f2 xl, f2 y, f2 yn, f2 yl) {
  dot2p d;
  d.s = prod2(xh, y);
  d.c = fma2(xh, y, prod2(xh, yn));
  d.c = fma2(xh, yl, d.c);
  d.c = fma2(xl, y, d.c);
  return d;
}
// TIGHT: the cross terms join the term's own error before it is added to c (one rounding of
// the size of c per term instead of three, in a longer chain).
template <bool TIGHT = false>
__device__ __forceinline__ void dot2p_add(dot2p& d, f2 xh, f2 xl, f2 y, f2 yn, f2 yl) {
  const f2 np = prod2(xh, yn);
  const f2 s1 = sub2(d.s, np);
  const f2 nv = sub2(d.s, s1);
  const f2 t = add2(s1, nv);
  f2 e = add2(sub2(d.s, t), fma2(xh, y, nv));
  if constexpr (TIGHT) {
    e = fma2(xh, yl, e);
    e = fma2(xl, y, e);
    d.c = add2(d.c, e);
  } else {
    f2 c = fma2(xh, yl, d.c);
    c = fma2(xl, y, c);
    d.c = add2(c, e);
  }
  d.s = s1;
}
__device__ __forceinline__ void dot2p_add(dot2p& d, dd2 x, dd2 y) { dot2p_add(d, x.h, x.l, y.h, neg2(y.h), y.l); }
// both lanes as one double
__device__ __forceinline__ double dot2p_get(dot2p d) {
  double a, b;
  dd2_to({d.s, d.c}, a, b);
  return a + b;
}

// the sum of a warp's pairs, both lanes of each, on lane 0: a fixed tree in three words
__device__ __forceinline__ double dot2p_warp_sum(dot2p d) {
  float s0, s1, c0, c1;
  upk(d.s, s0, s1);
  upk(d.c, c0, c1);
  ThreeWord v = ThreeWord{s0, c0, 0.f} + ThreeWord{s1, c1, 0.f};
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = v + ThreeWord{__shfl_down_sync(0xffffffffu, v.a, o), __shfl_down_sync(0xffffffffu, v.b, o),
                      __shfl_down_sync(0xffffffffu, v.c, o)};
  return to_double(v);
}

// real number r (0 re, 1 im) of complex component k of the pair (i, i + V/2) of field fld;
// nb = df_blocks(V)
__device__ __forceinline__ size_t dfp_at(int fld, int k, int r, int i, int nb) {
  return (((size_t)fld * nb + (i >> 5)) * 24 + 2 * k + r) * 32 + (i & 31);
}
__device__ __forceinline__ dd2 dfp_ld(const SpinorRef& f, size_t at) {
  const ulonglong2 w = *(reinterpret_cast<const ulonglong2*>(f.data) + at);
  return {w.x, w.y};
}
__device__ __forceinline__ dd2 dfp_ldg(const SpinorRef& f, size_t at) {
  const ulonglong2 w = __ldg(reinterpret_cast<const ulonglong2*>(f.data) + at);
  return {w.x, w.y};
}
__device__ __forceinline__ void dfp_st(const SpinorRef& f, size_t at, dd2 v) {
  *(reinterpret_cast<ulonglong2*>(f.data) + at) = make_ulonglong2(v.h, v.l);
}
// complex component k of the pair (i, i + V/2) of a field stored as P (P64, P32 or P64E)
template <int P>
__device__ __forceinline__ void dfp_load(const SpinorRef& f, int fld, int k, int i, dd2& re, dd2& im) {
  const int Vh = f.V >> 1;
  if constexpr (P == P64E) {
    re = dfp_ld(f, dfp_at(fld, k, 0, i, df_blocks(f.V)));
    im = dfp_ld(f, dfp_at(fld, k, 1, i, df_blocks(f.V)));
  } else if constexpr (P == P64) {
    const double2* p = reinterpret_cast<const double2*>(f.data) + ((size_t)fld * 12 + k) * f.V + i;
    const double2 a = p[0], b = p[Vh];
    re = dd2_from(a.x, b.x);
    im = dd2_from(a.y, b.y);
  } else {
    static_assert(P == P32, "dfp_load: P64E, P64 or P32");
    const float2* p = reinterpret_cast<const float2*>(f.data) + (((size_t)fld * 6 + (k >> 1)) * f.V + i) * 2 + (k & 1);
    const float2 a = p[0], b = p[2 * (size_t)Vh];
    re = {pk(a.x, b.x), 0ull};
    im = {pk(a.y, b.y), 0ull};
  }
}
template <int P>
__device__ __forceinline__ void dfp_store(const SpinorRef& f, int fld, int k, int i, dd2 re, dd2 im) {
  const int Vh = f.V >> 1;
  if constexpr (P == P64E) {
    dfp_st(f, dfp_at(fld, k, 0, i, df_blocks(f.V)), re);
    dfp_st(f, dfp_at(fld, k, 1, i, df_blocks(f.V)), im);
  } else {
    double ra, rb, ia, ib;
    dd2_to(re, ra, rb);
    dd2_to(im, ia, ib);
    if constexpr (P == P64) {
      double2* p = reinterpret_cast<double2*>(f.data) + ((size_t)fld * 12 + k) * f.V + i;
      p[0] = make_double2(ra, ia);
      p[Vh] = make_double2(rb, ib);
    } else {
      static_assert(P == P32, "dfp_store: P64E, P64 or P32");
      float2* p = reinterpret_cast<float2*>(f.data) + (((size_t)fld * 6 + (k >> 1)) * f.V + i) * 2 + (k & 1);
      p[0] = make_float2((float)ra, (float)ia);
      p[2 * (size_t)Vh] = make_float2((float)rb, (float)ib);
    }
  }
}

}  // namespace ovl
