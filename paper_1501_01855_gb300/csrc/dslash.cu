// Wilson kernel K of the overlap operator (Sec. 1, the equation for aK_xy):
//
//   K psi(x) = gamma5 [ psi(x) - kappa sum_mu ( (1-gamma_mu) U_mu(x) psi(x+mu)
//                                              + (1+gamma_mu) U_mu(x-mu)^dag psi(x-mu) ) ]
//
// One thread per (site, system). (1 -+ gamma_mu) has rank 2, so each neighbour is
// projected to a half spinor (2 spins x 3 colours), multiplied by the link and
// expanded again; the spin algebra below is the DeGrand-Rossi chiral basis,
// gamma5 = diag(1, 1, -1, -1). FP32 and FP16 links are 12-real (row 3 rebuilt in
// registers) and the eight neighbours are unrolled; the double-float kernel is in
// dfwilson.cu. Threads of one block that share a site but belong to different
// systems read the same links, so the link bytes of a multi-system launch come from L1
// once per block. Launch shapes (chosen per precision by the autotuner at create):
// BX consecutive sites x up to 4 systems per block; four threads per site, one per
// direction; 8x4x4x2 site tiles.
//
// Three fused epilogues cover every use in the sign function (Sec. 3):
//   MODE_K    out = K in, partial sums of ||out||^2 and ||in||^2
//             (first half of a multi-shift CG step: (p, K^2 p) = ||K p||^2);
//   MODE_R    r -= alpha (K t + sigma0 p), partial sums of ||r||^2
//             (second half: K^2 p + sigma0 p applied and consumed in one pass);
//   MODE_OVL  out = c1 v + c2 (y - kappa hop y) = c1 v + c2 gamma5 K y, optionally times
//             gamma5, with partial sums of (w, out): gamma5 eps(K) v and D(mu) v are
//             this with y = sum_i omega_i (K^2 + sigma_i)^-1 v.
// and two for the stored-basis Lanczos form of the same sum (lanczos.cu):
//   MODE_LZK  t = (1 / n_j) K W_j with W_j the system's current basis slot, ||t||^2;
//   MODE_LZL  W_{j+1} = K t - a W_j - b W_{j-1} (the three-term recurrence), ||W_{j+1}||^2.
#include "wilson.cuh"

namespace ovl {

// Register cap per thread, by link precision (and, for FP16 storage, spinor precision).
// Uncapped, the compiler hoists all neighbour loads and takes ~255 registers (8 warps
// per SM): the FP32/FP16 kernels are then latency-bound. Swept on 24^3x48 (ms per launch):
//   FP32 K, one system   64: 0.0619 (spills 148 B; the multi-shift r-update form 440 B)
//                        72: 0.0555   80: 0.0557 (best for 12 systems and for a whole FP32 sign)
//                        96: 0.0594
//   FP16 K, one system / 12 systems   72: 0.0575 / 0.5936   80: 0.0578 / 0.5798
//                                     96: 0.0574 / 0.6444  128: 0.0554 / 0.5816
// The FP16 cap moves its K launch by 4% at most, and at its best the launch takes as long
// as the FP32 one (0.0553 ms) with half the bytes: the bound is the latency of each site's
// chain of dependent loads, not HBM. FP16 keeps the FP32 cap.
#ifndef OVL_WILSON_REG_SP
#define OVL_WILSON_REG_SP 80
#endif
#ifndef OVL_WILSON_REG_HP
#define OVL_WILSON_REG_HP OVL_WILSON_REG_SP
#endif
template <int PL, int PIN> struct MaxReg {
  static constexpr int v = PL == P64 ? 255
                         : (PL == P16 && PIN == P16) ? OVL_WILSON_REG_HP : OVL_WILSON_REG_SP;
};

template <int MU, int S, typename T>
__device__ __forceinline__ void project(const cpx<T> p[12], cpx<T> h[6]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const cpx<T> p0 = p[c], p1 = p[3 + c], p2 = p[6 + c], p3 = p[9 + c];
    if constexpr (MU == 0) {          // h0 = p0 + S i p3, h1 = p1 + S i p2
      h[c] = S > 0 ? p0 + timesI(p3) : p0 - timesI(p3);
      h[3 + c] = S > 0 ? p1 + timesI(p2) : p1 - timesI(p2);
    } else if constexpr (MU == 1) {   // h0 = p0 - S p3, h1 = p1 + S p2
      h[c] = S > 0 ? p0 - p3 : p0 + p3;
      h[3 + c] = S > 0 ? p1 + p2 : p1 - p2;
    } else if constexpr (MU == 2) {   // h0 = p0 + S i p2, h1 = p1 - S i p3
      h[c] = S > 0 ? p0 + timesI(p2) : p0 - timesI(p2);
      h[3 + c] = S > 0 ? p1 - timesI(p3) : p1 + timesI(p3);
    } else {                          // h0 = p0 + S p2, h1 = p1 + S p3
      h[c] = S > 0 ? p0 + p2 : p0 - p2;
      h[3 + c] = S > 0 ? p1 + p3 : p1 - p3;
    }
  }
}

// acc += (1 + S gamma_mu) expanded from the half spinor w
template <int MU, int S, typename T>
__device__ __forceinline__ void accumulate(cpx<T> acc[12], const cpx<T> w[6]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const cpx<T> w0 = w[c], w1 = w[3 + c];
    acc[c] = acc[c] + w0;
    acc[3 + c] = acc[3 + c] + w1;
    if constexpr (MU == 0) {          // lower = (-S i w1, -S i w0)
      acc[6 + c] = acc[6 + c] + (S > 0 ? timesMinusI(w1) : timesI(w1));
      acc[9 + c] = acc[9 + c] + (S > 0 ? timesMinusI(w0) : timesI(w0));
    } else if constexpr (MU == 1) {   // lower = (S w1, -S w0)
      acc[6 + c] = S > 0 ? acc[6 + c] + w1 : acc[6 + c] - w1;
      acc[9 + c] = S > 0 ? acc[9 + c] - w0 : acc[9 + c] + w0;
    } else if constexpr (MU == 2) {   // lower = (-S i w0, S i w1)
      acc[6 + c] = acc[6 + c] + (S > 0 ? timesMinusI(w0) : timesI(w0));
      acc[9 + c] = acc[9 + c] + (S > 0 ? timesI(w1) : timesMinusI(w1));
    } else {                          // lower = (S w0, S w1)
      acc[6 + c] = S > 0 ? acc[6 + c] + w0 : acc[6 + c] - w0;
      acc[9 + c] = S > 0 ? acc[9 + c] + w1 : acc[9 + c] - w1;
    }
  }
}

// The six products of a real number as two chains of multiply-adds of three and their sum: 7
// operations (a sum of three complex products takes 8) with partial sums no larger than there; one
// chain of six takes 6 but rounds larger partial sums (error of FP64 K against 64 bits 1.5e-16
// against 1.4e-16). The diagonal entry of the row comes last in both chains: on smooth fields it is
// nearly one and the others are small, so that only two of the seven roundings are of the size of
// the sum, three on average in the order of the columns: FP32 K on 24^3 x 48 5.45e-8 of the norm,
// 5.70e-8 in the order of the columns, 5.65e-8 as three products; FP64 K on 16^3 x 32 1.344e-16,
// 1.376e-16 and 1.369e-16. With the stored third row: K of 12 FP64 systems on 16^3 x 32 4.16 -> 3.15 ms,
// FP32 sign of 12 systems 21.3 -> 20.8 ms (20.7 in the order of the columns). S = +1: a b, -1: conj(a) b;
// (a2, b2) the diagonal entry's.
template <int S, typename T>
__device__ __forceinline__ cpx<T> dot3(cpx<T> a0, cpx<T> b0, cpx<T> a1, cpx<T> b1, cpx<T> a2, cpx<T> b2) {
  const T i0 = S > 0 ? a0.i : -a0.i, i1 = S > 0 ? a1.i : -a1.i, i2 = S > 0 ? a2.i : -a2.i;
  return {fma(a2.r, b2.r, fma(-i0, b0.i, a0.r * b0.r)) + fma(-i2, b2.i, fma(-i1, b1.i, a1.r * b1.r)),
          fma(a2.r, b2.i, fma(i0, b0.r, a0.r * b0.i)) + fma(i2, b2.r, fma(i1, b1.r, a1.r * b1.i))};
}
template <typename T>
__device__ __forceinline__ void su3_mul(const cpx<T> u[9], const cpx<T> h[6], cpx<T> w[6]) {
#pragma unroll
  for (int sp = 0; sp < 2; ++sp)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int b = a == 0 ? 1 : 0, c = a == 2 ? 1 : 2;   // the other two, ascending
      w[3 * sp + a] = dot3<1>(u[3 * a + b], h[3 * sp + b], u[3 * a + c], h[3 * sp + c], u[4 * a], h[3 * sp + a]);
    }
}
template <typename T>
__device__ __forceinline__ void su3_dag_mul(const cpx<T> u[9], const cpx<T> h[6], cpx<T> w[6]) {
#pragma unroll
  for (int sp = 0; sp < 2; ++sp)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int b = a == 0 ? 1 : 0, c = a == 2 ? 1 : 2;   // the other two, ascending
      w[3 * sp + a] = dot3<-1>(u[3 * b + a], h[3 * sp + b], u[3 * c + a], h[3 * sp + c], u[4 * a], h[3 * sp + a]);
    }
}

// Per-thread sums for the epilogue reductions, kept in the compute type: GB300 runs
// FP64 (and FP32 <-> FP64 conversions) at a small fraction of its FP32 rate, so the FP32
// and FP16-storage kernels sum in FP32 (their own precision) and convert once; the
// double-float kernel sums with Dot2, which keeps its FP64-level accuracy on FP32 pipes.
template <typename T> struct Acc {
  T s = T(0);
  __device__ __forceinline__ void add(T x, T y) { s = fma(x, y, s); }
  __device__ __forceinline__ typename RedT<T>::type get() const { return s; }
};
template <typename T>
__device__ __forceinline__ void acc_norm(Acc<T>& a, const cpx<T>& z) {
  a.add(z.r, z.r);
  a.add(z.i, z.i);
}

// FIRST: this hop starts the sum (saves 24 additions).
template <int MU, int PIN, int PL, bool RO, typename T, bool FIRST = false>
__device__ __forceinline__ void hop_dir(const Geom& g, const LinkRef& L, const SpinorRef& in, int rhs, int s,
                                        const int x[4], int stride, cpx<T> acc[12]) {
  cpx<T> psi[12], h[6], w[6], u[9];
  // forward neighbour: (1 - gamma_mu) U_mu(x) psi(x + mu)
  {
    const bool wrap = x[MU] == g.L[MU] - 1;
    const int sf = wrap ? s - (g.L[MU] - 1) * stride : s + stride;
    load_spinor_gen<PIN, T, RO>(in, rhs, sf, psi);
    project<MU, -1>(psi, h);
    if (MU == 3 && g.bc_t && wrap) {
#pragma unroll
      for (int k = 0; k < 6; ++k) h[k] = -h[k];
    }
    load_link<PL, T>(L, MU, s, u);
    su3_mul(u, h, w);
    if constexpr (FIRST) {
      static_assert(MU == 0, "the first direction");
#pragma unroll
      for (int k = 0; k < 6; ++k) acc[k] = w[k];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        acc[6 + c] = timesI(w[3 + c]);
        acc[9 + c] = timesI(w[c]);
      }
    } else {
      accumulate<MU, -1>(acc, w);
    }
  }
  // backward neighbour: (1 + gamma_mu) U_mu(x - mu)^dag psi(x - mu)
  {
    const bool wrap = x[MU] == 0;
    const int sb = wrap ? s + (g.L[MU] - 1) * stride : s - stride;
    load_spinor_gen<PIN, T, RO>(in, rhs, sb, psi);
    project<MU, +1>(psi, h);
    if (MU == 3 && g.bc_t && wrap) {
#pragma unroll
      for (int k = 0; k < 6; ++k) h[k] = -h[k];
    }
    load_link<PL, T>(L, MU, sb, u);
    su3_dag_mul(u, h, w);
    accumulate<MU, +1>(acc, w);
  }
}

template <int PIN, int PL, bool RO, typename T>
__device__ __forceinline__ void hop(const Geom& g, const LinkRef& L, const SpinorRef& in, int rhs, int s,
                                    const int x[4], cpx<T> acc[12]) {
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = cmk(T(0), T(0));
  const int sy = g.L[0], sz = g.L[0] * g.L[1], st = sz * g.L[2];
  hop_dir<0, PIN, PL, RO, T>(g, L, in, rhs, s, x, 1, acc);
  hop_dir<1, PIN, PL, RO, T>(g, L, in, rhs, s, x, sy, acc);
  hop_dir<2, PIN, PL, RO, T>(g, L, in, rhs, s, x, sz, acc);
  hop_dir<3, PIN, PL, RO, T>(g, L, in, rhs, s, x, st, acc);
}

// Epilogue shared by both kernel variants: acc holds the hop sum of site s; v gets this
// thread's contributions to the NVRED partial sums (see the mode list at the top).
template <int MODE, int PIN, int POUT, int PA1, int PA2, typename T, typename LT>
__device__ __forceinline__ void wilson_epilogue(const DArgs& a, const LT* L, int rhs, int fin, int s, cpx<T> acc[12],
                                                typename RedT<T>::type v[NVRED]) {
  cpx<T> c[12];
  load_spinor_gen<PIN, T, kReadOnly<MODE>>(a.in, fin, s, c);
  T kap;   // the compute type's copies of the coefficients (conversions from FP64 are slow)
  if constexpr (std::is_same<T, float>::value) kap = a.kap_h;
  else kap = a.kappa;
  const bool red = a.partials != nullptr;
  if constexpr (MODE == MODE_LZK) {
    // t = (1 / n_j) gamma5 (W_j - kappa hop W_j)
    T sc;
    if constexpr (std::is_same<T, float>::value) sc = L->fn.x;
    else sc = L->inv_n;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      cpx<T> o = c[k] - kap * acc[k];
      if (k >= 6) o = -o;
      acc[k] = sc * o;
    }
    store_spinor_as<POUT, T>(a.out, rhs, s, acc);
    if (red) {
      Acc<T> n0;
#pragma unroll
      for (int k = 0; k < 12; ++k) acc_norm(n0, acc[k]);
      v[0] = n0.get();
    }
  } else if constexpr (MODE == MODE_LZL) {
    // W_{j+1} = gamma5 (t - kappa hop t) - a W_j - b W_{j-1}
    const int j = L->j;
    T ca, cb;
    if constexpr (std::is_same<T, float>::value) {
      ca = L->fa.x;
      cb = L->fb.x;
    } else {
      ca = L->a;
      cb = L->b;
    }
    cpx<T> w[12];
    load_spinor_as<PA1, T>(a.aux1, j * a.nrhs + rhs, s, w);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      cpx<T> o = c[k] - kap * acc[k];
      if (k >= 6) o = -o;
      acc[k] = o - ca * w[k];
    }
    if (j > 0) {
      load_spinor_as<PA1, T>(a.aux1, (j - 1) * a.nrhs + rhs, s, w);
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[k] = acc[k] - cb * w[k];
    }
    store_spinor_as<POUT, T>(a.out, (j + 1) * a.nrhs + rhs, s, acc);
    if (red) {
      Acc<T> n0;
#pragma unroll
      for (int k = 0; k < 12; ++k) acc_norm(n0, acc[k]);
      v[0] = n0.get();
    }
  } else if constexpr (MODE == MODE_K) {
    // K in = gamma5 (in - kappa acc)
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      cpx<T> o = c[k] - kap * acc[k];
      if (k >= 6) o = -o;
      acc[k] = o;
    }
    store_spinor_as<POUT, T>(a.out, rhs, s, acc);
    if (red) {
      Acc<T> n0, n1;
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        acc_norm(n0, acc[k]);
        acc_norm(n1, c[k]);
      }
      v[0] = n0.get();
      v[1] = n1.get();
    }
  } else if constexpr (MODE == MODE_R) {
    cpx<T> p[12], r[12];
    load_spinor_as<PA1, T>(a.aux1, rhs, s, p);
    load_spinor_as<PA2, T>(a.aux2, rhs, s, r);
    const T sg = (T)a.sigma0;
    const T al = (T)a.ms[rhs].alpha;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      cpx<T> o = c[k] - kap * acc[k];
      if (k >= 6) o = -o;
      o = o + sg * p[k];
      r[k] = r[k] - al * o;
    }
    store_spinor_as<PA2, T>(a.aux2, rhs, s, r);
    if (red) {
      Acc<T> n0;
#pragma unroll
      for (int k = 0; k < 12; ++k) acc_norm(n0, r[k]);
      v[0] = n0.get();
    }
  } else {
    cpx<T> w[12];
    T c1 = (T)a.c1, c2 = (T)a.c2;
    if (a.coef != nullptr) {
      c1 = (T)a.coef[2 * rhs];
      c2 = (T)a.coef[2 * rhs + 1];
    }
    if (c1 != T(0)) {
      load_spinor_as<PA1, T>(a.aux1, rhs, s, w);
    } else {
#pragma unroll
      for (int k = 0; k < 12; ++k) w[k] = cmk(T(0), T(0));
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      cpx<T> o = c1 * w[k] + c2 * (c[k] - kap * acc[k]);
      if (a.herm && k >= 6) o = -o;
      acc[k] = o;
    }
    store_spinor_as<POUT, T>(a.out, rhs, s, acc);
    if (red) {
      load_spinor_as<PA2, T>(a.aux2, rhs, s, w);
      Acc<T> dr, di, n0, n1;   // (w, out) = sum conj(w) out
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        dr.add(w[k].r, acc[k].r);
        dr.add(w[k].i, acc[k].i);
        di.add(w[k].r, acc[k].i);
        di.add(-w[k].i, acc[k].r);
        acc_norm(n0, acc[k]);
        acc_norm(n1, w[k]);
      }
      v[0] = dr.get();
      v[1] = di.get();
      v[2] = n0.get();
      v[3] = n1.get();
    }
  }
}

// Variant 0: one thread per (site, system) walks all eight neighbours; a block is BX
// consecutive sites (x fastest) times up to 4 systems.
// Variant 2 (TILED): a block is one system on a 4D tile of TX x TY x TZ x TT = 256 sites,
// so that the neighbours in all four directions mostly lie in the block's own tile
// (L1 hits) instead of BX/Lx rows away in z and t. Needs every extent divisible by the
// tile. Its block sum goes to the first of the tile's 256/BX partial slots (the others
// get zero), so the partial layout (system, BX-site block) is the same for all variants.
constexpr int TX = 8, TY = 4, TZ = 4, TT = 2;
template <int MODE, int PIN, int PL, int POUT, int PA1, int PA2, bool TILED>
__global__ void __launch_bounds__(256) __maxnreg__((MaxReg<PL, PIN>::v)) wilson_kernel(const DArgs a) {
  using T = typename Real<PL>::T;
  __shared__ double red[4 * (BX / 32) * NVRED];
  int sb, rhs, s;
  int x[4];
  bool live;
  if constexpr (TILED) {
    const int ntx = a.g.L[0] / TX, nty = a.g.L[1] / TY, ntz = a.g.L[2] / TZ;
    int b = blockIdx.x;
    const int bx = b % ntx;
    b /= ntx;
    const int by = b % nty;
    b /= nty;
    const int bz = b % ntz;
    const int bt = b / ntz;
    const int t = threadIdx.x;
    x[0] = bx * TX + (t & 7);
    x[1] = by * TY + ((t >> 3) & 3);
    x[2] = bz * TZ + ((t >> 5) & 3);
    x[3] = bt * TT + (t >> 7);
    s = ((x[3] * a.g.L[2] + x[2]) * a.g.L[1] + x[1]) * a.g.L[0] + x[0];
    rhs = blockIdx.y;
    sb = blockIdx.x * (TX * TY * TZ * TT / BX);
    live = rhs < a.nrhs;
  } else {
    sb = blockIdx.x / a.ngr;
    const int rg = blockIdx.x - sb * a.ngr;
    rhs = rg * blockDim.y + threadIdx.y;
    s = sb * BX + threadIdx.x;
    live = (s < a.g.V) && (rhs < a.nrhs);
    if (live) site_coords(a.g, s, x);
  }
  if constexpr (!kReadOnly<MODE>) {
    pdl_wait();
    pdl_release();
  }
  if (live && a.ms != nullptr && (MODE == MODE_K || MODE == MODE_R)) live = !a.ms[rhs].done;
  int fin = rhs;   // field index of the hop input (the basis slot in MODE_LZK)
  bool act = false;
  if constexpr (MODE == MODE_LZK || MODE == MODE_LZL) {
    act = rhs < a.nrhs && !a.lz[rhs].done;
    // a block whose systems are all done leaves at once: launches past the end of a sign cost
    // little more than their dispatch
    if (blockDim.y == 1 ? !act : !__syncthreads_or(act)) return;
    live = live && act;
    if (MODE == MODE_LZK && live) fin = a.lz[rhs].j * a.nrhs + rhs;
  }
  using R = typename RedT<T>::type;
  R v[NVRED] = {R(0), R(0), R(0), R(0)};
  if (live) {
    cpx<T> acc[12];
    hop<PIN, PL, kReadOnly<MODE>, T>(a.g, a.links, a.in, fin, s, x, acc);
    wilson_epilogue<MODE, PIN, POUT, PA1, PA2, T>(a, a.lz + rhs, rhs, fin, s, acc, v);
  }
  if (a.partials != nullptr) {
    double tot[NVRED];
    block_reduce_partials<R, nred(MODE)>(v, red, tot);
    if (threadIdx.x == 0 && rhs < a.nrhs) {
      store_partials<MODE>(a, rhs, sb, tot);
      if constexpr (TILED) {
        const double zero[NVRED] = {0.0, 0.0, 0.0, 0.0};
        for (int q = 1; q < TX * TY * TZ * TT / BX; ++q) store_partials<MODE>(a, rhs, sb + q, zero);
      }
    }
  }
  if constexpr (MODE == MODE_LZK || MODE == MODE_LZL) {
    if (threadIdx.x < 32 && act) lz_arrive<MODE>(a, rhs, TILED ? (int)gridDim.x : a.nsb);
  }
}

// true when the lattice can be covered by whole variant-2 tiles
bool wilson_tiles_fit(const Geom& g) {
  return g.L[0] % TX == 0 && g.L[1] % TY == 0 && g.L[2] % TZ == 0 && g.L[3] % TT == 0;
}

// FP32 K straight into the caller's canonical single-precision spinors (24 consecutive reals per
// site): a row of the block turns its 64 sites over in shared memory (rows of 25 reals: no bank
// conflicts) and writes whole 16-byte words, instead of an internal field written here and read
// again by the unpack kernel: 24^3 x 48 from caller buffers 111 -> 95 us, 12 systems 1.01 -> 0.85 ms.
constexpr int CT = 25;   // reals per tile row
__global__ void __launch_bounds__(4 * BX, 3) wilson_f32_canon_kernel(const DArgs a, float* canon) {
  extern __shared__ float tiles[];
  const int sb = blockIdx.x / a.ngr;
  const int rg = blockIdx.x - sb * a.ngr;
  const int rhs = rg * blockDim.y + threadIdx.y;
  const int s = sb * BX + threadIdx.x;
  float* tile = tiles + threadIdx.y * (BX * CT);
  if (s < a.g.V && rhs < a.nrhs) {
    int x[4];
    site_coords(a.g, s, x);
    cpx<float> acc[12], c[12];
    hop<P32, P32, true, float>(a.g, a.links, a.in, rhs, s, x, acc);
    load_spinor_gen<P32, float, true>(a.in, rhs, s, c);
    float* t = tile + threadIdx.x * CT;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      cpx<float> o = c[k] - a.kap_h * acc[k];
      if (k >= 6) o = -o;
      t[2 * k] = o.r;
      t[2 * k + 1] = o.i;
    }
  }
  __syncthreads();
  if (rhs >= a.nrhs) return;
  const int words = min(BX, a.g.V - sb * BX) * 6;
  float4* d = reinterpret_cast<float4*>(canon + ((size_t)rhs * a.g.V + (size_t)sb * BX) * 24);
  for (int e = threadIdx.x; e < words; e += BX) {
    const float* t = tile + (e / 6) * CT + (e % 6) * 4;
    d[e] = make_float4(t[0], t[1], t[2], t[3]);
  }
}

// Variant 1 (direction split): a block of 4 * BX threads covers BX sites of one system;
// warp w handles direction w % 4 (forward and backward hop) for the 32 sites of group
// w / 4, so every thread walks two neighbours instead of eight and the direction is
// uniform within a warp. The four partial sums meet in shared memory and the
// direction-0 warps finish the site.
template <int MODE, int PIN, int PL, int POUT, int PA1, int PA2>
__global__ void __launch_bounds__(4 * BX) __maxnreg__((MaxReg<PL, PIN>::v)) wilson_split_kernel(const DArgs a) {
  using T = typename Real<PL>::T;
  __shared__ cpx<T> part[3][BX][12];
  __shared__ double red[(4 * BX / 32) * NVRED];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int dir = warp & 3, grp = warp >> 2;
  const int sb = blockIdx.x / a.nrhs;
  const int rhs = blockIdx.x - sb * a.nrhs;
  const int sl = grp * 32 + lane;
  const int s = sb * BX + sl;
  bool live = s < a.g.V;
  if constexpr (!kReadOnly<MODE>) {
    pdl_wait();
    pdl_release();
  }
  if (live && a.ms != nullptr && (MODE == MODE_K || MODE == MODE_R)) live = !a.ms[rhs].done;
  int fin = rhs;
  if constexpr (MODE == MODE_LZK || MODE == MODE_LZL) {
    if (a.lz[rhs].done) return;   // every thread of the block
    if (MODE == MODE_LZK) fin = a.lz[rhs].j * a.nrhs + rhs;
  }
  cpx<T> acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = cmk(T(0), T(0));
  if (live) {
    int x[4];
    site_coords(a.g, s, x);
    const int sy = a.g.L[0], sz = sy * a.g.L[1], st = sz * a.g.L[2];
    if (dir == 0) hop_dir<0, PIN, PL, kReadOnly<MODE>, T>(a.g, a.links, a.in, fin, s, x, 1, acc);
    else if (dir == 1) hop_dir<1, PIN, PL, kReadOnly<MODE>, T>(a.g, a.links, a.in, fin, s, x, sy, acc);
    else if (dir == 2) hop_dir<2, PIN, PL, kReadOnly<MODE>, T>(a.g, a.links, a.in, fin, s, x, sz, acc);
    else hop_dir<3, PIN, PL, kReadOnly<MODE>, T>(a.g, a.links, a.in, fin, s, x, st, acc);
  }
  if (dir != 0) {
#pragma unroll
    for (int k = 0; k < 12; ++k) part[dir - 1][sl][k] = acc[k];
  }
  __syncthreads();
  using R = typename RedT<T>::type;
  R v[NVRED] = {R(0), R(0), R(0), R(0)};
  if (dir == 0 && live) {
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = acc[k] + part[0][sl][k] + part[1][sl][k] + part[2][sl][k];
    wilson_epilogue<MODE, PIN, POUT, PA1, PA2, T>(a, a.lz + rhs, rhs, fin, s, acc, v);
  }
  if (a.partials != nullptr) {
    double tot[NVRED];
    block_reduce_partials<R, nred(MODE)>(v, red, tot);
    if (threadIdx.x == 0) {
      store_partials<MODE>(a, rhs, sb, tot);
    }
  }
  if constexpr (MODE == MODE_LZK || MODE == MODE_LZL) {
    if (threadIdx.x < 32) lz_arrive<MODE>(a, rhs, a.nsb);
  }
}

// ---- FP32, the whole Lanczos iteration in one launch (lzp_run) ---------------------------
// A tile is 32 sites of one system: one warp (NS = 1), or four warps, one per direction, whose
// sums meet in shared memory (NS = 4, when that still gives every tile its warps at once).
template <int NS>
struct LzpBody32 {
  const LzPersist& p;
  const DArgs& a;
  cpx<float>* part;   // NS > 1: [warp][component][lane]
  cpx<float> acc[12];
  int rhs, s;
  bool in_tile, live;
  __device__ __forceinline__ LzpBody32(const LzPersist& q, cpx<float>* sm) : p(q), a(q.a), part(sm) {
    const int tile = blockIdx.x * p.tb + (threadIdx.x >> 5) / NS;
    rhs = tile % a.nrhs;
    s = tile / a.nrhs * 32 + lane_id();
    in_tile = tile < p.ntile && s < a.g.V;
  }
  template <int MODE>
  __device__ __forceinline__ void sum(int j, const LzpShared& sh) {
    live = in_tile && !sh.c[rhs].done;
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = cmk(0.f, 0.f);
    if (!live) return;
    const SpinorRef& in = MODE == MODE_LZK ? p.W : p.t;
    const int fin = MODE == MODE_LZK ? j * a.nrhs + rhs : rhs;
    int x[4];
    site_coords(a.g, s, x);
    const int sy = a.g.L[0], sz = sy * a.g.L[1], st = sz * a.g.L[2];
    const int dir = NS == 1 ? -1 : (threadIdx.x >> 5) % NS;
    if (NS == 1 || dir == 0) hop_dir<0, P32, P32, false, float, true>(a.g, a.links, in, fin, s, x, 1, acc);
    if (NS == 1 || dir == 1) hop_dir<1, P32, P32, false, float>(a.g, a.links, in, fin, s, x, sy, acc);
    if (NS == 1 || dir == 2) hop_dir<2, P32, P32, false, float>(a.g, a.links, in, fin, s, x, sz, acc);
    if (NS == 1 || dir == 3) hop_dir<3, P32, P32, false, float>(a.g, a.links, in, fin, s, x, st, acc);
  }
  template <int MODE>
  __device__ __forceinline__ void hop(int j, const LzpShared& sh) {
    sum<MODE>(j, sh);
    if constexpr (NS > 1) {
      const int w = threadIdx.x >> 5;
      if (w % NS != 0) {
#pragma unroll
        for (int k = 0; k < 12; ++k) part[(w * 12 + k) * 32 + lane_id()] = acc[k];
      }
    }
  }
  template <int MODE>
  __device__ __forceinline__ void finish(int j, LzpShared& sh) {
    const int w = threadIdx.x >> 5, lane = lane_id();
    if (NS > 1 && w % NS != 0) return;
    if constexpr (NS > 1) {
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        const cpx<float>* q = part + ((w + 1) * 12 + k) * 32 + lane;
        acc[k] = acc[k] + q[0] + q[12 * 32] + q[24 * 32];
      }
    }
    float v[NVRED] = {0.f, 0.f, 0.f, 0.f};
    // this phase's flags: a system found done since the hop keeps its vectors
    if (live && !sh.c[rhs].done)
      wilson_epilogue<MODE, P32, P32, P32, P32, float>(MODE == MODE_LZK ? p.a : p.l, &sh.c[rhs], rhs,
                                                       MODE == MODE_LZK ? j * a.nrhs + rhs : rhs, s, acc, v);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[0] += __shfl_down_sync(0xffffffffu, v[0], o);
    if (lane == 0) sh.acc[w][rhs] = (double)v[0];
  }
};
template <int NS, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 1) lz_persistent_f32_kernel(const LzPersist p) {
  extern __shared__ cpx<float> parts32[];
  __shared__ LzpShared sh;
  LzpBody32<NS> body(p, parts32);
  lzp_run(p, body, sh);
}

Shape make_shape(int V, int nrhs) {
  Shape s;
  s.nsb = (V + BX - 1) / BX;
  s.by = nrhs < 4 ? nrhs : 4;
  s.ngr = (nrhs + s.by - 1) / s.by;
  return s;
}

template <int MODE, int PIN, int PL, int POUT, int PA1, int PA2>
static void run(DArgs a, cudaStream_t st) {
  Shape sh = make_shape(a.g.V, a.nrhs);
  a.nsb = sh.nsb;
  a.ngr = sh.ngr;
  if (a.variant == 1) {
    // one system per block; partials keep the (system, BX-site block) layout of variant 0
    launch_step(wilson_split_kernel<MODE, PIN, PL, POUT, PA1, PA2>, dim3((unsigned)(sh.nsb * a.nrhs)), dim3(4 * BX), 0, st, a);
  } else if (a.variant == 2 && wilson_tiles_fit(a.g)) {
    const unsigned ntiles = (unsigned)(a.g.V / (TX * TY * TZ * TT));
    launch_step(wilson_kernel<MODE, PIN, PL, POUT, PA1, PA2, true>, dim3(ntiles, (unsigned)a.nrhs), dim3(TX * TY * TZ * TT), 0, st, a);
  } else {
    launch_step(wilson_kernel<MODE, PIN, PL, POUT, PA1, PA2, false>, sh.grid(), sh.block(), 0, st, a);
  }
}

static DArgs base_args(const Geom& g, double kappa, LinkRef links, int nrhs) {
  DArgs a;
  a.g = g;
  a.kappa = kappa;
  const float2 kf = split_df(kappa);
  a.kap_h = kf.x;
  a.kap_l = kf.y;
  a.links = links;
  a.in = a.out = a.aux1 = a.aux2 = SpinorRef{nullptr, nullptr, g.V};
  a.nrhs = nrhs;
  a.nsb = a.ngr = 0;
  a.partials = nullptr;
  a.ms = nullptr;
  a.sigma0 = 0;
  a.c1 = a.c2 = 0;
  a.coef = nullptr;
  a.herm = 0;
  a.variant = nrhs >= 4 ? links.variant_multi : links.variant;
  a.lz = nullptr;
  a.lzc = LzCtl{nullptr, nullptr, nullptr, nullptr, 0, nullptr, 0};
  return a;
}

bool launch_lz_persistent(int prec, const Geom& g, double kappa, LinkRef links, SpinorRef W, SpinorRef t, int nrhs,
                          const LzCtl& ctl, double* part, unsigned int* bar, unsigned long long wait_ns,
                          LzpShape* shape, int nsm, cudaStream_t st) {
  if (nrhs > LZP_SYS) return false;
  LzPersist p;
  p.a = base_args(g, kappa, links, nrhs);
  p.a.lz = ctl.lz;
  p.a.lzc = ctl;
  p.a.partials = part;   // the epilogues form their partial sums
  p.a.in = W;
  p.a.out = t;
  p.l = p.a;
  p.l.in = t;
  p.l.out = p.l.aux1 = W;
  p.W = W;
  p.t = t;
  p.part = part;
  p.bar = bar;
  p.wait_ns = wait_ns;
  if (prec == P64E) return launch_lz_persistent_df(p, shape, nsm, st);
  if (prec != P32) return false;
  // FP32: every tile has its warps at once, up to 27 per SM (72 registers; up to 19: 102)
  p.ntile = (g.V + 31) / 32 * nrhs;
  p.tb = (p.ntile + nsm - 1) / nsm;
  *shape = {4 * p.tb <= 19 ? 4 : 1, p.tb};
  if (4 * p.tb <= 19)
    return lzp_launch(lz_persistent_f32_kernel<4, 20>, p, 4, 4 * 12 * 32 * sizeof(cpx<float>), 4, nsm, st);
  if (p.tb <= 19) return lzp_launch(lz_persistent_f32_kernel<1, 20>, p, 1, 0, 19, nsm, st);
  if (p.tb <= LZP_WARPS - 1)
    return lzp_launch(lz_persistent_f32_kernel<1, LZP_WARPS>, p, 1, 0, LZP_WARPS - 1, nsm, st);
  return false;
}

#define OVL_BAD_COMBO() note_bad_combo(__func__)

bool launch_wilson_K_canon32(const Geom& g, double kappa, LinkRef links, SpinorRef in, float* canon, int nrhs,
                             cudaStream_t st) {
  DArgs a = base_args(g, kappa, links, nrhs);
  if (a.variant == 1 || reinterpret_cast<uintptr_t>(canon) % 16 != 0) return false;
  a.in = in;
  const Shape sh = make_shape(g.V, nrhs);
  a.nsb = sh.nsb;
  a.ngr = sh.ngr;
  wilson_f32_canon_kernel<<<sh.grid(), sh.block(), sh.by * BX * CT * sizeof(float), st>>>(a, canon);
  return true;
}

void launch_wilson_K(int pin, int plink, int pout, const Geom& g, double kappa, LinkRef links, SpinorRef in,
                     SpinorRef out, int nrhs, double* partials, const MsRhs* ms, cudaStream_t st) {
  DArgs a = base_args(g, kappa, links, nrhs);
  a.in = in;
  a.out = out;
  a.partials = partials;
  a.ms = ms;
  if (pin == P64 && plink == P64 && pout == P64) run<MODE_K, P64, P64, P64, P64, P64>(a, st);
  else if (pin == P32 && plink == P32 && pout == P32) run<MODE_K, P32, P32, P32, P32, P32>(a, st);
  else if (pin == P16 && plink == P16 && pout == P16) run<MODE_K, P16, P16, P16, P16, P16>(a, st);
  else if (pin == P32 && plink == P16 && pout == P32) run<MODE_K, P32, P16, P32, P32, P32>(a, st);
  else if (pin == P32 && plink == P16 && pout == P16) run<MODE_K, P32, P16, P16, P32, P32>(a, st);
  else if (pin == P64E && plink == P64E && pout == P64E) run_wilson_df(MODE_K, P64E, a, st);
  else OVL_BAD_COMBO();
}

void launch_wilson_mscg_r(int pt, int plink, int pr, int pp, const Geom& g, double kappa, LinkRef links,
                          SpinorRef t, SpinorRef p0, SpinorRef r, int nrhs, double sigma0, double* partials,
                          const MsRhs* ms, cudaStream_t st) {
  DArgs a = base_args(g, kappa, links, nrhs);
  a.in = t;
  a.aux1 = p0;
  a.aux2 = r;
  a.sigma0 = sigma0;
  a.partials = partials;
  a.ms = ms;
  if (pt == P64 && plink == P64 && pr == P64 && pp == P64) run<MODE_R, P64, P64, P64, P64, P64>(a, st);
  else if (pt == P32 && plink == P32 && pr == P32 && pp == P32) run<MODE_R, P32, P32, P32, P32, P32>(a, st);
  else if (pt == P16 && plink == P16 && pr == P32 && pp == P16) run<MODE_R, P16, P16, P32, P16, P32>(a, st);
  else if (pt == P64E && plink == P64E && pr == P64E && pp == P64E) run_wilson_df(MODE_R, P64E, a, st);
  else OVL_BAD_COMBO();
}

void launch_wilson_lzK(int pw, int plink, int pt, const Geom& g, double kappa, LinkRef links, SpinorRef W,
                       SpinorRef t, int nrhs, double* partials, const LzCtl& ctl, cudaStream_t st) {
  DArgs a = base_args(g, kappa, links, nrhs);
  a.in = W;
  a.out = t;
  a.partials = partials;
  a.lz = ctl.lz;
  a.lzc = ctl;
  if (pw == P64 && plink == P64 && pt == P64) run<MODE_LZK, P64, P64, P64, P64, P64>(a, st);
  else if (pw == P32 && plink == P32 && pt == P32) run<MODE_LZK, P32, P32, P32, P32, P32>(a, st);
  else if (pw == P16 && plink == P16 && pt == P16) run<MODE_LZK, P16, P16, P16, P16, P16>(a, st);
  else if (pw == P64E && plink == P64E && pt == P64E) run_wilson_df(MODE_LZK, P64E, a, st);
  else OVL_BAD_COMBO();
}

void launch_wilson_lzL(int pt, int plink, int pw, const Geom& g, double kappa, LinkRef links, SpinorRef t,
                       SpinorRef W, int nrhs, double* partials, const LzCtl& ctl, cudaStream_t st) {
  DArgs a = base_args(g, kappa, links, nrhs);
  a.in = t;
  a.out = W;
  a.aux1 = W;
  a.partials = partials;
  a.lz = ctl.lz;
  a.lzc = ctl;
  if (pt == P64 && plink == P64 && pw == P64) run<MODE_LZL, P64, P64, P64, P64, P64>(a, st);
  else if (pt == P32 && plink == P32 && pw == P32) run<MODE_LZL, P32, P32, P32, P32, P32>(a, st);
  else if (pt == P16 && plink == P16 && pw == P16) run<MODE_LZL, P16, P16, P16, P16, P16>(a, st);
  else if (pt == P64E && plink == P64E && pw == P64E) run_wilson_df(MODE_LZL, P64E, a, st);
  else OVL_BAD_COMBO();
}

void launch_wilson_ovl(int py, int plink, int pv, const Geom& g, double kappa, LinkRef links, SpinorRef y,
                       SpinorRef v, SpinorRef out, SpinorRef w, int nrhs, double c1, double c2,
                       const double* coef, int herm, double* partials, cudaStream_t st) {
  DArgs a = base_args(g, kappa, links, nrhs);
  a.in = y;
  a.aux1 = v;
  a.out = out;
  a.aux2 = w;
  a.c1 = c1;
  a.c2 = c2;
  a.coef = coef;
  a.herm = herm;
  a.partials = partials;
  if (py == P64 && plink == P64 && pv == P64) run<MODE_OVL, P64, P64, P64, P64, P64>(a, st);
  else if (py == P32 && plink == P32 && pv == P32) run<MODE_OVL, P32, P32, P32, P32, P32>(a, st);
  else if (py == P32 && plink == P32 && pv == P64) run<MODE_OVL, P32, P32, P64, P64, P64>(a, st);
  else if (py == P32 && plink == P16 && pv == P32) run<MODE_OVL, P32, P16, P32, P32, P32>(a, st);
  else if (py == P32 && plink == P16 && pv == P64) run<MODE_OVL, P32, P16, P64, P64, P64>(a, st);
  else if (py == P64 && plink == P64 && pv == P32) run<MODE_OVL, P64, P64, P32, P32, P32>(a, st);
  else if (py == P64E && plink == P64E && pv == P64) run_wilson_df(MODE_OVL, P64, a, st);
  else if (py == P64E && plink == P64E && pv == P32) run_wilson_df(MODE_OVL, P32, a, st);
  else OVL_BAD_COMBO();
}

}  // namespace ovl
