// Stored-basis Lanczos evaluation of the Zolotarev sum (Sec. 3):
//
//   y = sum_i omega_i (K^2 + sigma_i)^-1 v,   eps(K) v = K y.
//
// Every shifted system has the same Krylov space K_k(K^2, v), and its Galerkin (CG)
// solution after k steps is x_i = ||v|| V_k (T_k + sigma_i)^-1 e_1, with V_k the Lanczos
// basis and T_k the tridiagonal matrix of the recurrence. The multi-shift CG of mscg.cu
// carries one search direction per pole and updates all of them every step (two spinor
// passes per active pole and step); here the basis itself is kept in HBM instead, one
// vector per step, so that a step is two Wilson launches (their last blocks do the
// scalar work), and y comes at the end from N_Z tridiagonal solves (scalars) and a single
// pass over the stored vectors.
//
// Per step j (lz[rhs].j = j, unnormalised vectors W_l with v_l = W_l / n_l), two Wilson
// launches whose last block per system also runs the scalar step (wilson.cuh, lz_step):
//   MODE_LZK   t = K v_j;  alpha_j = ||t||^2,  a = alpha_j / n_j,  b = beta_{j-1} / n_{j-1}
//   MODE_LZL   W_{j+1} = K t - a W_j - b W_{j-1};  beta_j = ||W_{j+1}|| = n_{j+1}, for every
//              pole the LDL^T pivot d_j = alpha_j + sigma_i - beta_{j-1}^2 / d_{j-1} and the
//              residual norm rho_i <- rho_i beta_j / d_j of its Galerkin solution
//              (||r_i|| = ||v|| prod_l beta_l / d_l), the error bound sum_i |w_i| g_i rho_i
//              and the stopping test.
// The stopping rule is the one of the multi-shift CG (pole i contributes at most
// |w_i| g_i ||r_i|| to the error of eps(K) v, g_i = max_[a,b] x / (x^2 + sigma_i)); all
// poles keep improving until the sum is within eta ||v||.
//
// A cycle holds at most cap vectors. When it fills up, every pole's residual is
// r_i = -||v|| (T_k + sigma_i)^-1_{k-1,0} W_k, parallel to the last vector, so the rest
// of the sum is the same problem started from W_k with weights w_i ||v|| (-y_i,k-1): the
// cycle's part of y is added and the next cycle starts there.
#include "dfpair.cuh"
#include "kernels.h"

namespace ovl {

// Fixed-order sum over the site-block partials (slot 0) of one system.
__device__ __forceinline__ double lz_sum_partials(const double* partials, int nsb, int rhs) {
  __shared__ double sh[128];
  double a = 0.0;
  for (int b = threadIdx.x; b < nsb; b += blockDim.x) a += partials[((size_t)rhs * nsb + b) * NVRED];
  sh[threadIdx.x] = a;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  const double r = sh[0];
  __syncthreads();
  return r;
}

// ---------------------------------------------------------------- init / restart
template <int PV, int PW, int PY>
__global__ void __launch_bounds__(256) lz_init_kernel(SpinorRef v, SpinorRef W, SpinorRef y, int nrhs, int V,
                                                      int nsb, int ngr, double* partials) {
  using T = typename Real<PW>::T;
  __shared__ double red[4 * (BX / 32) * 2];
  const int sb = blockIdx.x / ngr;
  const int rg = blockIdx.x - sb * ngr;
  const int rhs = rg * blockDim.y + threadIdx.y;
  const int s = sb * BX + threadIdx.x;
  double acc[2] = {0.0, 0.0};
  if (s < V && rhs < nrhs) {
    cpx<T> a[12];
    load_spinor_as<PV, T>(v, rhs, s, a);
    store_spinor_as<PW, T>(W, rhs, s, a);
    // the norm of the stored (rounded) start vector, which the recurrence sees
    load_spinor_as<PW, T>(W, rhs, s, a);
    cpx<double> z[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      acc[0] += to_d(a[k].r) * to_d(a[k].r) + to_d(a[k].i) * to_d(a[k].i);
      z[k] = cmk(0.0, 0.0);
    }
    store_spinor_any<PY>(y, rhs, s, z);
  }
  block_reduce_rows<2>(acc, red);
  if (threadIdx.x == 0 && rhs < nrhs) {
    partials[((size_t)rhs * nsb + sb) * NVRED + 0] = acc[0];
    partials[((size_t)rhs * nsb + sb) * NVRED + 1] = 0.0;
  }
}

// Double-float: one thread per pair of sites and system.
constexpr int DP = 32;   // pairs per block: the partial sums keep the 64-site blocks
template <int PV>
__global__ void __launch_bounds__(128) lz_init_df_kernel(SpinorRef v, SpinorRef W, SpinorRef y, int nrhs, int Vh,
                                                         int nsb, int ngr, double* partials) {
  const int sb = blockIdx.x / ngr;
  const int rhs = (blockIdx.x - sb * ngr) * blockDim.y + threadIdx.y;
  const int i = sb * DP + threadIdx.x;
  dot2p d = {0ull, 0ull};
  if (i < Vh && rhs < nrhs) {
#pragma unroll 4
    for (int k = 0; k < 12; ++k) {
      dd2 re, im;
      dfp_load<PV>(v, rhs, k, i, re, im);
      dfp_store<P64E>(W, rhs, k, i, re, im);
      dfp_store<P64E>(y, rhs, k, i, dd2_zero(), dd2_zero());
      dot2p_add(d, re, re);
      dot2p_add(d, im, im);
    }
  }
  double s = dot2p_get(d);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (threadIdx.x == 0 && rhs < nrhs) {
    partials[((size_t)rhs * nsb + sb) * NVRED + 0] = s;
    partials[((size_t)rhs * nsb + sb) * NVRED + 1] = 0.0;
  }
}

void launch_lz_init(int pv, int pw, int py, SpinorRef v, SpinorRef W, SpinorRef y, int nrhs, int V,
                    double* partials, cudaStream_t st) {
  Shape sh = make_shape(V, nrhs);
#define LZI(A, B, C) lz_init_kernel<A, B, C><<<sh.grid(), sh.block(), 0, st>>>(v, W, y, nrhs, V, sh.nsb, sh.ngr, partials)
  if (pv == P64 && pw == P64 && py == P64) LZI(P64, P64, P64);
  else if (pw == P64E && py == P64E && (pv == P64 || pv == P32)) {
    const dim3 block(DP, sh.by), grid(sh.grid());
    if (pv == P64) lz_init_df_kernel<P64><<<grid, block, 0, st>>>(v, W, y, nrhs, V / 2, sh.nsb, sh.ngr, partials);
    else lz_init_df_kernel<P32><<<grid, block, 0, st>>>(v, W, y, nrhs, V / 2, sh.nsb, sh.ngr, partials);
  }
  else if (pv == P64 && pw == P32 && py == P32) LZI(P64, P32, P32);
  else if (pv == P32 && pw == P32 && py == P32) LZI(P32, P32, P32);
  else if (pv == P64 && pw == P16 && py == P32) LZI(P64, P16, P32);
  else if (pv == P32 && pw == P16 && py == P32) LZI(P32, P16, P32);
  else if (pv == P32 && pw == P64 && py == P64) LZI(P32, P64, P64);
  else note_bad_combo("lz_init");
#undef LZI
}

// W_0 = W_j for the systems whose cycle filled up (status 3); partials of ||W_0||^2.
template <int PW>
__global__ void __launch_bounds__(256) lz_restart_kernel(SpinorRef W, const LzRhs* lz, int nrhs, int V, int nsb,
                                                         int ngr, double* partials) {
  using T = typename Real<PW>::T;
  __shared__ double red[4 * (BX / 32) * 2];
  const int sb = blockIdx.x / ngr;
  const int rg = blockIdx.x - sb * ngr;
  const int rhs = rg * blockDim.y + threadIdx.y;
  const int s = sb * BX + threadIdx.x;
  double acc[2] = {0.0, 0.0};
  if (s < V && rhs < nrhs && !lz[rhs].finished && lz[rhs].status == 3) {
    cpx<T> a[12];
    load_spinor_as<PW, T>(W, lz[rhs].j * nrhs + rhs, s, a);
    store_spinor_as<PW, T>(W, rhs, s, a);
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[0] += to_d(a[k].r) * to_d(a[k].r) + to_d(a[k].i) * to_d(a[k].i);
  }
  block_reduce_rows<2>(acc, red);
  if (threadIdx.x == 0 && rhs < nrhs) {
    partials[((size_t)rhs * nsb + sb) * NVRED + 0] = acc[0];
    partials[((size_t)rhs * nsb + sb) * NVRED + 1] = 0.0;
  }
}

void launch_lz_restart(int pw, SpinorRef W, const LzRhs* lz, int nrhs, int V, double* partials, cudaStream_t st) {
  Shape sh = make_shape(V, nrhs);
  if (pw == P64) lz_restart_kernel<P64><<<sh.grid(), sh.block(), 0, st>>>(W, lz, nrhs, V, sh.nsb, sh.ngr, partials);
  else if (pw == P64E) lz_restart_kernel<P64E><<<sh.grid(), sh.block(), 0, st>>>(W, lz, nrhs, V, sh.nsb, sh.ngr, partials);
  else if (pw == P32) lz_restart_kernel<P32><<<sh.grid(), sh.block(), 0, st>>>(W, lz, nrhs, V, sh.nsb, sh.ngr, partials);
  else lz_restart_kernel<P16><<<sh.grid(), sh.block(), 0, st>>>(W, lz, nrhs, V, sh.nsb, sh.ngr, partials);
}

// ---------------------------------------------------------------- scalars
// Start a cycle: n_0 = ||W_0||. First cycle: weights omega_i and the budget eta ||v||
// (|eta|: the sign of eta selects the multi-shift CG's rule and does not matter here).
// Later cycles keep the weights set by lz_coef and the budget.
__global__ void lz_start_kernel(LzRhs* lz, const double* partials, int nsb, const Poles* P, const double* eta,
                                int maxit, int cap, int first) {
  const int rhs = blockIdx.x;
  LzRhs& L = lz[rhs];
  const double nn = lz_sum_partials(partials, nsb, rhs);
  if (!first && (L.finished || L.status != 3)) {
    // done in an earlier cycle, whose part is in y: nothing of it is combined again
    if (threadIdx.x == 0) L.j = 0;
    return;
  }
  const double n0 = sqrt(nn);
  for (int i = threadIdx.x; i < P->n; i += blockDim.x) {
    if (first) L.w[i] = P->omega[i];
    L.rd[i] = 0.0;
    L.rho[i] = n0;
  }
  if (threadIdx.x == 0) {
    if (first) {
      L.thr = fabs(eta[rhs]) * n0;
      L.even = eta[rhs] < 0.0 ? 1 : 0;
      L.total = 0;
      L.maxit = maxit;
      L.cycles = 0;
      L.finished = 0;
      L.w_reads = 0;
    }
    L.cap = cap;
    L.vnorm = n0;
    L.inv_n = n0 > 0.0 ? 1.0 / n0 : 0.0;
    L.inv_nprev = 0.0;
    L.fn = split_df(L.inv_n);
    L.fa = L.fb = make_float2(0.f, 0.f);
    L.a = L.b = L.alpha = L.beta_prev = 0.0;
    L.err = 0.0;
    L.j = 0;
    L.status = 0;
    L.cycles += 1;
    // nothing left to do: a zero vector (or, on a restart, a remainder already within budget)
    L.done = (n0 == 0.0) ? 1 : 0;
    if (L.done) L.finished = 1;
  }
}

void launch_lz_start(LzRhs* lz, const double* partials, int nsb, int nrhs, const Poles* poles, const double* eta,
                     int maxit, int cap, int first, cudaStream_t st) {
  lz_start_kernel<<<nrhs, 128, 0, st>>>(lz, partials, nsb, poles, eta, maxit, cap, first);
}
// ---------------------------------------------------------------- coefficients
// One block per system. Thread i (pole) solves (T_k + sigma_i) y_i = e_1 by the LDL^T
// factorisation of T_k + sigma_i (pivots d_l; L unit lower bidiagonal with l_l =
// beta_l / d_l): forward z_0 = 1, z_l = -(beta_{l-1} / d_{l-1}) z_{l-1}; back
// y_{k-1} = z_{k-1} / d_{k-1}, y_l = z_l / d_l - (beta_l / d_l) y_{l+1}. Y holds 2 cap
// doubles per pole and system (y, then the reciprocal pivots). Then coefW_l = n_0 sum_i w_i y_il / n_l
// is the coefficient of the stored W_l in y. A cycle that filled up passes its remainder
// on: w_i <- w_i n_0 (-y_i,k-1).
// A serial chain per pole, so what counts is its latency: one FP64 division per step (160 ns; a
// multiply-add 31) with the reciprocal kept, T in shared memory, and the backward pass' loads
// eight at a time ahead of its chain. 115 steps, 20 poles: 180 -> 60 us.
// gave_up (may be null): set when the one-launch form of the cycle gave up, of which nothing is used.
__global__ void lz_coef_kernel(LzRhs* lz, const double* ahist, const double* bhist, int cap, const Poles* P,
                               double* Y, double* coefW, const unsigned int* gave_up) {
  extern __shared__ double tri[];   // alpha, beta: cap each
  const int rhs = blockIdx.x;
  LzRhs& L = lz[rhs];
  if (gave_up != nullptr && *gave_up != 0u) {
    if (threadIdx.x == 0) L.j = 0;   // no vectors to combine
    return;
  }
  const int k = L.j;
  const int np = P->n;
  double *al = tri, *be = tri + cap;
  for (int l = threadIdx.x; l < k; l += blockDim.x) {
    al[l] = ahist[(size_t)rhs * cap + l];
    be[l] = bhist[(size_t)rhs * cap + l];
  }
  __syncthreads();
  double* Yr = Y + (size_t)rhs * np * 2 * cap;
  double* cw = coefW + (size_t)rhs * cap;
  const bool active = k > 0 && L.status != 2;
  for (int i = threadIdx.x; i < np && active; i += blockDim.x) {
    const double sg = P->sigma0 + P->ds[i];
    const double wi = L.w[i];
    double* y = Yr + (size_t)i * 2 * cap;
    double* r = y + cap;
    // forward: y_l <- w_i z_l / d_l
    double rl = 1.0 / (al[0] + sg), z = 1.0, last = rl;
    r[0] = rl;
    y[0] = wi * rl;
    for (int l = 1; l < k; ++l) {
      const double b = be[l - 1];
      z *= -(b * rl);
      rl = 1.0 / (al[l] + sg - b * b * rl);
      r[l] = rl;
      last = z * rl;
      y[l] = wi * last;
    }
    if (L.status == 3) L.w[i] = wi * L.vnorm * (-last);
    // backward, y_{l+1} in v
    double v = wi * last;
    for (int l0 = k - 2; l0 >= 0; l0 -= 8) {
      double yy[8], rr[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (l0 - u >= 0) {
          yy[u] = y[l0 - u];
          rr[u] = r[l0 - u];
        }
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (l0 - u >= 0) {
          v = yy[u] - (be[l0 - u] * rr[u]) * v;
          y[l0 - u] = v;
        }
    }
  }
  __syncthreads();
  for (int l = threadIdx.x; l < cap; l += blockDim.x) {
    double c = 0.0;
    if (active && l < k) {
#pragma unroll 8
      for (int i = 0; i < np; ++i) c += Yr[(size_t)i * 2 * cap + l];
      const double nl = l == 0 ? L.vnorm : be[l - 1];
      c = nl > 0.0 ? L.vnorm * c / nl : 0.0;
    }
    cw[l] = c;
  }
}

void launch_lz_coef(LzRhs* lz, const double* ahist, const double* bhist, int cap, const Poles* poles, double* Y,
                    double* coefW, const unsigned int* gave_up, int nrhs, cudaStream_t st) {
  lz_coef_kernel<<<nrhs, 128, 2 * sizeof(double) * (size_t)cap, st>>>(lz, ahist, bhist, cap, poles, Y, coefW, gave_up);
}

// ---------------------------------------------------------------- combine
// y += sum_{l < k} coefW_l W_l. Double-float: one thread per 16-byte chunk (one real number of
// a pair of sites), every stored vector's chunk read once, eight loads in flight; coefficients
// converted to double-float once per block in shared memory. Bound by HBM on large batches;
// the chunk as a grid dimension keeps a small lattice from running 24 chunks in series.
__global__ void __launch_bounds__(128) lz_combine_df_kernel(SpinorRef W, SpinorRef y, const double* coefW,
                                                            const LzRhs* lz, int cap, int nrhs, int Vh, int nb) {
  extern __shared__ f2 cf[];   // per stored vector: high word, its negative, low word (both lanes)
  const int rhs = blockIdx.y;
  const int k = lz[rhs].j;
  for (int l = threadIdx.x; l < k; l += blockDim.x) {
    const fac2 c = fac2_bc(coefW[(size_t)rhs * cap + l]);
    cf[3 * l] = c.h;
    cf[3 * l + 1] = c.n;
    cf[3 * l + 2] = c.l;
  }
  __syncthreads();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;   // chunk of the field
  if (e / 768 * 32 + (e & 31) >= Vh || k == 0) return;
  const size_t at = (size_t)rhs * nb * 768 + e;
  const size_t slot = (size_t)nrhs * nb * 768;
  dd2 acc = dfp_ld(y, at);
  int l = 0;
  for (; l + 8 <= k; l += 8) {
    dd2 w[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) w[u] = dfp_ldg(W, at + (size_t)(l + u) * slot);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const f2* c = cf + 3 * (l + u);
      acc = dd2_add(acc, dd2_mul({c[0], c[1], c[2]}, w[u]));
    }
  }
  for (; l < k; ++l) {
    const f2* c = cf + 3 * l;
    acc = dd2_add(acc, dd2_mul({c[0], c[1], c[2]}, dfp_ldg(W, at + (size_t)l * slot)));
  }
  dfp_st(y, at, acc);
}

// FP32 and FP64: the same, one thread per 16-byte chunk, which is contiguous over the whole field
// (the spinor-at-a-time form below loaded one stored vector after the other: on a small lattice a
// chain of one load latency per vector). FP32 sign on 10 x 6 x 14 x 12 588 -> 572 us, solve on
// 16^3 x 32 287 -> 284 ms.
__device__ __forceinline__ void axpy_word(float4& y, float c, const float4& w) {
  y.x += c * w.x;
  y.y += c * w.y;
  y.z += c * w.z;
  y.w += c * w.w;
}
__device__ __forceinline__ void axpy_word(double2& y, double c, const double2& w) {
  y.x += c * w.x;
  y.y += c * w.y;
}
template <typename W4, typename T>
__global__ void __launch_bounds__(128) lz_combine_words_kernel(const W4* W, W4* y, const double* coefW, const LzRhs* lz,
                                                               int cap, int nrhs, int words) {
  extern __shared__ double cfd[];
  T* cf = reinterpret_cast<T*>(cfd);
  const int rhs = blockIdx.y;
  const int k = lz[rhs].j;
  if (k == 0) return;
  for (int l = threadIdx.x; l < k; l += blockDim.x) cf[l] = (T)coefW[(size_t)rhs * cap + l];
  __syncthreads();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= words) return;
  const size_t slot = (size_t)nrhs * words;
  const W4* p = W + (size_t)rhs * words + e;
  W4* q = y + (size_t)rhs * words + e;
  W4 acc = *q;
  int l = 0;
  for (; l + 8 <= k; l += 8) {
    W4 w[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) w[u] = __ldcs(p + (size_t)(l + u) * slot);
#pragma unroll
    for (int u = 0; u < 8; ++u) axpy_word(acc, cf[l + u], w[u]);
  }
  for (; l < k; ++l) axpy_word(acc, cf[l], __ldcs(p + (size_t)l * slot));
  *q = acc;
}

// FP16 storage (a scale per site): whole spinors, accumulated in the compute type of y.
template <int PW, int PY>
__global__ void __launch_bounds__(256) lz_combine_kernel(SpinorRef W, SpinorRef y, const double* coefW,
                                                         const LzRhs* lz, int cap, int nrhs, int V, int ngr) {
  using T = typename Real<PY>::T;
  const int sb = blockIdx.x / ngr;
  const int rg = blockIdx.x - sb * ngr;
  const int rhs = rg * blockDim.y + threadIdx.y;
  const int s = sb * BX + threadIdx.x;
  if (s >= V || rhs >= nrhs) return;
  const int k = lz[rhs].j;
  if (k == 0) return;
  cpx<T> acc[12], w[12];
  load_spinor_as<PY, T>(y, rhs, s, acc);
  for (int l = 0; l < k; ++l) {
    load_spinor_as<PW, T>(W, l * nrhs + rhs, s, w);
    const T cl = (T)coefW[(size_t)rhs * cap + l];
#pragma unroll
    for (int q = 0; q < 12; ++q) acc[q] = acc[q] + cl * w[q];
  }
  store_spinor_as<PY, T>(y, rhs, s, acc);
}

void launch_lz_combine(int pw, int py, SpinorRef W, SpinorRef y, const double* coefW, const LzRhs* lz, int cap,
                       int nrhs, int V, cudaStream_t st) {
  Shape sh = make_shape(V, nrhs);
  if (pw == P64E && py == P64E) {
    const size_t smem = 3 * sizeof(f2) * (size_t)cap;   // cap <= 1024: 24 KB
    lz_combine_df_kernel<<<dim3(df_blocks(V) * 6, nrhs), 128, smem, st>>>(W, y, coefW, lz, cap, nrhs, V / 2, df_blocks(V));
    return;
  }
  const size_t smem = sizeof(double) * (size_t)cap;
  if (pw == P64 && py == P64) {
    lz_combine_words_kernel<double2, double><<<dim3((12 * V + 127) / 128, nrhs), 128, smem, st>>>(
        static_cast<const double2*>(W.data), static_cast<double2*>(y.data), coefW, lz, cap, nrhs, 12 * V);
  } else if (pw == P32 && py == P32) {
    lz_combine_words_kernel<float4, float><<<dim3((6 * V + 127) / 128, nrhs), 128, smem, st>>>(
        static_cast<const float4*>(W.data), static_cast<float4*>(y.data), coefW, lz, cap, nrhs, 6 * V);
  } else if (pw == P16 && py == P32) {
    lz_combine_kernel<P16, P32><<<sh.grid(), sh.block(), 0, st>>>(W, y, coefW, lz, cap, nrhs, V, sh.ngr);
  } else {
    note_bad_combo("lz_combine");
  }
}

}  // namespace ovl
