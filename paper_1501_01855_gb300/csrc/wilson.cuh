// What the Wilson kernels of every precision share (dslash.cu: FP64, FP32, FP16 storage;
// dfwilson.cu: double-float): launch arguments, the block sums of the epilogues' partial
// sums, and the scalar step of the stored-basis Lanczos that the last block of a launch runs.
#pragma once
#include "kernels.h"

namespace ovl {

enum { MODE_K = 0, MODE_R = 1, MODE_OVL = 2, MODE_LZK = 3, MODE_LZL = 4 };

// Per-thread sums of the epilogue reductions are kept in the compute type (RedT).
template <typename T> struct RedT { using type = double; };
template <> struct RedT<float> { using type = float; };

struct DArgs {
  Geom g;
  double kappa;
  LinkRef links;
  SpinorRef in, out, aux1, aux2;
  int nrhs, nsb, ngr;
  double* partials;
  const MsRhs* ms;
  double sigma0;
  double c1, c2;
  const double* coef;
  int herm;
  int variant;   // launch shape (see LinkRef)
  LzRhs* lz;
  LzCtl lzc;
};

// threads that take part in a block's scalar step (the first 256 of the block)
__device__ __forceinline__ int lz_tid() { return (threadIdx.z * blockDim.y + threadIdx.y) * blockDim.x + threadIdx.x; }
__device__ __forceinline__ int lz_threads() { return min(256, (int)(blockDim.x * blockDim.y * blockDim.z)); }

// ---- the scalar step of the stored-basis Lanczos, fused into its Wilson launches -------
// Called by the whole block for a system whose last partial sum this block wrote. The
// sum over the site-block partials runs in a fixed order (thread-strided, then a fixed
// tree), so the result does not depend on which block came last.
__device__ __forceinline__ double lz_block_sum(const double* partials, int nsb, int rhs, double* sm) {
  const int tid = lz_tid(), nt = lz_threads();
  // eight loads in flight per thread (a block of 64 threads sums 2048 partials of a 16^3 x 32
  // lattice: one dependent L2 load after another would hold the launch for microseconds);
  // the eight running sums are combined in a fixed order
  const double* base = partials + (size_t)rhs * nsb * NVRED;
  double acc8[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  int b = tid < nt ? tid : nsb;
  for (; b + 7 * nt < nsb; b += 8 * nt) {
#pragma unroll
    for (int u = 0; u < 8; ++u) acc8[u] += __ldcg(base + (size_t)(b + u * nt) * NVRED);
  }
  for (int u = 0; b < nsb; b += nt, ++u) acc8[u & 7] += __ldcg(base + (size_t)b * NVRED);
  const double v = ((acc8[0] + acc8[1]) + (acc8[2] + acc8[3])) + ((acc8[4] + acc8[5]) + (acc8[6] + acc8[7]));
  if (tid < nt) sm[tid] = v;
  for (int i = nt + tid; i < 256; i += nt) sm[i] = 0.0;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (tid < o) sm[tid] += sm[tid + o];
    __syncthreads();
  }
  const double r = sm[0];
  __syncthreads();
  return r;
}

template <int MODE>
__device__ void lz_finish(const DArgs& a, int rhs) {
  __shared__ double sm[256], em[256];
  const int tid = lz_tid(), nt = lz_threads();
  LzRhs& L = a.lz[rhs];
  const bool skip = L.done != 0;   // read by every thread before any write below
  __syncthreads();
  if (!skip) {
    const double tot = lz_block_sum(a.partials, a.nsb, rhs, sm);
    if constexpr (MODE == MODE_LZK) {
      if (tid == 0) {
        a.lzc.ahist[(size_t)rhs * a.lzc.hcap + L.j] = tot;
        L.alpha = tot;
        L.a = tot * L.inv_n;
        L.b = L.j > 0 ? L.beta_prev * L.inv_nprev : 0.0;
        if (!(tot > 0.0) || !isfinite(tot)) {
          L.done = 1;
          L.status = 2;   // K^2 is positive definite: breakdown
          L.finished = 1;
        }
      }
    } else {
      const Poles* P = a.lzc.poles;
      const double beta = sqrt(tot);
      const int j = L.j;
      const double alpha = L.alpha, bp = L.beta_prev;
      double e = 0.0, m = 0.0;
      for (int i = tid < nt ? tid : P->n; i < P->n; i += nt) {
        const double sg = P->sigma0 + P->ds[i];
        const double d = alpha + sg - (j > 0 ? bp * bp / L.d[i] : 0.0);
        L.d[i] = d;
        L.rho[i] *= beta / d;
        const double ei = fabs(L.w[i]) * P->gbound[i] * L.rho[i];
        e += ei;
        m = fmax(m, ei);
      }
      if (tid < nt) {
        sm[tid] = e;
        em[tid] = m;
      }
      for (int i = nt + tid; i < 256; i += nt) sm[i] = em[i] = 0.0;
      __syncthreads();
      for (int o = 128; o > 0; o >>= 1) {
        if (tid < o) {
          sm[tid] += sm[tid + o];
          em[tid] = fmax(em[tid], em[tid + o]);
        }
        __syncthreads();
      }
      if (tid == 0) {
        a.lzc.bhist[(size_t)rhs * a.lzc.hcap + j] = beta;
        L.err = sm[0];
        L.total += 1;
        L.w_reads += (j > 0 ? 2 : 1);
        L.inv_nprev = L.inv_n;
        L.inv_n = beta > 0.0 ? 1.0 / beta : 0.0;
        L.beta_prev = beta;
        L.j = j + 1;
        if (!isfinite(beta) || !isfinite(sm[0])) {
          L.done = 1;
          L.status = 2;
          L.finished = 1;
        } else if ((L.even ? em[0] * P->n <= L.thr : sm[0] <= L.thr) || beta == 0.0) {
          // within budget, or an invariant subspace (the Galerkin solutions are exact)
          L.done = 1;
          L.status = 0;
          L.finished = 1;
        } else if (L.total >= L.maxit) {
          L.done = 1;
          L.status = 1;
          L.finished = 1;
        } else if (L.j + 1 > L.cap - 1) {
          L.done = 1;
          L.status = 3;   // W_{j+2} would not fit: restart from W_{j+1}
        }
      }
    }
  }
  if (tid == 0) a.lzc.ctr[rhs] = 0u;
  __syncthreads();
}

// After the block's partial sums are written (by thread x = 0 of each row y, for system
// rhs_y): count the block in, and finish every system for which it came last. nblk: blocks
// that write partials for one system. Every thread of the block calls this.
template <int MODE>
__device__ __forceinline__ void lz_arrive(const DArgs& a, int rhs_row, int nblk) {
  __shared__ int last[8], rows[8];
  if (threadIdx.x == 0 && threadIdx.z == 0) {
    int f = 0;
    if (rhs_row < a.nrhs) {
      __threadfence();   // this row's partial sum before the count
      f = atomicAdd(&a.lzc.ctr[rhs_row], 1u) == (unsigned)(nblk - 1) ? 1 : 0;
    }
    last[threadIdx.y] = f;
    rows[threadIdx.y] = rhs_row;
  }
  __syncthreads();
  for (int y = 0; y < (int)blockDim.y; ++y) {
    if (last[y]) {   // shared, so the same for every thread of the block
      __threadfence();
      lz_finish<MODE>(a, rows[y]);
    }
  }
}

// Block sum of the per-thread partials: warp stage in R (FP32 for the FP32 kernels),
// then FP64 across warps in a fixed order; the result is valid on thread (0, y).
template <typename R>
__device__ __forceinline__ void block_reduce_partials(R v[NVRED], double* smem, double out[NVRED]) {
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int nwarp = blockDim.x >> 5;
#pragma unroll
  for (int j = 0; j < NVRED; ++j) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[j] += __shfl_down_sync(0xffffffffu, v[j], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < NVRED; ++j) smem[(threadIdx.y * nwarp + warp) * NVRED + j] = (double)v[j];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < NVRED; ++j) {
      double t = 0.0;
      for (int w = 0; w < nwarp; ++w) t += smem[(threadIdx.y * nwarp + w) * NVRED + j];
      out[j] = t;
    }
  }
}

// The double-float kernel (dfwilson.cu) in mode `mode`; pio: the storage of the vector operands of
// MODE_OVL (P64 or P32), P64E otherwise.
void run_wilson_df(int mode, int pio, DArgs a, cudaStream_t st);

}  // namespace ovl
