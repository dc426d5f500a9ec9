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
  float kap_h, kap_l;   // kappa as hi + lo
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

// Programmatic dependent launch of the Lanczos steps: a launch whose predecessor's blocks have
// all started may take the SMs they leave free, compute its indices and fetch links, and waits
// (the hardware's wait for the complete predecessor, memory included) before it reads
// anything that a launch writes. Every thread of every block waits, so that a launch is complete
// only after its predecessor. Fields read after the wait are read by ordinary loads: the
// read-only path is for data that nothing writes while the kernel runs.
template <int MODE> constexpr bool kReadOnly = MODE != MODE_LZK && MODE != MODE_LZL;
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename K>
inline void launch_step(K kernel, dim3 grid, dim3 block, size_t smem, cudaStream_t st, const DArgs& a) {
  if (!a.lzc.pdl) {
    kernel<<<grid, block, smem, st>>>(a);
    return;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, a);
}

// ---- the scalar step of the stored-basis Lanczos, fused into its Wilson launches -------
// Every block writes the partial sum of each of its systems and counts itself in; the block that
// comes last for a system sums the partials in a fixed order (so that the result does not
// depend on which block that is) and updates the system's state. A row of the block
// (threadIdx.y) is one system, its first warp does this; the others leave. The step is a serial chain
// at the end of every launch, so it is kept to few dependent steps: the partials lie next to
// each other and each lane reads up to 32 at a time, the state is read while they are on their
// way, the sums are warp shuffles, and a pole's pivot costs one FP64 division (its reciprocal is
// kept). The coefficients the next launch multiplies by are rounded to double-float here, once
// per system: FP64 conversions run at 1/64 of the FP32 rate, and every thread of every launch
// made them.

__device__ __forceinline__ int lane_id() {
  int l;
  asm("mov.u32 %0, %%laneid;" : "=r"(l));
  return l;
}
// first partial sum of system rhs (16-byte aligned)
__device__ __forceinline__ double* lz_partials(const DArgs& a, int rhs) {
  return a.partials + (size_t)rhs * ((a.nsb + 1) & ~1);
}

__device__ __forceinline__ double lz_warp_sum(const double* base, int nsb) {
  const double2* b2 = reinterpret_cast<const double2*>(base);
  const int n2 = nsb >> 1, lane = lane_id();
  double t[4] = {0.0, 0.0, 0.0, 0.0};
  for (int p = lane; p < n2; p += 16 * 32) {
    double2 v[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u] = p + u * 32 < n2 ? __ldcg(b2 + p + u * 32) : make_double2(0.0, 0.0);
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (p - lane + u * 32 < n2) t[u & 3] += v[u].x + v[u].y;   // uniform: FP64 adds only where there are partials
  }
  if ((nsb & 1) && lane == 0) t[0] += __ldcg(base + nsb - 1);
  double r = (t[0] + t[1]) + (t[2] + t[3]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  return r;
}

// The first warp of a row, all lanes: the step of system rhs from its sum tot.
template <int MODE>
__device__ __forceinline__ void lz_step(const DArgs& a, int rhs, double tot, int j, double inv_n,
                                        double inv_nprev, double bp, double alpha) {
  LzRhs& L = a.lz[rhs];
  const int lane = lane_id();
  if constexpr (MODE == MODE_LZK) {
    if (lane != 0) return;
    a.lzc.ahist[(size_t)rhs * a.lzc.hcap + j] = tot;
    const double ca = tot * inv_n, cb = j > 0 ? bp * inv_nprev : 0.0;
    L.alpha = tot;
    L.a = ca;
    L.b = cb;
    L.fa = split_df(ca);
    L.fb = split_df(cb);
    if (!(tot > 0.0) || !isfinite(tot)) {
      L.done = 1;
      L.status = 2;   // K^2 is positive definite: breakdown
      L.finished = 1;
    }
  } else {
    const Poles* P = a.lzc.poles;
    const int np = P->n;
    const double beta = sqrt(tot), bp2 = bp * bp;
    double e = 0.0, m = 0.0, inv_beta = 0.0;
    for (int i0 = 0; i0 <= np; i0 += 32) {   // lane np of the poles takes 1 / beta
      const int i = i0 + lane;
      const bool pole = i < np;
      const double d = pole ? alpha + (P->sigma0 + P->ds[i]) - bp2 * L.rd[i] : beta;
      const double r = 1.0 / d;
      if (pole) {
        const double rho = L.rho[i] * (beta * r);
        L.rd[i] = r;
        L.rho[i] = rho;
        const double ei = fabs(L.w[i]) * P->gbound[i] * rho;
        e += ei;
        m = fmax(m, ei);
      } else if (i == np) {
        inv_beta = r;
      }
    }
    inv_beta = __shfl_sync(0xffffffffu, inv_beta, np & 31);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, o);
      m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    if (lane != 0) return;
    a.lzc.bhist[(size_t)rhs * a.lzc.hcap + j] = beta;
    L.err = e;
    const int total = L.total + 1;
    L.total = total;
    L.w_reads += (j > 0 ? 2 : 1);
    L.inv_nprev = inv_n;
    inv_beta = beta > 0.0 ? inv_beta : 0.0;
    L.inv_n = inv_beta;
    L.fn = split_df(inv_beta);
    L.beta_prev = beta;
    L.j = j + 1;
    if (!isfinite(beta) || !isfinite(e)) {
      L.done = 1;
      L.status = 2;
      L.finished = 1;
    } else if ((L.even ? m * np <= L.thr : e <= L.thr) || beta == 0.0) {
      // within budget, or an invariant subspace (the Galerkin solutions are exact)
      L.done = 1;
      L.status = 0;
      L.finished = 1;
    } else if (total >= L.maxit) {
      L.done = 1;
      L.status = 1;
      L.finished = 1;
    } else if (j + 2 > L.cap - 1) {
      L.done = 1;
      L.status = 3;   // W_{j+2} would not fit: restart from W_{j+1}
    }
  }
}

// After the block's partial sum of system rhs has been written (by lane 0 of this warp): count
// the block in, and run the step if it came last. nblk: blocks that write partials for one
// system. Called by the first warp of each row whose system is not done, all lanes (a system
// that is done is left alone by every block, its count included).
template <int MODE>
__device__ __forceinline__ void lz_arrive(const DArgs& a, int rhs, int nblk) {
  int last = 0;
  const int lane = lane_id();
  if (lane == 0) {
    __threadfence();   // the partial sum before the count
    last = atomicAdd(&a.lzc.ctr[rhs], 1u) == (unsigned)(nblk - 1) ? 1 : 0;
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return;
  __threadfence();
  const LzRhs& L = a.lz[rhs];
  const int j = L.j;
  const double inv_n = L.inv_n, inv_nprev = L.inv_nprev, bp = L.beta_prev, alpha = L.alpha;
  const double tot = lz_warp_sum(lz_partials(a, rhs), a.nsb);
  __syncwarp();   // every lane has read the state before lane 0 changes it
  lz_step<MODE>(a, rhs, tot, j, inv_n, inv_nprev, bp, alpha);
  if (lane == 0) a.lzc.ctr[rhs] = 0u;
}

// partial sums that a mode produces (the others are zero)
__host__ __device__ constexpr int nred(int mode) { return mode == MODE_OVL ? 4 : mode == MODE_K ? 2 : 1; }
// The Lanczos modes keep their one partial sum per block side by side (lz_partials).
template <int MODE>
__device__ __forceinline__ void store_partials(const DArgs& a, int rhs, int sb, const double tot[NVRED]) {
  if constexpr (MODE == MODE_LZK || MODE == MODE_LZL) {
    lz_partials(a, rhs)[sb] = tot[0];
  } else {
#pragma unroll
    for (int j = 0; j < NVRED; ++j) a.partials[((size_t)rhs * a.nsb + sb) * NVRED + j] = tot[j];
  }
}

// Block sum of the per-thread partials: warp stage in R (FP32 for the FP32 kernels),
// then FP64 across warps in a fixed order; the result is valid on thread (0, y).
template <typename R, int NV>
__device__ __forceinline__ void block_reduce_partials(R v[NVRED], double* smem, double out[NVRED]) {
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int nwarp = blockDim.x >> 5;
#pragma unroll
  for (int j = 0; j < NV; ++j) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[j] += __shfl_down_sync(0xffffffffu, v[j], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < NV; ++j) smem[(threadIdx.y * nwarp + warp) * NVRED + j] = (double)v[j];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < NVRED; ++j) {
      double t = 0.0;
      if (j < NV)
        for (int w = 0; w < nwarp; ++w) t += smem[(threadIdx.y * nwarp + w) * NVRED + j];
      out[j] = t;
    }
  }
}

// The double-float kernel (dfwilson.cu) in mode `mode`; pio: the storage of the vector operands of
// MODE_OVL (P64 or P32), P64E otherwise.
void run_wilson_df(int mode, int pio, DArgs a, cudaStream_t st);

}  // namespace ovl
