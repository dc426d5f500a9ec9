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

// ---- the Lanczos iteration as one cooperative launch ------------------------------------
// With few sites a step of two launches is latency: dispatch, the chain from the last block's
// partial sum to the next launch's coefficient (4 to 9 us), cold instruction caches. Here the
// blocks stay: each phase (K: t = K v_j, L: W_{j+1}) ends in a barrier of the grid instead of a
// launch, every block has one more warp that sums the blocks' partials of the phase before and
// forms the coefficients while the others are still in the hop sum (they meet before the
// epilogue), and block s also runs the poles' recurrence and the stopping test of system s, whose
// result is read one phase later. The arithmetic of a step is that of lz_step.
struct LzPersist {
  DArgs a, l;          // of the K phases (in W, out t) and of the L phases (in t, out and aux1 W)
  SpinorRef W, t;
  double* part;        // [phase][system][block]
  unsigned int* bar;   // arrivals, error, stop flags set in K phases, in L phases (each read in the other)
  int tb, ntile;       // tiles a block holds at a time, tiles of the launch
  unsigned long long wait_ns;   // limit of a barrier's wait
};
struct LzCoef {        // what the epilogues take from LzRhs
  float2 fn, fa, fb;
  int j, done;
};
constexpr int LZP_WARPS = 28;   // of a block, at most
struct LzpShared {
  LzCoef c[LZP_SYS];
  double acc[LZP_WARPS][LZP_SYS];   // partial sums of this phase by warp and system
  int ok;
};

__device__ __forceinline__ unsigned int lzp_acquire(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// One lane of the block: arrive and wait for the k-th barrier of the grid. The wait ends after
// the limit (zero: at once), or when another block has given up; the launch then ends everywhere.
__device__ __forceinline__ int lzp_barrier(unsigned int* bar, unsigned int target, unsigned long long limit) {
  if (limit == 0) {
    atomicExch(bar + 1, 1u);
    return 0;
  }
  __threadfence();
  atomicAdd(bar, 1u);
  unsigned long long t0 = 0;
  for (int k = 0;; ++k) {
    if (lzp_acquire(bar) >= target) return 1;
    if ((k & 255) == 255) {
      unsigned long long t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (t0 == 0) t0 = t;
      if (lzp_acquire(bar + 1) != 0u) return 0;
      if (t - t0 > limit) {
        atomicExch(bar + 1, 1u);
        return 0;
      }
    }
  }
}

// The last warp of a block, lanes split among the systems.
struct LzpScalar {
  int n, lps, sys, sl, grid;
  bool act;
  int done;
  double inv_n, inv_nprev, bp, bpp, alpha;   // 1 / n_j, 1 / n_{j-1}, beta_{j-1}, beta_{j-2}, alpha
  // the designated block of a system: two poles per lane
  int ds;
  double rd[2], rho[2], w[2], gb[2], sg[2];
  __device__ __forceinline__ void init(const LzPersist& p) {
    const int lane = lane_id();
    n = p.a.nrhs;
    lps = n == 1 ? 32 : n == 2 ? 16 : 8;
    sys = lane / lps;
    sl = lane - sys * lps;
    act = sys < n;
    grid = gridDim.x;
    const LzRhs& L = p.a.lzc.lz[act ? sys : 0];
    done = L.done;
    inv_n = L.inv_n;
    inv_nprev = bp = bpp = alpha = 0.0;
    ds = (int)blockIdx.x < n ? blockIdx.x : -1;
    if (ds >= 0) {
      const LzRhs& D = p.a.lzc.lz[ds];
      const Poles* P = p.a.lzc.poles;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int i = lane + 32 * k;
        const bool pole = i < P->n;
        rd[k] = 0.0;
        rho[k] = pole ? D.rho[i] : 0.0;
        w[k] = pole ? fabs(D.w[i]) : 0.0;
        gb[k] = pole ? P->gbound[i] : 0.0;
        sg[k] = pole ? P->sigma0 + P->ds[i] : 1.0;
      }
    }
  }
  __device__ __forceinline__ double total(const LzPersist& p, int phase) const {
    const double* b = p.part + (size_t)(phase * n + (act ? sys : 0)) * LZP_BLOCKS;
    double s = 0.0;
    for (int k = sl; k < grid; k += 8 * lps) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = k + u * lps < grid ? __ldcg(b + k + u * lps) : 0.0;
      s += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
    for (int o = lps >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  }
  // coefficients of the epilogue of phase K (0) or L (1) of step j
  __device__ __forceinline__ void coefficients(const LzPersist& p, int phase, int j, LzpShared& sh) {
    if (j > 0 || phase == 1) done |= (int)__ldcg(p.bar + 2 + (1 - phase) * LZP_SYS + (act ? sys : 0));
    if (phase == 0) {
      if (j > 0) {
        bpp = bp;
        bp = sqrt(total(p, 1));
        inv_nprev = inv_n;
        inv_n = bp > 0.0 ? 1.0 / bp : 0.0;
      }
      if (act && sl == 0) sh.c[sys].fn = split_df(inv_n);
    } else {
      alpha = total(p, 0);
      if (act && sl == 0) {
        sh.c[sys].fa = split_df(alpha * inv_n);
        sh.c[sys].fb = split_df(j > 0 ? bp * inv_nprev : 0.0);
      }
    }
    if (act && sl == 0) {
      sh.c[sys].j = j;
      sh.c[sys].done = done;
    }
  }
  // the designated block: alpha_j, or step j - 1 (its beta is bp), into the system's state
  __device__ __forceinline__ void record(const LzPersist& p, int phase, int j) {
    if (ds < 0) return;
    const int lane = lane_id(), from = ds * lps;
    const double al = __shfl_sync(0xffffffffu, alpha, from);
    const double be = __shfl_sync(0xffffffffu, bp, from), bpv = __shfl_sync(0xffffffffu, bpp, from);
    if (__shfl_sync(0xffffffffu, done, from)) return;
    LzRhs& L = p.a.lzc.lz[ds];
    const size_t row = (size_t)ds * p.a.lzc.hcap;
    if (phase == 1) {
      if (lane == 0) {
        p.a.lzc.ahist[row + j] = al;
        if (!(al > 0.0) || !isfinite(al)) {
          L.j = j;
          L.done = 1;
          L.status = 2;   // K^2 is positive definite: breakdown
          L.finished = 1;
          __stcg(p.bar + 2 + LZP_SYS + ds, 1u);
        }
      }
      return;
    }
    if (j == 0) return;
    double e = 0.0, m = 0.0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (k == 1 && p.a.lzc.poles->n <= 32) break;
      const double r = 1.0 / (al + sg[k] - bpv * bpv * rd[k]);
      rd[k] = r;
      rho[k] *= be * r;
      const double ei = w[k] * gb[k] * rho[k];
      e += ei;
      m = fmax(m, ei);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, o);
      m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    if (lane != 0) return;
    const int step = j - 1;
    p.a.lzc.bhist[row + step] = be;
    const int total = L.total + 1;
    L.total = total;
    L.w_reads += (step > 0 ? 2 : 1);
    int stop = 1, status = 0, fin = 1;
    if (!isfinite(be) || !isfinite(e)) status = 2;
    else if ((L.even ? m * p.a.lzc.poles->n <= L.thr : e <= L.thr) || be == 0.0) status = 0;
    else if (total >= L.maxit) status = 1;
    else if (step + 2 > L.cap - 1) {   // the cycle is full: restart from its last vector
      status = 3;
      fin = 0;
    } else stop = 0;
    if (stop) {
      L.err = e;
      L.alpha = al;
      L.beta_prev = be;
      L.j = j;
      L.done = 1;
      L.status = status;
      L.finished = fin;
      __stcg(p.bar + 2 + ds, 1u);
    }
  }
};

// Body: hop<MODE>(j, sh) forms the hop sums of the block's tiles, finish<MODE>(j, sh) their
// epilogues and leaves each warp's partial sum in sh.acc.
// The two roles run the same sequence of block barriers in loops of their own, so that neither
// holds the other's registers.
__device__ __forceinline__ void lzp_block_barrier() { asm volatile("bar.sync 0;" ::: "memory"); }
__device__ __forceinline__ bool lzp_all_done(const LzpShared& sh, int n) {
  int all = 1;   // the flags are those of the phase before: the same in every block
  for (int s = 0; s < n; ++s) all &= sh.c[s].done != 0;
  return all != 0;
}
template <typename Body>
__device__ __forceinline__ void lzp_run(const LzPersist& p, Body& body, LzpShared& sh) {
  const int warps = (blockDim.x >> 5) - 1, warp = threadIdx.x >> 5, lane = lane_id();
  const int n = p.a.nrhs;
  for (int e = threadIdx.x; e < LZP_WARPS * LZP_SYS; e += blockDim.x) (&sh.acc[0][0])[e] = 0.0;
  for (int e = threadIdx.x; e < n; e += blockDim.x) sh.c[e].done = p.a.lzc.lz[e].done;
  lzp_block_barrier();
  if (warp == warps) {
    LzpScalar sc;
    sc.init(p);
    for (int j = 0;; ++j) {
#pragma unroll
      for (int phase = 0; phase < 2; ++phase) {
        sc.coefficients(p, phase, j, sh);
        lzp_block_barrier();
        if (lzp_all_done(sh, n)) return;
        sc.record(p, phase, j);
        lzp_block_barrier();
        lzp_block_barrier();
        if (!sh.ok) return;
      }
    }
  }
  unsigned int target = 0;
  for (int j = 0;; ++j) {
#pragma unroll
    for (int phase = 0; phase < 2; ++phase) {
      if (phase == 0) body.template hop<MODE_LZK>(j, sh);
      else body.template hop<MODE_LZL>(j, sh);
      lzp_block_barrier();
      if (lzp_all_done(sh, n)) return;
      if (phase == 0) body.template finish<MODE_LZK>(j, sh);
      else body.template finish<MODE_LZL>(j, sh);
      lzp_block_barrier();
      target += gridDim.x;
      if (warp == 0) {
        for (int s = 0; s < n; ++s) {
          double v = lane < warps ? sh.acc[lane][s] : 0.0;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane == 0) __stcg(p.part + (size_t)(phase * n + s) * LZP_BLOCKS + blockIdx.x, v);
        }
        if (lane == 0) sh.ok = lzp_barrier(p.bar, target, p.wait_ns);
      }
      lzp_block_barrier();
      if (!sh.ok) return;
    }
  }
}

// The double-float kernel (dfwilson.cu) in mode `mode`; pio: the storage of the vector operands of
// MODE_OVL (P64 or P32), P64E otherwise.
void run_wilson_df(int mode, int pio, DArgs a, cudaStream_t st);
// Its Lanczos iteration in one launch; false when the launch is too large for it.
bool launch_lz_persistent_df(LzPersist& p, LzpShape* shape, int nsm, cudaStream_t st);
// Cooperative launch of p.tb tiles of tw warps per block (and one warp more); false when the blocks
// do not fit at once (a block takes each of its tiles once, so none may be missing). max_tiles: the most
// tiles a block of this kernel takes; its shared memory is the limit that is set, the same on every
// call, since contexts in other threads launch the same kernel with other sizes.
template <typename K>
bool lzp_launch(K kernel, LzPersist& p, int tw, size_t smem_tile, int max_tiles, int nsm, cudaStream_t st) {
  const int threads = 32 * (p.tb * tw + 1);
  const size_t smem = smem_tile * p.tb;
  const int grid = (p.ntile + p.tb - 1) / p.tb;
  if (smem_tile * max_tiles > 40 * 1024 &&
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(smem_tile * max_tiles)) !=
          cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (grid < p.a.nrhs || grid > LZP_BLOCKS || grid > per * nsm) return false;
  void* args[] = {&p};
  if (cudaLaunchCooperativeKernel((const void*)kernel, dim3((unsigned)grid), dim3((unsigned)threads), args, smem, st) !=
      cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

}  // namespace ovl
