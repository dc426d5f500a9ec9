// The double-float Wilson kernel: K of dslash.cu (same modes, same meaning of its arguments)
// with FP64-level accuracy on the FP32 pipes.
//
// Arithmetic: packed double-float (dfpair.cuh), lane 0 the site i of the first half of the
// lattice in t, lane 1 the site i + V/2. Fields hold the pair's high words and low words as
// one 16-byte chunk per real number, links likewise, so every load is a natural operand.
//
// Threads: two lanes of a warp share a pair of sites, lane `half` holding upper spin `half`.
// The projection (1 -+ gamma_mu) leaves two half spinors h0, h1 (upper spins 0 and 1 plus a
// power of i times a lower spin); the thread builds h_half, multiplies it by the link of the
// hop (eight-slot link field: U_mu(x), or U_mu(x - mu)^dag, boundary sign folded in) and adds
// the result to its upper spin and, times a power of i, to one lower spin: spin 3 - half for
// mu <= 1, which the other lane owns (the sums change lanes once, after mu = 1), spin
// 2 + half for mu >= 2. One rolled loop body serves every hop (unrolled over all eight it
// leaves the instruction cache): a power of i only chooses which of the two chunks (re, im)
// of the lower spin is loaded into which operand, and a sign, which rides on a multiply-add.
//
// What bounds it (ncu, 16^3 x 16, 6 systems, Lanczos modes): the FP32 pipes are busy 55% to 58% of the
// cycles (527 packed operations per thread and hop), the rest is the latency of the loads that three
// warps per scheduler do not cover. 168 registers (12 warps per SM) against 128 (16 warps, spilling and
// scheduled with less overlap): 0.530 against 0.841 ms on 16^3 x 32 with 12 systems. Measured there
// against the scalar kernel before it (one thread per site, 12 operations per product term):
// K launch 0.678 -> 0.517 ms, on 24^3 x 48 2.61 ms (3.0 G site applications/s; 2.4 before), one
// system on 16^3 x 32 0.070 -> 0.060 ms; a whole sign to 1e-10, 12 systems, 181 -> 146 ms. Error against
// FP64 4.7e-15 of the norm (4.8e-15 before), with the hops shared among groups 3.4e-15 to 4.4e-15.
#include "dfpair.cuh"
#include "wilson.cuh"

namespace ovl {

namespace {

// P pairs of sites per block: 32 (64 sites: the partial sums keep the BX layout), or 8 for eight
// groups on the smallest launches, which would otherwise leave most SMs without a block.
// Resident blocks per SM that the registers are capped for:
constexpr int df_resident(int G, int P) { return G == 1 ? 6 : G == 2 || P == 8 ? 3 : G == 4 ? 2 : 1; }

__device__ __forceinline__ void prefetch_l1(const void* p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// hop n seen from one thread
struct Hop {
  int nbr;        // index of the neighbour pair
  bool swap;      // its lanes are exchanged (the hop leaves this half of the lattice in t)
  int other;      // lower spin the projection pairs with spin `half`
  int a, b;       // powers of i of the projection and of the lower-spin sum
};
__device__ __forceinline__ Hop hop_of(const Geom& g, int lth, const int x[4], int i, int half, int n) {
  const int mu = n >> 1;
  const bool fwd = (n & 1) == 0;
  const int sS = fwd ? 2 : 0;   // (1 + S gamma_mu) with S = i^sS
  const bool lo3 = mu <= 1;
  const int a0 = sS + (mu == 0 || mu == 2 ? 1 : mu == 1 ? 2 : 0);
  const int a1 = sS + (mu == 0 ? 1 : mu == 2 ? 3 : 0);
  const int b0 = sS + (mu == 0 || mu == 2 ? 3 : 0);
  const int b1 = sS + (mu == 0 ? 3 : mu == 1 ? 2 : mu == 2 ? 1 : 0);
  Hop h;
  h.other = lo3 ? 3 - half : 2 + half;
  h.a = (half == 0 ? a0 : a1) & 3;
  h.b = ((half == 0) == lo3 ? b1 : b0) & 3;
  const int xm = mu == 0 ? x[0] : mu == 1 ? x[1] : mu == 2 ? x[2] : x[3];
  const int lm = mu == 0 ? g.L[0] : mu == 1 ? g.L[1] : mu == 2 ? g.L[2] : lth;
  const int st = mu == 0 ? 1 : mu == 1 ? g.L[0] : mu == 2 ? g.L[0] * g.L[1] : g.L[0] * g.L[1] * g.L[2];
  const bool wrap = fwd ? xm == lm - 1 : xm == 0;
  h.nbr = fwd ? (wrap ? i - (lm - 1) * st : i + st) : (wrap ? i + (lm - 1) * st : i - st);
  h.swap = wrap && mu == 3;
  return h;
}

// where the chunks of pair i of a field of nb blocks, and of the links of its hop n, begin
__device__ __forceinline__ const ulonglong2* pair_at(const SpinorRef& in, size_t fblk, int i) {
  return reinterpret_cast<const ulonglong2*>(in.data) + ((fblk + (i >> 5)) * 768 + (i & 31));
}
__device__ __forceinline__ const ulonglong2* link_at(const LinkRef& L, int i, int n) {
  return reinterpret_cast<const ulonglong2*>(L.data) + ((size_t)((i >> 5) * 8 + n) * 576 + (i & 31));
}
// Prefetch of the next hop into L1, shared out over the lanes of a warp: eight pairs in a row
// make a 128-byte line of every chunk, so of the sixteen lanes that hold them lane `m` fetches
// chunks m and m + 16 at its own pair (one prefetch per lane and chunk asked for every line
// sixteen times: 21 instructions per lane and hop instead of these 2 to 4).
__device__ __forceinline__ void prefetch_spinor(const ulonglong2* b, int m) {
  prefetch_l1(b + m * 32);
  if (m < 8) prefetch_l1(b + (m + 16) * 32);
}
__device__ __forceinline__ void prefetch_link(const ulonglong2* u, int m) {
  prefetch_l1(u + m * 32);
  if (m < 2) prefetch_l1(u + (m + 16) * 32);
}
__device__ __forceinline__ void prefetch_l2_spinor(const ulonglong2* b, int m) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(b + m * 32));
  if (m < 8) asm volatile("prefetch.global.L2 [%0];" ::"l"(b + (m + 16) * 32));
}
// the operands of colour c of the projection: re, im of the upper spin and of the (i^a times)
// lower spin of the neighbour
struct Oper {
  ulonglong2 p0, p1, q0, q1;
};
__device__ __forceinline__ Oper load_oper(const ulonglong2* b, int half, const Hop& h, int c) {
  const ulonglong2* p = b + half * 192;
  const ulonglong2* q0 = b + h.other * 192 + (h.a & 1) * 32;
  const ulonglong2* q1 = b + h.other * 192 + 32 - (h.a & 1) * 32;
  return {p[64 * c], p[64 * c + 32], q0[64 * c], q1[64 * c]};
}
__device__ __forceinline__ float sgn_re(int k) { return k == 1 || k == 2 ? -1.f : 1.f; }
__device__ __forceinline__ float sgn_im(int k) { return k >= 2 ? -1.f : 1.f; }

// up[c][r]: upper spin `half`; low[c][r]: the lower spin of the current half of the hops.
// b, u: the neighbour's chunks and the link of this hop.
template <bool TIGHT>
__device__ __forceinline__ void hop_pair(const ulonglong2* b, const ulonglong2* u, int half, const Hop& h,
                                         dd2 up[3][2], dd2 low[3][2]) {
  const f2 ar = bc(sgn_re(h.a)), ai = bc(sgn_im(h.a));
  dot2p wr[3], wi[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const Oper o = load_oper(b, half, h, c);
    dd2 hr = dd2_lazy({o.p0.x, o.p0.y}, {o.q0.x, o.q0.y}, ar);
    dd2 hi = dd2_lazy({o.p1.x, o.p1.y}, {o.q1.x, o.q1.y}, ai);
    if (h.swap) {
      hr = {swap2(hr.h), swap2(hr.l)};
      hi = {swap2(hi.h), swap2(hi.l)};
    }
    const f2 nr = neg2(hr.h), ni = neg2(hi.h), nil = neg2(hi.l);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const ulonglong2 ur = __ldg(u + (3 * a + c) * 64), ui = __ldg(u + (3 * a + c) * 64 + 32);
      // w = U h: re = sum (Ur hr - Ui hi), im = sum (Ur hi + Ui hr)
      if (c == 0) {
        wr[a] = dot2p_first(ur.x, ur.y, hr.h, nr, hr.l);
        wi[a] = dot2p_first(ur.x, ur.y, hi.h, ni, hi.l);
      } else {
        dot2p_add<TIGHT>(wr[a], ur.x, ur.y, hr.h, nr, hr.l);
        dot2p_add<TIGHT>(wi[a], ur.x, ur.y, hi.h, ni, hi.l);
      }
      dot2p_add<TIGHT>(wr[a], ui.x, ui.y, ni, hi.h, nil);
      dot2p_add<TIGHT>(wi[a], ui.x, ui.y, hr.h, nr, hr.l);
    }
  }
  const bool oddb = (h.b & 1) != 0;
  const f2 br = bc(sgn_re(h.b)), bi = bc(sgn_im(h.b));
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const dd2 r = {wr[a].s, wr[a].c}, m = {wi[a].s, wi[a].c};
    up[a][0] = dd2_lazy(up[a][0], r);
    up[a][1] = dd2_lazy(up[a][1], m);
    low[a][0] = dd2_lazy(low[a][0], oddb ? m : r, br);
    low[a][1] = dd2_lazy(low[a][1], oddb ? r : m, bi);
  }
}

__device__ __forceinline__ dd2 shfl_pair(dd2 v) {
  return {__shfl_xor_sync(0xffffffffu, v.h, 1), __shfl_xor_sync(0xffffffffu, v.l, 1)};
}

// The epilogue of N complex components kc .. kc + N - 1 of the pair (the mode list of dslash.cu):
// hop sums in, partial sums into d. Every load is issued before the first store (which may alias
// them as far as the compiler can know).
struct DfScal {
  fac2 kap, s0, s1;   // -kappa; LZK: 1 / n_j; LZL: -a, -b; R: sigma0, -alpha; OVL: c1, c2
};
template <int MODE, int PIO, int N>
__device__ __forceinline__ void df_epilogue(const DArgs& a, const DfScal& k, int rhs, int fin, int j, int kc, int i,
                                            const dd2 (*sum)[2], dot2p d[4]) {
  const int nb = df_blocks(a.g.V);
  const bool red = a.partials != nullptr;
  const bool two = MODE == MODE_LZL ? j > 0 : MODE == MODE_OVL ? a.coef != nullptr || a.c1 != 0.0 : true;
  dd2 o[N][2], w[N][2], y[N][2];
#pragma unroll
  for (int c = 0; c < N; ++c)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      o[c][r] = dfp_ld(a.in, dfp_at(fin, kc + c, r, i, nb));
      if constexpr (MODE == MODE_R) {
        w[c][r] = dfp_ld(a.aux1, dfp_at(rhs, kc + c, r, i, nb));
        y[c][r] = dfp_ld(a.aux2, dfp_at(rhs, kc + c, r, i, nb));
      } else if constexpr (MODE == MODE_LZL) {
        w[c][r] = dfp_ld(a.aux1, dfp_at(j * a.nrhs + rhs, kc + c, r, i, nb));
        if (two) y[c][r] = dfp_ld(a.aux1, dfp_at((j - 1) * a.nrhs + rhs, kc + c, r, i, nb));
      }
    }
  if constexpr (MODE == MODE_OVL) {
#pragma unroll
    for (int c = 0; c < N; ++c) {
      if (two) dfp_load<PIO>(a.aux1, rhs, kc + c, i, w[c][0], w[c][1]);
      if (red) dfp_load<PIO>(a.aux2, rhs, kc + c, i, y[c][0], y[c][1]);
    }
  }
#pragma unroll
  for (int c = 0; c < N; ++c) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      // in - kappa hop; gamma5 negates the lower spins
      dd2 t = dd2_add(o[c][r], dd2_mul(k.kap, sum[c][r]));
      if (MODE != MODE_OVL && kc >= 6) t = dd2_neg(t);
      if constexpr (MODE == MODE_K) {
        if (red) dot2p_add(d[1], o[c][r], o[c][r]);
      } else if constexpr (MODE == MODE_R) {
        t = dd2_add(y[c][r], dd2_mul(k.s1, dd2_add(t, dd2_mul(k.s0, w[c][r]))));
      } else if constexpr (MODE == MODE_LZK) {
        t = dd2_mul(k.s0, t);
      } else if constexpr (MODE == MODE_LZL) {
        t = dd2_add(t, dd2_mul(k.s0, w[c][r]));
        if (two) t = dd2_add(t, dd2_mul(k.s1, y[c][r]));
      } else {
        t = dd2_mul(k.s1, t);
        if (two) t = dd2_add(dd2_mul(k.s0, w[c][r]), t);
        if (a.herm && kc >= 6) t = dd2_neg(t);
      }
      if (MODE != MODE_OVL && red) dot2p_add(d[0], t, t);
      o[c][r] = t;
    }
    if constexpr (MODE == MODE_OVL) {
      if (red) {
        dot2p_add(d[0], y[c][0], o[c][0]);   // (w, out) = sum conj(w) out
        dot2p_add(d[0], y[c][1], o[c][1]);
        dot2p_add(d[1], y[c][0], o[c][1]);
        dot2p_add(d[1], dd2_neg(y[c][1]), o[c][0]);
        dot2p_add(d[2], o[c][0], o[c][0]);
        dot2p_add(d[2], o[c][1], o[c][1]);
        dot2p_add(d[3], y[c][0], y[c][0]);
        dot2p_add(d[3], y[c][1], y[c][1]);
      }
    }
  }
  const SpinorRef& out = MODE == MODE_R ? a.aux2 : a.out;
  const int fld = MODE == MODE_LZL ? (j + 1) * a.nrhs + rhs : rhs;
#pragma unroll
  for (int c = 0; c < N; ++c) dfp_store<MODE == MODE_OVL ? PIO : P64E>(out, fld, kc + c, i, o[c][0], o[c][1]);
}

// G groups of threads (threadIdx.z) share the eight hops of a pair, 8 / G each; their sums
// meet in shared memory, where group z finishes the components z, z + G, .. of the spinor.
template <int MODE, int PIO, int G, int P>
__global__ void __launch_bounds__(2 * P * G, df_resident(G, P)) df_wilson_kernel(const DArgs a) {
  constexpr int NR = nred(MODE);
  extern __shared__ ulonglong2 part[];   // G > 1: [z][component (6 x re, im)][thread x]
  constexpr int NW = 2 * P * G / 32;   // warps
  __shared__ double red[NW][NR];
  const int half = threadIdx.x & 1;
  const int grp = G > 1 ? threadIdx.z : 0;
  const int sb = blockIdx.x / a.nrhs;   // the systems of one site block together: they share its links in L1 / L2
  const int rhs = blockIdx.x - sb * a.nrhs;
  const int Vh = a.g.V >> 1;
  const int i = sb * P + (threadIdx.x >> 1);
  bool live = i < Vh;
  const int m = (threadIdx.x >> 1 & 7) + 8 * half;   // this lane's share of the prefetches
  const int n0 = grp * (8 / G), n1 = n0 + 8 / G;
  if (live) prefetch_link(link_at(a.links, i, n0), m);
  if constexpr (!kReadOnly<MODE>) {
    pdl_wait();
    pdl_release();
  }
  if (live && a.ms != nullptr && (MODE == MODE_K || MODE == MODE_R)) live = !a.ms[rhs].done;
  int fin = rhs, j = 0;   // field index of the hop input (the basis slot in MODE_LZK)
  if constexpr (MODE == MODE_LZK || MODE == MODE_LZL) {
    if (a.lz[rhs].done) return;   // every thread of the block
    j = a.lz[rhs].j;
    if (MODE == MODE_LZK) fin = j * a.nrhs + rhs;
  }
  dd2 up[3][2], low[3][2];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int r = 0; r < 2; ++r) up[c][r] = low[c][r] = dd2_zero();
  {
    const int lth = a.g.L[3] >> 1;
    const size_t fblk = (size_t)fin * df_blocks(a.g.V);
    int x[4] = {0, 0, 0, 0};
    if (live) site_coords(a.g, i, x);
    Hop h = hop_of(a.g, lth, x, i, half, n0);
    const ulonglong2* b = pair_at(a.in, fblk, h.nbr);
    const ulonglong2* u = link_at(a.links, i, n0);
    if (live) {
      prefetch_spinor(b, m);
      if constexpr (MODE == MODE_LZL) {   // the basis vectors of the epilogue come from HBM
        prefetch_l2_spinor(pair_at(a.aux1, (size_t)(j * a.nrhs + rhs) * df_blocks(a.g.V), i), m);
        if (j > 0) prefetch_l2_spinor(pair_at(a.aux1, (size_t)((j - 1) * a.nrhs + rhs) * df_blocks(a.g.V), i), m);
      }
    }
#pragma unroll 1
    for (int n = n0; n < n1; ++n) {
      if (live) {
        const int nn = min(n + 1, n1 - 1);
        const Hop nx = hop_of(a.g, lth, x, i, half, nn);
        const ulonglong2 *bn = pair_at(a.in, fblk, n + 1 < n1 ? nx.nbr : i), *un = link_at(a.links, i, nn);
        prefetch_spinor(bn, m);   // after the last hop the epilogue reads the pair itself
        if (n + 1 < n1) prefetch_link(un, m);
        hop_pair<(G >= 4)>(b, u, half, h, up, low);
        h = nx;
        b = bn;
        u = un;
      }
      // the lower spins of mu <= 1 belong to the other lane: exchanged after the last of them
      // (every lane of the warp takes part: the hops of a warp are the same, or with P = 8 the
      // two hops of one direction)
      if (n == min(n1 - 1, 3)) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            low[c][r] = shfl_pair(dd2_norm(low[c][r]));
            up[c][r] = dd2_norm(up[c][r]);
          }
      }
    }
  }
  dot2p d[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) d[k] = {0ull, 0ull};
  DfScal k;
  if (live) {
    k.kap = fac2_minus(make_float2(a.kap_h, a.kap_l));
    if constexpr (MODE == MODE_LZK) {
      const float2 f = a.lz[rhs].fn;
      k.s0 = {bc(f.x), bc(-f.x), bc(f.y)};
    } else if constexpr (MODE == MODE_LZL) {
      k.s0 = fac2_minus(a.lz[rhs].fa);
      k.s1 = fac2_minus(a.lz[rhs].fb);
    } else if constexpr (MODE == MODE_R) {
      k.s0 = fac2_bc(a.sigma0);
      k.s1 = fac2_bc(-a.ms[rhs].alpha);
    } else if constexpr (MODE == MODE_OVL) {
      k.s0 = fac2_bc(a.coef ? a.coef[2 * rhs] : a.c1);
      k.s1 = fac2_bc(a.coef ? a.coef[2 * rhs + 1] : a.c2);
    }
  }
  if constexpr (G == 1) {
    if (live) {
      df_epilogue<MODE, PIO, 3>(a, k, rhs, fin, j, 3 * half, i, up, d);
      df_epilogue<MODE, PIO, 3>(a, k, rhs, fin, j, 6 + 3 * half, i, low, d);
    }
  } else {
    constexpr int X = 2 * P;
    ulonglong2* mine = part + grp * 12 * X + threadIdx.x;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        mine[(2 * c + r) * X] = make_ulonglong2(up[c][r].h, up[c][r].l);
        mine[(6 + 2 * c + r) * X] = make_ulonglong2(low[c][r].h, low[c][r].l);
      }
    __syncthreads();
    if (live) {
      for (int q = grp; q < 6; q += G) {
        const ulonglong2* s = part + 2 * q * X + threadIdx.x;
        dd2 t[1][2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          t[0][r] = {s[r * X].x, s[r * X].y};
#pragma unroll
          for (int z = 1; z < G; ++z) {
            const ulonglong2 w = s[(z * 12 + r) * X];
            t[0][r] = dd2_add(t[0][r], {w.x, w.y});
          }
        }
        df_epilogue<MODE, PIO, 1>(a, k, rhs, fin, j, q < 3 ? 3 * half + q : 3 + 3 * half + q, i, t, d);
      }
    }
  }
  if (a.partials != nullptr) {
    // lanes in three words, a fixed tree; then FP64 over the warps in the order z, x
    const int lin = threadIdx.z * 2 * P + threadIdx.x;
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      const double v = dot2p_warp_sum(d[q]);
      if ((lin & 31) == 0) red[lin >> 5][q] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.z == 0) {
      double tot[NVRED] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int q = 0; q < NR; ++q)
        for (int w = 0; w < NW; ++w) tot[q] += red[w][q];
      store_partials<MODE>(a, rhs, sb, tot);
    }
  }
  if constexpr (MODE == MODE_LZK || MODE == MODE_LZL) {
    if (threadIdx.z * 2 * P + threadIdx.x < 32) lz_arrive<MODE>(a, rhs, a.nsb);
  }
}

template <int MODE, int PIO, int G, int P = 32>
void run_g(DArgs a, cudaStream_t st) {
  a.nsb = ((a.g.V >> 1) + P - 1) / P;
  const size_t smem = G == 1 ? 0 : sizeof(ulonglong2) * 2 * P * 12 * G;
  if (smem > 40 * 1024)   // with the static arrays, past the 48 KB that need no opt-in
    cudaFuncSetAttribute(df_wilson_kernel<MODE, PIO, G, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  launch_step(df_wilson_kernel<MODE, PIO, G, P>, dim3((unsigned)(a.nsb * a.nrhs)), dim3(2 * P, 1, G), smem, st, a);
}

template <int MODE, int PIO>
void run_m(const DArgs& a, cudaStream_t st) {
  switch (a.variant >= 0 ? a.variant : wilson_df_variant(a.g.V, a.nrhs)) {
    case 0: run_g<MODE, PIO, 1>(a, st); break;
    case 3: run_g<MODE, PIO, 2>(a, st); break;
    case 2: run_g<MODE, PIO, 4>(a, st); break;
    default:
      // small blocks where the caller does not read partial sums per 64 sites and where blocks of 32
      // pairs would leave half of the 152 SMs without one
      if constexpr (MODE == MODE_LZK || MODE == MODE_LZL || MODE == MODE_K) {
        if ((long long)a.g.V * a.nrhs <= 32 * 152 && (MODE != MODE_K || a.partials == nullptr)) {
          run_g<MODE, PIO, 8, 8>(a, st);
          break;
        }
      }
      run_g<MODE, PIO, 8>(a, st);
  }
}

// ---- the whole Lanczos iteration in one launch (lzp_run) --------------------------------
// A tile is P pairs of one system in G groups, as in df_wilson_kernel.
template <int G, int P>
struct LzpBodyDf {
  static constexpr int X = 2 * P, T = X * G;   // threads of a group, of a tile
  const LzPersist& p;
  const DArgs& a;
  ulonglong2* part;   // of this tile: [group][component (6 x re, im)][thread x]
  int rhs, i, half, grp, x;
  bool in_tile;
  __device__ __forceinline__ LzpBodyDf(const LzPersist& q, ulonglong2* sm) : p(q), a(q.a) {
    const int slot = threadIdx.x / T, lin = threadIdx.x % T, tile = blockIdx.x * p.tb + slot;
    part = sm + slot * (G * 12 * X);
    x = lin % X;
    half = x & 1;
    grp = lin / X;
    rhs = tile % a.nrhs;
    i = tile / a.nrhs * P + (x >> 1);
    in_tile = tile < p.ntile && i < (a.g.V >> 1);
  }
  template <int MODE>
  __device__ __forceinline__ void hop(int j, const LzpShared& sh) {
    const bool live = in_tile && !sh.c[rhs].done;
    dd2 up[3][2], low[3][2];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int r = 0; r < 2; ++r) up[c][r] = low[c][r] = dd2_zero();
    const SpinorRef& in = MODE == MODE_LZK ? p.W : p.t;
    const int nb = df_blocks(a.g.V), lth = a.g.L[3] >> 1, m = (x >> 1 & 7) + 8 * half;
    const size_t fblk = (size_t)(MODE == MODE_LZK ? j * a.nrhs + rhs : rhs) * nb;
    int xc[4] = {0, 0, 0, 0};
    if (live) {
      site_coords(a.g, i, xc);
      if constexpr (MODE == MODE_LZL) {
        // what the epilogue reads besides: on its way from HBM or L2 while the hops are summed
        if (grp == 0) prefetch_l2_spinor(pair_at(p.W, (size_t)(j * a.nrhs + rhs) * nb, i), m);
        if (grp == 1 && j > 0) prefetch_l2_spinor(pair_at(p.W, (size_t)((j - 1) * a.nrhs + rhs) * nb, i), m);
      }
    }
    const int n0 = grp * (8 / G), n1 = n0 + 8 / G;
    Hop h = hop_of(a.g, lth, xc, i, half, n0);
#pragma unroll 1
    for (int n = n0; n < n1; ++n) {
      if (live) {
        const int nn = min(n + 1, n1 - 1);
        const Hop nx = hop_of(a.g, lth, xc, i, half, nn);
        if (n + 1 < n1) {
          prefetch_spinor(pair_at(in, fblk, nx.nbr), m);
          prefetch_link(link_at(a.links, i, nn), m);
        }
        hop_pair<(G >= 4)>(pair_at(in, fblk, h.nbr), link_at(a.links, i, n), half, h, up, low);
        h = nx;
      }
      if (n == min(n1 - 1, 3)) {   // as in df_wilson_kernel; with P = 8 both groups of a warp come here in the same turn
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            low[c][r] = shfl_pair(dd2_norm(low[c][r]));
            up[c][r] = dd2_norm(up[c][r]);
          }
      }
    }
    ulonglong2* mine = part + grp * 12 * X + x;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        mine[(2 * c + r) * X] = make_ulonglong2(up[c][r].h, up[c][r].l);
        mine[(6 + 2 * c + r) * X] = make_ulonglong2(low[c][r].h, low[c][r].l);
      }
  }
  template <int MODE>
  __device__ __forceinline__ void finish(int j, LzpShared& sh) {
    const LzCoef& L = sh.c[rhs];
    dot2p d[4];
    d[0] = {0ull, 0ull};
    if (in_tile && !L.done) {
      DfScal k;
      k.kap = fac2_minus(make_float2(a.kap_h, a.kap_l));
      if constexpr (MODE == MODE_LZK) {
        k.s0 = {bc(L.fn.x), bc(-L.fn.x), bc(L.fn.y)};
      } else {
        k.s0 = fac2_minus(L.fa);
        k.s1 = fac2_minus(L.fb);
      }
      for (int q = grp; q < 6; q += G) {
        const ulonglong2* s = part + 2 * q * X + x;
        dd2 t[1][2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          t[0][r] = {s[r * X].x, s[r * X].y};
#pragma unroll
          for (int z = 1; z < G; ++z) {
            const ulonglong2 w = s[(z * 12 + r) * X];
            t[0][r] = dd2_add(t[0][r], {w.x, w.y});
          }
        }
        df_epilogue<MODE, P64E, 1>(MODE == MODE_LZK ? p.a : p.l, k, rhs, MODE == MODE_LZK ? j * a.nrhs + rhs : rhs, j,
                                   q < 3 ? 3 * half + q : 3 + 3 * half + q, i, t, d);
      }
    }
    const double v = dot2p_warp_sum(d[0]);
    if (lane_id() == 0) sh.acc[threadIdx.x >> 5][rhs] = v;
  }
};
template <int G, int P, int TB>
__global__ void __launch_bounds__(2 * P * G * TB + 32, 1) lz_persistent_df_kernel(const LzPersist p) {
  extern __shared__ ulonglong2 part[];
  __shared__ LzpShared sh;
  LzpBodyDf<G, P> body(p, part);
  lzp_run(p, body, sh);
}
template <int G, int P, int TB>
bool lzp_df(LzPersist& p, LzpShape* shape, int nsm, cudaStream_t st) {
  p.ntile = ((p.a.g.V >> 1) + P - 1) / P * p.a.nrhs;
  p.tb = (p.ntile + nsm - 1) / nsm;
  *shape = {G, p.tb};
  return p.tb <= TB && lzp_launch(lz_persistent_df_kernel<G, P, TB>, p, 2 * P * G / 32,
                                  sizeof(ulonglong2) * G * 12 * 2 * P, TB, nsm, st);
}

}  // namespace

// A phase is mostly the latency of the hops that a thread takes one after the other: eight groups on
// 8 pairs while the SMs hold every tile at 96 registers or more (9728 sites x systems on 152 SMs; 80
// registers spill: 8^3 x 16 2.2 instead of 2.1 ms), four groups on 8 pairs up to 21888 (9 tiles at 96
// registers), two on 16 pairs up to 34048. Sign to 1e-10 with four / two groups, ms: 10080 sites 2.60 /
// 3.82, 12288 2.62 / 3.68, 16384 2.99 / 3.87, 20000 3.92 / 4.15, 20480 3.95 / 4.05. Requesting the
// epilogue's operands before the hops made every size slower (4^4 1.35 -> 1.39 ms).
bool launch_lz_persistent_df(LzPersist& p, LzpShape* shape, int nsm, cudaStream_t st) {
  return lzp_df<8, 8, 3>(p, shape, nsm, st) || lzp_df<8, 8, 4>(p, shape, nsm, st) ||
         lzp_df<4, 8, 7>(p, shape, nsm, st) || lzp_df<4, 8, 9>(p, shape, nsm, st) ||
         lzp_df<2, 16, 5>(p, shape, nsm, st) || lzp_df<2, 16, 7>(p, shape, nsm, st);
}

// Two threads per pair and system, times 1, 2, 4 or 8 groups. One group is the cheapest form
// (no exchange in shared memory) once its threads fill the SMs; below, the hops of a pair are
// spread over more groups. The lines are those of the 152 SMs they were measured on. K launches, us with 1 / 2 / 4 / 8 groups: 49152 threads (8^4, 12
// systems) 24.6 / 24.7 / 30.8 / 32.9; 32768 (8^3 x 16, 4) 18.5 / 18.5 / 22.6 / 22.6; 20736 (12^4, 1)
// 18.5 / 14.5 / 18.5 / 18.6; 16384 (8^4, 4) 14.4 / 12.4 / 12.4 / 12.6; 8192 (8^3 x 16, 1)
// 14.4 / 10.3 / 8.3 / 8.3; 4096 (8^4, 1) 14.4 / 10.4 / 8.3 / 8.2.
int wilson_df_variant(int V, int nrhs) {
  const long long threads = (long long)V * nrhs;
  return threads >= 40000 ? 0 : threads >= 18000 ? 3 : threads >= 9000 ? 2 : 1;
}

void run_wilson_df(int mode, int pio, DArgs a, cudaStream_t st) {
  if (mode == MODE_K) run_m<MODE_K, P64E>(a, st);
  else if (mode == MODE_R) run_m<MODE_R, P64E>(a, st);
  else if (mode == MODE_LZK) run_m<MODE_LZK, P64E>(a, st);
  else if (mode == MODE_LZL) run_m<MODE_LZL, P64E>(a, st);
  else if (pio == P64) run_m<MODE_OVL, P64>(a, st);
  else run_m<MODE_OVL, P32>(a, st);
}

}  // namespace ovl
