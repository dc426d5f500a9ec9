// Gram blocks G[i][j] += (A_i, [gamma5] B_j) on the fifth-generation tensor cores, accurate
// to FP64 level: the dense contractions of the Ritz step (Alg. 6: E = V^dag V,
// M = (V^D)^dag V^D + 2 mu delta V^dag gamma5 V^D) and of the deflated starts (Sec. 4:
// Psi^dag b, (D Psi)^dag b), on FP64 or FP32 fields.
//
// Method: error-free splitting of the operands into small integers (Ozaki, Ogita, Oishi and
// Rump, "Error-free transformations of matrix multiplication by using fast routines of
// matrix multiplication", 2012), with BF16 slices and FP32 accumulation in tensor memory.
// Every vector i gets a power-of-two scale 2^e_i above its largest element; each real
// element x is written in six balanced base-128 digits a_1 .. a_6 (a_1 in [-128, 128], the
// others in [-64, 64]), x = 2^e_i sum_s a_s 2^(-7 s) up to 9/8 2^(e_i - 43), without bias, by FP32
// arithmetic (tg_digits). Digits are exact in BF16 and
// their products exact in the tensor core; for each group g = s + t (2 .. 8) the products
// a_s b_t summed over 512 reals stay within 2^24 in magnitude, so the FP32 accumulator holds
// that sum exactly. Every 512 reals the seven group sums are read from tensor memory and
// added, scaled by 2^(-7 g), into a normalised double-float (hi + lo FP32) accumulator per output;
// the partial results of the CTAs that split the sum are added in FP64 in a fixed order.
// The last digit is rounded to nearest; the pairs with s + t > 8 (weight 2^-63 and below) are left out.
// The error is then that of the representation and one rounding of 2^-48 of the running sum per 512
// reals: on Gaussian data at most 4.2e-14 of |A_i| |B_j| over 70 x 70 vectors of 6144 reals with scales
// 1e-30 to 1e30, 1e-15 for FP32 fields, and 1.3e-13 on the diagonal of vectors of 1.6 M reals that one
// CTA sums whole (640 x 640; 7.6e-11 when the low word was not normalised).
//
// Complex arithmetic: vectors are read as interleaved (re, im) reals. With the A operand
// rows [A_i (64 vectors); A'_i] where A' = (-im, re) per complex element, one MMA of
// M = 128 rows against N = 64 B vectors gives Re (a, b) = sum a.b in rows 0..63 and
// Im (a, b) = sum a'.b in rows 64..127.
//
// One CTA (512 threads) per SM. Warps 1 .. 15 slice stages of 16 complex elements of 64 A and 64 B
// vectors into the canonical no-swizzle K-major layout (core matrices of 8 rows x 16 bytes), three
// stages in shared memory, the next stage's elements already loaded; warp 0 issues a stage's 52
// MMAs (2 K-steps x 26 digit pairs) when its slices are complete (full) and commits them to the
// barrier that frees it (empty). All warps read a chunk's sums out of tensor memory once its
// MMAs are done (fbar), two stages into the next chunk, whose MMAs wait for that (flushed). With
// block barriers instead (two per stage, operands staged by cp.async) the warps waited for each
// other 3.5 cycles per issued instruction. Bound now by the ALU pipe of the slicing (55% busy,
// tensor pipe 34%). FP64 fields, 16^3 x 32: 128 x 128 17.6 -> 7.3 ms, 64 x 64 8.7 -> 2.1, 64 x 12 8.6 -> 1.7
// (more than half of that was the exponent pass, below).
// Waits are bounded (wait_ns, 2 s by default): one that gives up sets the error flag, the CTA skips the
// rest, warp by warp (warp_wait), waits once more (again bounded) for the MMAs it has committed, frees its tensor memory
// and returns, and the host reports OVL_ETIMEOUT.
#include <limits.h>
#include <stdint.h>

#include <algorithm>

#include "dfpair.cuh"
#include "kernels.h"

namespace ovl {

namespace {

constexpr int TG_THREADS = 512;
constexpr int TG_S = 6;                          // base-128 digits per real (42 bits)
constexpr int TG_G = 7;                          // groups s + t = 2 .. 8 kept
constexpr int TG_NA = 64;                        // A vectors per tile (M = 128 rows with A')
constexpr int TG_NB = 64;                        // B vectors per tile (N)
constexpr int TG_CPT = TG_NB / (TG_THREADS / 128);   // output columns per thread in the flush
constexpr int TG_KC = 16;                        // complex elements per stage (32 reals)
constexpr int TG_CHUNK = 16;                     // stages per exact accumulation (512 reals)
constexpr int TG_TILE_A = 128 * 32 * 2;          // bytes of one digit tile of A (128 rows x 32 bf16)
constexpr int TG_TILE_B = TG_NB * 32 * 2;        // bytes of one digit tile of B
constexpr int TG_STAGE = TG_S * (TG_TILE_A + TG_TILE_B);
constexpr int TG_BUF = 3;                        // digit stages in shared memory
constexpr int TG_SMEM = TG_BUF * TG_STAGE + 1024;   // and alignment
__host__ __device__ constexpr int tg_esize(int p) { return p == P64 ? 16 : 8; }
constexpr int TG_SLICERS = TG_THREADS / 32 - 1;  // warps 1 .. 15 slice, warp 0 issues the MMAs
constexpr int TG_TASKS = (64 + TG_SLICERS - 1) / TG_SLICERS;   // slicing tasks per warp and stage, at most
constexpr int TG_TMEM_COLS = 512;
static_assert(TG_G * TG_NB <= TG_TMEM_COLS, "group accumulators exceed the tensor-memory allocation");                // 7 groups x 64 columns, rounded to a power of 2
constexpr int TG_EXP_ZERO = -4000;               // scale exponent of an all-zero vector
constexpr unsigned long long TG_DRAIN_NS = 2000000000ull;   // the exit's wait for MMAs in flight

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Shared-memory matrix descriptor, K-major without swizzle: start address, leading byte
// offset (distance of core matrices along K), stride byte offset (along the rows), version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)((lbo & 0x3FFFF) >> 4) << 16;
  d |= (uint64_t)((sbo & 0x3FFFF) >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// true once the barrier's phase with this parity has completed, false after the limit or when
// another thread has given up (*gave_up). A limit of zero gives up without a look.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* gave_up,
                                          unsigned long long limit) {
  const unsigned long long t0 = global_ns();
  while (limit != 0) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (gave_up != nullptr && *gave_up) return false;
    if (global_ns() - t0 > limit) break;
  }
  if (gave_up != nullptr) *gave_up = 1;
  return false;
}
// The wait of a whole warp: true when every lane saw the phase complete. Lanes poll for
// themselves and may disagree when the time runs out; what follows (warp barriers, tcgen05.ld,
// the way out) takes the warp as one, so they vote first.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* gave_up,
                                          unsigned long long limit) {
  const bool ok = mbar_wait(bar, parity, gave_up, limit);
  return __all_sync(0xffffffffu, ok) != 0;
}

// a <- fl(a + b); the rounding error
__device__ __forceinline__ float two_sum(float& a, float b) {
  const float s = a + b, v = s - a;
  const float e = (a - (s - v)) + (b - v);
  a = s;
  return e;
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(da), "l"(db), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// binary exponent of the larger part of a complex element in global memory
template <int P>
struct TgLoad;
template <>
struct TgLoad<P64> {
  static __device__ __forceinline__ int expo(const void* base, size_t q) {
    const ulonglong2 w = __ldg(reinterpret_cast<const ulonglong2*>(base) + q);
    return max((int)((w.x >> 52) & 0x7FF), (int)((w.y >> 52) & 0x7FF)) - 1023;
  }
};
template <>
struct TgLoad<P32> {
  static __device__ __forceinline__ int expo(const void* base, size_t q) {
    const uint2 w = __ldg(reinterpret_cast<const uint2*>(base) + q);
    return max((int)((w.x >> 23) & 0xFF), (int)((w.y >> 23) & 0xFF)) - 127;
  }
};

// The six digits of one complex element (from the raw staging buffer) as BF16 pairs (real in the
// low half), negated when neg (gamma5 on B), by FP32 arithmetic on the FMA pipe, real and
// imaginary part on the two lanes of the packed instructions: with r = x 2^-e, six times
// d = round(128 r) by the 1.5 x 2^23 addition (exact for |128 r| < 2^22) and r <- 128 r - d
// (exact: the remainder of a float after its nearest integer), so d_0 is in [-128, 128], the
// others in [-64, 64], and x 2^-e = sum_s d_s 2^(-7 (s + 1)) up to 2^-43. A digit is an integer of
// at most 8 bits, so the upper half of its float is its exact BF16.
// FP32 operands: r by two power-of-two factors. FP64 operands, from their bits (conversions from
// FP64 are slow): r is the float of the leading 24 bits; the other 29, rounded to a second float
// (a 32-bit integer conversion, on a pipe that is idle otherwise), join the remainder after three
// digits, when 21 of the leading bits are spent (the third digit is chosen with them, so that the
// fourth stays in its range; that sum is rounded at 2^-46 or finer). Every rounding is to nearest, so
// an element is off by 2^-43, in rare cases up to 9/8 of that, without bias; cutting at 47 bits instead
// put 1.0e-14 on every diagonal entry of Gaussian data. About 75 instructions per element, against
// 270 for taking the digits out of a 64-bit fixed-point integer: a 64 x 64 tile on 16^4 1.43 -> 0.81 ms
// with the pipeline below.
__device__ __forceinline__ float tg_pow2(int k) { return __int_as_float((127 + k) << 23); }
// the digit of s (r itself, or r and what follows it, rounded); r becomes its remainder
__device__ __forceinline__ uint32_t tg_digit(f2 s, f2& r) {
  const f2 M = bc(12582912.0f), c128 = bc(128.0f);
  const f2 t = fma2(s, c128, M);
  const f2 dg = sub2(t, M);
  r = fma2(r, c128, sub2(M, t));
  return __byte_perm((uint32_t)dg, (uint32_t)(dg >> 32), 0x7632);
}
// x 2^-e as hi (24 bits) + lo 2^-21; thr = max(e + 897, 1): smaller exponent fields give 0
__device__ __forceinline__ void tg_split64(uint2 w, int e, int thr, uint32_t flip, float& hi, float& lo) {
  const int t = (int)((w.y >> 20) & 0x7FFu);
  const uint32_t sg = (w.y ^ flip) & 0x80000000u;
  const int ex = t - 896 - e;   // exponent field of the float, <= 126
  const uint32_t m = __funnelshift_l(w.x, w.y, 3) & 0x7FFFFFu;
  const bool z = t < thr;
  hi = __uint_as_float(z ? 0u : ((uint32_t)ex << 23) | m | sg);
  // the other 29 bits v, rounded to 24: v 2^(t - 1023 - 52 - e), times 2^21 in lo
  const float f = __uint2float_rn(w.x & 0x1FFFFFFFu);
  lo = __fmul_rn(f, __uint_as_float(z || ex <= 31 ? 0u : ((uint32_t)(ex - 31) << 23) | sg));
}
template <int P>
__device__ __forceinline__ void tg_digits(uint4 w4, int e, bool neg, uint32_t pd[TG_S]) {
  if constexpr (P == P32) {
    float2 w = make_float2(__uint_as_float(w4.x), __uint_as_float(w4.y));
    if (e == TG_EXP_ZERO) w = make_float2(0.f, 0.f);
    const int ec = e == TG_EXP_ZERO ? 0 : e;
    const int e1 = ec / 2, e2 = ec - e1;   // 2^-e as two factors inside the FP32 range
    const float g = neg ? -tg_pow2(-e2) : tg_pow2(-e2);
    f2 r = fma2(fma2(pk(w.x, w.y), bc(tg_pow2(-e1)), 0ull), bc(g), 0ull);
#pragma unroll
    for (int d = 0; d < TG_S; ++d) pd[d] = tg_digit(r, r);
  } else {
    const uint4 w = w4;
    const int thr = max(e + 897, 1);
    const uint32_t flip = neg ? 0x80000000u : 0u;
    float hr, lr, hi, li;
    tg_split64(make_uint2(w.x, w.y), e, thr, flip, hr, lr);
    tg_split64(make_uint2(w.z, w.w), e, thr, flip, hi, li);
    f2 r = pk(hr, hi);
    const f2 low = pk(lr, li);
    pd[0] = tg_digit(r, r);
    pd[1] = tg_digit(r, r);
    // the third digit sees the low part too, so that the fourth stays within 64
    pd[2] = tg_digit(fma2(low, bc(0.0078125f), r), r);
    r = add2(r, low);
    pd[3] = tg_digit(r, r);
    pd[4] = tg_digit(r, r);
    pd[5] = tg_digit(r, r);
  }
}

// complex element q of vector row of X (nx vectors of nq elements, the tile's first at x0)
template <int P>
__device__ __forceinline__ uint4 tg_load(const void* X, int nx, int row, size_t nq, size_t q) {
  if (row >= nx || q >= nq) return make_uint4(0u, 0u, 0u, 0u);
  if constexpr (P == P64) {
    return __ldg(reinterpret_cast<const uint4*>(X) + (size_t)row * nq + q);
  } else {
    const uint2 w = __ldg(reinterpret_cast<const uint2*>(X) + (size_t)row * nq + q);
    return make_uint4(w.x, w.y, 0u, 0u);
  }
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// the scale exponent e of a vector (every |x| < 2^e) from the largest binary exponent of its
// elements; a zero or subnormal-only vector reads as the minimum exponent field
template <int P>
__device__ __forceinline__ int tg_exponent(int raw) {
  return raw <= (P == P64 ? -1023 : -127) ? TG_EXP_ZERO : raw + 1;
}

}  // namespace

// Per vector: the largest binary exponent of its elements (ex starts at a very negative value).
// Many blocks per vector (one per vector read the operands of a 128 x 128 block at 1.2 TB/s, as
// long as the contraction itself), eight loads in flight per thread.
template <int P>
__global__ void __launch_bounds__(256) tc_gram_exp_kernel(const void* X, size_t nq, int* ex) {
  __shared__ int smax;
  if (threadIdx.x == 0) smax = INT_MIN;
  __syncthreads();
  const char* base = reinterpret_cast<const char*>(X) + (size_t)blockIdx.x * nq * tg_esize(P);
  int m = INT_MIN;
  const size_t step = (size_t)gridDim.y * blockDim.x;
  for (size_t q = (size_t)blockIdx.y * blockDim.x + threadIdx.x; q < nq; q += 8 * step) {
    int v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = q + u * step < nq ? TgLoad<P>::expo(base, q + u * step) : INT_MIN;
#pragma unroll
    for (int u = 0; u < 8; ++u) m = max(m, v[u]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(&smax, m);
  __syncthreads();
  if (threadIdx.x == 0) atomicMax(ex + blockIdx.x, smax);
}

// grid: (splits of the K range, A tiles x B tiles). partial: per CTA 2 x 64 x 64 doubles
// (Re rows, then Im rows), scaled by 2^(e_i + e_j).
template <int P>
__global__ void __launch_bounds__(TG_THREADS, 1)
    tc_gram_kernel(const void* A, int na, const void* B, int nb, size_t nq, int g5q, const int* exa, const int* exb,
                   double* partial, int* err, unsigned long long wait_ns) {
  extern __shared__ unsigned char sm_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>(((uintptr_t)sm_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint32_t tmem_base;
  __shared__ __align__(8) uint64_t full[TG_BUF], empty[TG_BUF], fbar, flushed, drain;
  __shared__ int abort_flag;
  __shared__ int ea_s[TG_NA], eb_s[TG_NB];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int split = blockIdx.x, nsplit = gridDim.x;
  const int ntb = (nb + TG_NB - 1) / TG_NB;
  const int ta = blockIdx.y / ntb, tb = blockIdx.y - ta * ntb;
  const int a0 = ta * TG_NA, b0 = tb * TG_NB;
  const size_t nstage_all = (nq + TG_KC - 1) / TG_KC;
  const size_t st0 = nstage_all * split / nsplit, st1 = nstage_all * (split + 1) / nsplit;
  const int nst = (int)(st1 - st0);

  if (tid < TG_NA) ea_s[tid] = a0 + tid < na ? tg_exponent<P>(exa[a0 + tid]) : TG_EXP_ZERO;
  else if (tid < TG_NA + TG_NB) eb_s[tid - TG_NA] = b0 + tid - TG_NA < nb ? tg_exponent<P>(exb[b0 + tid - TG_NA]) : TG_EXP_ZERO;
  if (tid == 0) {
    abort_flag = 0;
    for (int b = 0; b < TG_BUF; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[b])), "r"(TG_SLICERS));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[b])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&fbar)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&drain)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&flushed)), "r"(TG_THREADS / 32));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(TG_TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  // instruction descriptor: D F32, A and B BF16, both K-major, N = 64, M = 128
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TG_NB >> 3) << 17) | ((128u >> 4) << 24);

  // epilogue ownership: TMEM lane (row) 32 (warp % 4) + lane, columns 16 (warp / 4) .. + 15
  const int row = (warp & 3) * 32 + lane;
  const int cbase = (warp >> 2) * TG_CPT;
  float acc_h[TG_CPT], acc_l[TG_CPT];
#pragma unroll
  for (int c = 0; c < TG_CPT; ++c) acc_h[c] = acc_l[c] = 0.f;

  // One accumulation chunk's group sums are exact integers in FP32: the three smallest weights added
  // plainly (at most 2^-18: off by 2^-42 of a chunk whose digits are all at their bounds), the others in
  // double-float, then one double-float addition to the running sum, which stays normalised (|low| <=
  // half an ulp of high): however many chunks a CTA sums, each adds one rounding of 2^-48. Every
  // warp, once the chunk's MMAs are done (fbar); false when a wait gave up.
  auto flush = [&](int chunk) -> bool {
    if (!warp_wait(smem_u32(&fbar), (uint32_t)chunk & 1u, &abort_flag, wait_ns)) return false;
    asm volatile("tcgen05.fence::after_thread_sync;");
    constexpr int NC = 4;   // columns at a time: every group's sums loaded before one wait
#pragma unroll
    for (int c0 = 0; c0 < TG_CPT; c0 += NC) {
      uint32_t v[TG_G][NC];
      const uint32_t at = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(cbase + c0);
#pragma unroll
      for (int g = 0; g < TG_G; ++g)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(v[g][0]), "=r"(v[g][1]), "=r"(v[g][2]), "=r"(v[g][3])
                     : "r"(at + (uint32_t)(g * TG_NB)));
      // the wait names the registers: nothing that uses them moves above it
      static_assert(TG_G == 7 && NC == 4, "the wait below lists 28 registers");
      asm volatile("tcgen05.wait::ld.sync.aligned;"
                   : "+r"(v[0][0]), "+r"(v[0][1]), "+r"(v[0][2]), "+r"(v[0][3]), "+r"(v[1][0]), "+r"(v[1][1]),
                     "+r"(v[1][2]), "+r"(v[1][3]), "+r"(v[2][0]), "+r"(v[2][1]), "+r"(v[2][2]), "+r"(v[2][3]),
                     "+r"(v[3][0]), "+r"(v[3][1]), "+r"(v[3][2]), "+r"(v[3][3]), "+r"(v[4][0]), "+r"(v[4][1]),
                     "+r"(v[4][2]), "+r"(v[4][3]), "+r"(v[5][0]), "+r"(v[5][1]), "+r"(v[5][2]), "+r"(v[5][3]),
                     "+r"(v[6][0]), "+r"(v[6][1]), "+r"(v[6][2]), "+r"(v[6][3])::"memory");
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        auto x = [&](int g) {   // exact: times 2^(-7 (g + 2))
          return __uint_as_float(v[g][c]) * __int_as_float((127 - 7 * (g + 2)) << 23);
        };
        float ch = x(3), cl = (x(6) + x(5)) + x(4);
        cl += two_sum(ch, x(2));
        cl += two_sum(ch, x(1));
        cl += two_sum(ch, x(0));
        float &h = acc_h[c0 + c], &l = acc_l[c0 + c];
        l = two_sum(h, ch) + (l + cl);
        const float r = h + l;
        l -= r - h;
        h = r;
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&flushed));
    return true;
  };
  const int nchunk = (nst + TG_CHUNK - 1) / TG_CHUNK;
  bool ok = true;
  if (warp == 0) {
    for (int it = 0; ok && it < nst; ++it) {
      const int s = it % TG_BUF, cs = it % TG_CHUNK;
      ok = warp_wait(smem_u32(&full[s]), (uint32_t)(it / TG_BUF) & 1u, &abort_flag, wait_ns);
      // the accumulators restart: the last chunk must have been read out
      if (ok && cs == 0 && it > 0) ok = flush(it / TG_CHUNK - 1);
      if (ok && cs == 0 && it > 0)
        ok = warp_wait(smem_u32(&flushed), (uint32_t)(it / TG_CHUNK - 1) & 1u, &abort_flag, wait_ns);
      if (!ok) break;
      if (lane == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        // descriptors of digit 0, K-step 0 of this stage; the others differ only in the start
        // address (field in the low bits, in units of 16 bytes; no carry out of it below 256 KB)
        unsigned char* stA = sm + s * TG_STAGE;
        const uint64_t da0 = smem_desc(smem_u32(stA), 2048, 128),
                       db0 = smem_desc(smem_u32(stA + TG_S * TG_TILE_A), 1024, 128);
        const uint32_t acc_chunk = cs > 0 ? 1u : 0u;
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {   // two K-steps of 16 reals (2 core-matrix columns each)
#pragma unroll
          for (int g = 0; g < TG_G; ++g) {         // group g + 2 = s + t
            const int first = g > TG_S - 1 ? g - TG_S + 1 : 0;
#pragma unroll
            for (int ds = first; ds <= (g < TG_S - 1 ? g : TG_S - 1); ++ds) {
              // digit ds of A, g - ds of B (0-based); the first pair of a group starts its sum
              const uint64_t da = da0 + (uint64_t)((ds * TG_TILE_A + kk * 2 * 2048) >> 4);
              const uint64_t db = db0 + (uint64_t)(((g - ds) * TG_TILE_B + kk * 2 * 1024) >> 4);
              mma_bf16(tmem + (uint32_t)(g * TG_NB), da, db, idesc, (kk > 0 || ds > first) ? 1u : acc_chunk);
            }
          }
        }
        mma_commit(smem_u32(&empty[s]));
        if (cs == TG_CHUNK - 1 || it == nst - 1) mma_commit(smem_u32(&fbar));
      }
      __syncwarp();
    }
    if (ok && nst > 0) ok = flush(nchunk - 1);
  } else {
    // Slicing: 64 tasks of 32 elements (8 rows x 4 of the stage's 16 columns), 32 of A and 32 of B.
    // The next stage's elements are loaded while this one's are sliced.
    const int rl = lane >> 2, kp = lane & 3;
    uint4 raw[TG_TASKS];
    auto load = [&](int i, int it) {
      const int task = warp - 1 + i * TG_SLICERS;
      if (task >= 64 || it >= nst) return;
      const int tt = task & 31, r = (tt >> 2) * 8 + rl;
      const size_t q = (st0 + it) * TG_KC + (tt & 3) * 4 + kp;
      raw[i] = task < 32 ? tg_load<P>(A, na, a0 + r, nq, q) : tg_load<P>(B, nb, b0 + r, nq, q);
    };
#pragma unroll
    for (int i = 0; i < TG_TASKS; ++i) load(i, 0);
    for (int it = 0; ok && it < nst; ++it) {
      const int s = it % TG_BUF;
      if (it >= TG_BUF) ok = warp_wait(smem_u32(&empty[s]), (uint32_t)(it / TG_BUF - 1) & 1u, &abort_flag, wait_ns);
      if (!ok) break;
      unsigned char* stA = sm + s * TG_STAGE;
      unsigned char* stB = stA + TG_S * TG_TILE_A;
      const size_t q0 = (st0 + it) * TG_KC;
#pragma unroll
      for (int i = 0; i < TG_TASKS; ++i) {
        const int task = warp - 1 + i * TG_SLICERS;
        if (task >= 64) break;
        const int tt = task & 31, rg = tt >> 2, kc = tt & 3, r = rg * 8 + rl, j = kc * 4 + kp;
        const uint4 w = raw[i];
        load(i, it + 1);
        uint32_t pd[TG_S];   // digit s of (re, im) as a BF16 pair
        if (task < 32) {
          tg_digits<P>(w, ea_s[r], false, pd);
          // A row r and A' row 64 + r: (re, im) and (-im, re)
          const uint32_t off = (uint32_t)((kc * 16 + rg) * 128 + rl * 16 + kp * 4);
#pragma unroll
          for (int d = 0; d < TG_S; ++d) {
            *reinterpret_cast<uint32_t*>(stA + d * TG_TILE_A + off) = pd[d];
            *reinterpret_cast<uint32_t*>(stA + d * TG_TILE_A + off + 8 * 128) = __byte_perm(pd[d], 0u, 0x1032) ^ 0x8000u;
          }
        } else {
          tg_digits<P>(w, eb_s[r], g5q && q0 + j >= (size_t)g5q, pd);
          const uint32_t off = (uint32_t)((kc * 8 + rg) * 128 + rl * 16 + kp * 4);
#pragma unroll
          for (int d = 0; d < TG_S; ++d) *reinterpret_cast<uint32_t*>(stB + d * TG_TILE_B + off) = pd[d];
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&full[s]));
      // the previous chunk is read out two stages into the next one, while its last MMAs run
      if (it % TG_CHUNK == 1 && it > TG_CHUNK) ok = flush(it / TG_CHUNK - 1);
    }
    // what is left: the chunk before the last when the last one has a single stage, and the last
    if (ok && nst > TG_CHUNK && nst % TG_CHUNK == 1) ok = flush(nchunk - 2);
    if (ok && nst > 0) ok = flush(nchunk - 1);
  }
  if (!ok) abort_flag = 1;
  __syncthreads();
  // after an abort, MMAs still in flight must not outlive the tensor memory: one more bounded
  // wait for a commit that covers all of them
  if (abort_flag && tid == 0) {
    mma_commit(smem_u32(&drain));
    mbar_wait(smem_u32(&drain), 0u, nullptr, TG_DRAIN_NS);
  }
  __syncthreads();
  if (abort_flag && tid == 0) atomicExch(err, 1);
  if (!abort_flag) {
    const int i = row & 63, reim = row >> 6;
    const int ei = ea_s[i];
    double* out = partial + ((size_t)blockIdx.y * nsplit + split) * 2 * TG_NA * TG_NB + (size_t)reim * TG_NA * TG_NB +
                  (size_t)i * TG_NB;
#pragma unroll
    for (int c = 0; c < TG_CPT; ++c) {
      const int ej = eb_s[cbase + c];
      const double v = (ei == TG_EXP_ZERO || ej == TG_EXP_ZERO) ? 0.0
                                                               : ldexp((double)acc_h[c] + (double)acc_l[c], ei + ej);
      out[cbase + c] = v;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TG_TMEM_COLS));
}

// G[i][j] += sum over the splits (FP64, fixed order)
__global__ void tc_gram_reduce_kernel(const double* partial, int na, int nb, int nsplit, double* G) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= na * nb) return;
  const int i = e / nb, j = e - i * nb;
  const int ntb = (nb + TG_NB - 1) / TG_NB;
  const int tile = (i / TG_NA) * ntb + j / TG_NB;
  const int ri = i % TG_NA, cj = j % TG_NB;
  double re = 0.0, im = 0.0;
  for (int s = 0; s < nsplit; ++s) {
    const double* p = partial + ((size_t)tile * nsplit + s) * 2 * TG_NA * TG_NB;
    re += p[(size_t)ri * TG_NB + cj];
    im += p[(size_t)TG_NA * TG_NB + (size_t)ri * TG_NB + cj];
  }
  G[2 * e] += re;
  G[2 * e + 1] += im;
}

// Both sides of one precision: an FP64 field holds one component per 16-byte chunk and an FP32 field
// two, so element q of the one is not the component and site of element q of the other.
bool tc_gram_supported(int pa, int pb) { return pa == pb && (pa == P64 || pa == P32); }

int tc_gram_splits(int na, int nb, int V, int nsm) {
  const int tiles = ((na + TG_NA - 1) / TG_NA) * ((nb + TG_NB - 1) / TG_NB);
  const long long nstage = ((long long)12 * V + TG_KC - 1) / TG_KC;
  // whole splits in one wave of one CTA per SM: rounding up left a second wave of a single CTA
  // for 9 tiles (192 x 192: 153 CTAs on 152 SMs, twice the time)
  long long ns = nsm / tiles;
  const long long maxs = (nstage + TG_CHUNK - 1) / TG_CHUNK;   // at least one chunk per split
  if (ns > maxs) ns = maxs;
  if (ns < 1) ns = 1;
  return (int)ns;
}

size_t tc_gram_work_doubles(int na, int nb, int nsplit) {
  const size_t tiles = (size_t)((na + TG_NA - 1) / TG_NA) * ((nb + TG_NB - 1) / TG_NB);
  return tiles * nsplit * 2 * TG_NA * TG_NB;
}

// A (na vectors), B (nb vectors): fields of precision p (P64 or P32), 12 V complex elements
// each in the library layout (gamma5 negates the elements from 6 V on). G: na x nb complex
// FP64 (device), accumulated.
// partial: tc_gram_work_doubles doubles; ex: na + nb ints; err: device int set to 1 when a
// bounded wait gives up (after wait_ns).
void launch_tc_gram(int p, const void* A, int na, const void* B, int nb, int V, int g5, int nsplit, double* G,
                    double* partial, int* ex, int* err, unsigned long long wait_ns, cudaStream_t st) {
  const size_t nq = (size_t)12 * V;
  int* exa = ex;
  int* exb = ex + na;
  cudaMemsetAsync(ex, 0x80, sizeof(int) * (na + nb), st);   // about -2.1e9: below every exponent
  // enough blocks to fill the chip whatever the number of vectors, and at least 16 elements a thread
  auto blocks = [&](int n) {
    return (unsigned)std::max<size_t>(1, std::min<size_t>((1216 + n - 1) / n, (nq + 4095) / 4096));
  };
  const int tiles = ((na + TG_NA - 1) / TG_NA) * ((nb + TG_NB - 1) / TG_NB);
  dim3 grid((unsigned)nsplit, (unsigned)tiles);
  const int g5q = g5 ? (int)(6 * (size_t)V) : 0;
#define TG(P)                                                                                      \
  do {                                                                                             \
    tc_gram_exp_kernel<P><<<dim3(na, blocks(na)), 256, 0, st>>>(A, nq, exa);                       \
    tc_gram_exp_kernel<P><<<dim3(nb, blocks(nb)), 256, 0, st>>>(B, nq, exb);                       \
    cudaFuncSetAttribute(tc_gram_kernel<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, TG_SMEM); \
    tc_gram_kernel<P><<<grid, TG_THREADS, TG_SMEM, st>>>(A, na, B, nb, nq, g5q, exa, exb, partial, err, wait_ns); \
  } while (0)
  if (p == P64) TG(P64);
  else TG(P32);
#undef TG
  const int nn = na * nb;
  tc_gram_reduce_kernel<<<(nn + 255) / 256, 256, 0, st>>>(partial, na, nb, nsplit, G);
}

}  // namespace ovl
