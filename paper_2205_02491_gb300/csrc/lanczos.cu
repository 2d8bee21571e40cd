// Lanczos spectral-bound estimation (Algorithm 1, line 2) on the device.
//
// All runs advance together, two launches per step: the product of A with one vector per run (hemv_kernel, or
// hemv_dfma_kernel in the native mode; A streamed once per step), and the rest of the step (lanczos_step_kernel, one cluster of CTAs per run): three-term
// update, one classical Gram-Schmidt reorthogonalisation against the run's basis, normalisation.  The tridiagonal T
// of each run is diagonalised by one block per run, and one block computes b_sup = max(theta_max + |beta_last|),
// mu_1 = min theta_min, theta_max and the density-of-states quantile mu_ne = smallest pooled Ritz value whose
// cumulative weight (1/runs) sum tau_j^2 reaches ne/n, clamped into (mu_1, b_sup) by 1e-3 of the spectral span.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "common.cuh"
#include "kernels.h"
#include "tcgen05.cuh"

namespace chase {

constexpr int LZ_MAXR = 8;      // runs
constexpr int LZ_MAXS = 64;     // steps

// ---------------------------------------------------------------- fixed-point operands
// An entry x of a vector with |x| < 2^e is held as r = round(x 2^(54 - e)), |r| <= 2^54, in balanced base-256 digits
// r = sum_t d_t 256^t, t = 0..6, d_t in [-128, 127]: adding 128 to every digit makes them the bytes of an integer.  An
// entry of A is cut to 56 bits and a sign, seven plain base-256 digits: most of the work is cutting A, once per step.
constexpr int LZ_NONFINITE = 0x7fffffff;
constexpr int NDIG = 7;
constexpr unsigned long long DIGIT_BIAS = 0x80808080808080ull;
__device__ __forceinline__ long long to_fixed(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int be = (int)((b >> 52) & 0x7ff);
  long long m = b & 0xfffffffffffffll;
  if (be != 0) m |= 0x10000000000000ll;
  const int sh = (be != 0 ? be : 1) - 1075 + 54 - e;
  long long r;
  if (sh >= 0) {
    r = m << (sh < 1 ? sh : 1);
  } else {
    const int rs = sh > -62 ? -sh : 62;
    r = ((m >> (rs - 1)) + 1) >> 1;
  }
  return b < 0 ? -r : r;
}
// exponent e with |x| < 2^e from the largest magnitude's bit pattern (0: all zero)
__device__ __forceinline__ int exponent_of_bits(unsigned long long m) {
  if (m >= 0x7ff0000000000000ull) return LZ_NONFINITE;
  const int be = (int)(m >> 52);
  return (be != 0 ? be : 1) - 1022;
}
template <typename T> __device__ __forceinline__ unsigned long long magnitude_bits(T v) {
  const unsigned long long a = (unsigned long long)__double_as_longlong(fabs(S<T>::re(v)));
  const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(S<T>::im(v)));
  return a > b ? a : b;
}

// largest magnitude of every row of A (its bits' upper half is enough for the exponent): grid (rows, column chunks)
constexpr int ROWMAX_COLS = 128;
template <typename T>
__global__ void __launch_bounds__(128) row_max_kernel(int64_t n, const T* __restrict__ A, int64_t lda, unsigned* rmax) {
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (i >= n) return;
  const int64_t j0 = (int64_t)blockIdx.y * ROWMAX_COLS, j1 = j0 + ROWMAX_COLS < n ? j0 + ROWMAX_COLS : n;
  unsigned long long m = 0ull;
#pragma unroll 8
  for (int64_t j = j0; j < j1; ++j) {
    const unsigned long long v = magnitude_bits<T>(A[i + j * lda]);
    m = m > v ? m : v;
  }
  atomicMax(&rmax[i], (unsigned)(m >> 32));
}

// |x| 2^(56 - e) cut to an integer below 2^56 for |x| < 2^e, c = 1029 + e: the mantissa with its leading bit at 62, shifted
// right by c minus the biased exponent.  Exact zero for x = 0; subnormal x only with e below -966, which the caller scales.
__device__ __forceinline__ unsigned long long cut56(uint32_t lo, uint32_t hi, int c) {
  const uint32_t mh = (__funnelshift_l(lo, hi, 10) & 0x3fffffffu) | 0x40000000u;
  const uint32_t n = min((uint32_t)(c - (int)((hi >> 20) & 0x7ffu)), 63u);
  return ((unsigned long long)mh << 32 | (lo << 10)) >> n;
}
// base-256 digits t = 0..6 of two numbers as f16 pairs in units of 2^-24: a digit's byte with the number's sign bit is
// that f16 subnormal, exactly, without a conversion
__device__ __forceinline__ void digit_pairs(double x0, double x1, int c, uint32_t (&out)[NDIG]) {
  const uint32_t h0 = (uint32_t)__double2hiint(x0), h1 = (uint32_t)__double2hiint(x1);
  const unsigned long long r0 = cut56((uint32_t)__double2loint(x0), h0, c), r1 = cut56((uint32_t)__double2loint(x1), h1, c);
  const uint32_t sgn = __byte_perm(h0, h1, 0x7632) & 0x80008000u;
  const uint32_t l0 = (uint32_t)r0, l1 = (uint32_t)r1, u0 = (uint32_t)(r0 >> 32), u1 = (uint32_t)(r1 >> 32);
  const uint32_t p[3] = {__byte_perm(l0, l1, 0x5410), __byte_perm(l0, l1, 0x7632), __byte_perm(u0, u1, 0x5410)};
#pragma unroll
  for (int t = 0; t < 6; ++t) out[t] = ((t & 1 ? p[t >> 1] >> 8 : p[t >> 1]) & 0x00ff00ffu) | sgn;
  out[6] = __byte_perm(u0, u1, 0x7632) | sgn;
}

// Vectors as the products' right operand: for every 64 columns of A (rows of X) and form, 64 rows of 64 f16 digits in
// the 128-byte-swizzled K-major layout that the MMA reads, so that one bulk copy brings a block to shared memory.  Row
// (6 - u) 8 + c is digit u of vector column c (8 real columns: up to 8 runs; complex: re and im of up to 4).  Complex:
// form 0 multiplies Re A (columns re, im of each run), form 1 multiplies Im A (columns -im, re).
constexpr int HK = 64;                    // columns of A per block
constexpr int FORM_HALVES = 64 * HK;
template <typename T> struct Frag {
  static constexpr int FORMS = S<T>::cplx ? 2 : 1;
  static constexpr int RUNS = S<T>::cplx ? 4 : 8;       // runs per group of 8 columns
  static constexpr int BLOCK_HALVES = FORMS * FORM_HALVES;
};
inline int64_t frag_halves(int64_t n, bool cplx, int runs) {
  const int per = cplx ? 4 : 8;
  return (n + HK - 1) / HK * ((runs + per - 1) / per) * ((cplx ? 2 : 1) * FORM_HALVES);
}
// writes digit t = 0..6 of entry j of a run's vector
template <typename T>
__device__ __forceinline__ void write_frag(__half* X, int64_t nkb, int64_t j, int run, long long re, long long im) {
  using F = Frag<T>;
  const int grp = run / F::RUNS, r = run % F::RUNS, kk = (int)(j & (HK - 1));
  __half* base = X + ((int64_t)grp * nkb + j / HK) * F::BLOCK_HALVES;
  auto at = [&](int row) { return base + row * HK + (((kk >> 3) ^ (row & 7)) << 3) + (kk & 7); };
  unsigned long long wr = (unsigned long long)re + DIGIT_BIAS, wi = (unsigned long long)im + DIGIT_BIAS;
  for (int t = 0; t < NDIG; ++t, wr >>= 8, wi >>= 8) {
    const int row = (NDIG - 1 - t) * 8;
    const __half dr = __int2half_rn((int)(wr & 0xff) - 128);
    if (F::FORMS == 2) {
      const __half di = __int2half_rn((int)(wi & 0xff) - 128);
      __half* c0 = at(row + 2 * r);
      __half* c1 = at(row + 2 * r + 1);
      c0[0] = dr;
      c1[0] = di;
      c0[FORM_HALVES] = __hneg(di);
      c1[FORM_HALVES] = dr;
    } else {
      *at(row + r) = dr;
    }
  }
}

// part[c][r][i] = sum_{j in chunk c} A[i,j] X[j,r] for up to 8 real columns (4 complex runs, re and im interleaved).
// FP64 multiply-adds bound a plain version (GB300: 2 per SM and clock; four complex vectors take 16 per element of A,
// 1.78 ms at n = 8192 where reading A takes 0.16 ms).  Here both are fixed-point numbers in seven 8-bit digits,
// multiplied on the tensor cores (f16 digits, FP32 sums).  With mma.sync the 34 digit pairs that count bound it (0.44
// ms).  tcgen05 takes digit t of A (128 rows x 16 columns in TMEM) against all digits of X at once: X's digits are the
// MMA's columns, and accumulator columns of one level t + u coincide when digit t's window starts 6 - t groups of 8
// columns along, so seven MMAs per form do all pairs; levels past 7 (below 2^-56 of the scales' product) fall into
// columns nobody reads.  Sums are exact over 32 columns (at most 7 pairs x 2 planes x 32 products of 255 x 128 < 2^24),
// then go to integers (at most 128 of them).
// Warps 0-3 add up the accumulators; warps 4-11 (two groups of 128 threads, one row per thread, alternating 16-column
// steps) make digits in registers and store them to their group's TMEM operand; warp 12 issues MMAs, warp 13 copies X.
// Each thread brings its own entries of A through shared memory with cp.async (64 KB in flight per SM), so no barrier
// guards them.  Registers: 512 threads at 128; the sums take 160, the digits 136, the rest keep 80.
// What bounds it: the integer instructions that cut A's entries into digits, next to the HBM time: complex, n = 8192,
// 4 runs: 208 us a step (5.2 TB/s), 436 with mma.sync.
constexpr int HEMV_ROWS = 128;
constexpr int HEMV_THREADS = 512;        // warps 14, 15 idle: whole warpgroups
constexpr int HSTEP = 16;                // columns per MMA step
constexpr int H_XSTAGES = 4;
constexpr int NLEV = 8;
constexpr int H_ACC = 80;                // TMEM columns per accumulator: 72 written
constexpr int H_A0 = 2 * H_ACC;          // then one operand per producer group
constexpr int H_ASLOT = 2 * NDIG * 8;    // 14 digit planes of 8 columns
constexpr unsigned long long H_DRAIN_NS = 2000000000ull;  // limit of the waits for copies and MMAs in flight at the end
constexpr int LZ_STATUS_QL = 1, LZ_STATUS_WAIT = 2;       // bits of the status word: no QL convergence, a wait ran out
template <typename T> struct Hemv {
  static constexpr int SLOTS = S<T>::cplx ? 2 : 4;                            // steps of A in flight per thread
  static constexpr int A_BYTES = SLOTS * 2 * HSTEP * 128 * (int)sizeof(T);   // 128 KB
  static constexpr int X_BYTES = Frag<T>::BLOCK_HALVES * 2;
  static constexpr int SMEM = 1024 + H_XSTAGES * X_BYTES + A_BYTES + 256;
};

// bounded wait: false after wait_ns or when another role gave up
__device__ __forceinline__ bool hemv_wait(uint32_t bar, uint32_t parity, volatile int* gave_up, unsigned long long wait_ns) {
  unsigned long long t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (oz::mbar_try(bar, parity)) return true;
    if ((it & 255) == 255) {
      if (*gave_up) return false;
      const unsigned long long t = oz::globaltimer();
      if (t0 == 0) t0 = t;
      else if (t - t0 > wait_ns) {
        *gave_up = 1;
        return false;
      }
    }
  }
}
// D (+)= A B, A (f16, 128 x 16) in TMEM
__device__ __forceinline__ void mma_tmem_a(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void tmem_st(uint32_t a, const uint32_t (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
               : "memory");
}
__device__ __forceinline__ void tmem_st(uint32_t a, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(a), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
// 16 accumulator columns; the wait takes the registers in and out, so that no use moves before it
__device__ __forceinline__ void tmem_ld16(uint32_t a, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(a));
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                 "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

template <typename T>
__global__ void __launch_bounds__(HEMV_THREADS, 1) hemv_kernel(int64_t n, const T* __restrict__ A, int64_t lda,
                                                                const unsigned* __restrict__ rmax,
                                                                const __half* __restrict__ X,
                                                                const int* __restrict__ xe, int cols, int runs, T* part,
                                                                unsigned long long wait_ns, int* status) {
  using s = S<T>;
  using F = Frag<T>;
  using H = Hemv<T>;
  using oz::smem_u32;
  extern __shared__ __align__(1024) unsigned char hemv_smem[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)hemv_smem + 1023) & ~(uintptr_t)1023);
  unsigned char* abuf = smem + H_XSTAGES * H::X_BYTES;
  uint64_t* xfull = (uint64_t*)(abuf + H::A_BYTES);  // a block of X has landed
  uint64_t* xempty = xfull + H_XSTAGES;              // its MMAs are done
  uint64_t* afull = xempty + H_XSTAGES;              // a group's digits are in TMEM
  uint64_t* aempty = afull + 2;                      // their MMAs are done
  uint64_t* dfull = aempty + 2;                      // an accumulator is complete
  uint64_t* dempty = dfull + 2;                      // it has been read
  uint64_t* drain = dempty + 2;
  uint32_t* tmem_slot = (uint32_t*)(drain + 1);
  volatile int* gave_up = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < H_XSTAGES; ++i) {
      oz::mbar_init(smem_u32(&xfull[i]), 1);
      oz::mbar_init(smem_u32(&xempty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      oz::mbar_init(smem_u32(&afull[i]), 4);
      oz::mbar_init(smem_u32(&aempty[i]), 1);
      oz::mbar_init(smem_u32(&dfull[i]), 1);
      oz::mbar_init(smem_u32(&dempty[i]), 4);
    }
    oz::mbar_init(smem_u32(drain), 1);
    // a limit below a microsecond, less than any wait for memory takes, has run out before the first one
    *gave_up = wait_ns < 1000ull;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  oz::fence_before();
  __syncthreads();
  oz::fence_after();
  grid_dependency_wait();
  const uint32_t tmem = *tmem_slot;

  const int64_t row = (int64_t)blockIdx.x * HEMV_ROWS + (warp & 3) * 32 + lane;  // warps 0-11
  const int64_t jbeg = (int64_t)blockIdx.y * cols, jend = jbeg + cols < n ? jbeg + cols : n;
  const int grp = blockIdx.z;
  const int nblk = (int)((jend - jbeg + HK - 1) / HK);  // blocks of 64 columns
  const int ea = row < n && warp < 12 ? exponent_of_bits((unsigned long long)rmax[row] << 32 | 0xffffffffull) : 0;
  const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);

  if (warp < 4) {
    // ------------------------------------------------------------ sums of the accumulators
    asm volatile("setmaxnreg.inc.sync.aligned.u32 160;");
    int sum[NLEV][8];
#pragma unroll
    for (int l = 0; l < NLEV; ++l)
#pragma unroll
      for (int q = 0; q < 8; ++q) sum[l][q] = 0;
    bool ok = true;
    for (int k = 0; k < 2 * nblk; ++k) {
      const int b = k & 1;
      ok = __all_sync(0xffffffffu, hemv_wait(smem_u32(&dfull[b]), (k >> 1) & 1, gave_up, wait_ns));
      if (!ok) break;
      oz::fence_after();
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        uint32_t r[16];
        tmem_ld16(lane_addr + (uint32_t)(b * H_ACC + h * 16), r);
#pragma unroll
        for (int q = 0; q < 16; ++q) sum[2 * h + (q >> 3)][q & 7] += __float2int_rn(__uint_as_float(r[q]) * 16777216.0f);
      }
      oz::fence_before();
      __syncwarp();
      if (lane == 0) oz::mbar_arrive(smem_u32(&dempty[b]));
    }
    // levels 0-3 and 4-7 as two integers; value = (hi 2^32 + lo) 2^40, in units of 2^(ea + ex - 110)
    if (row < n) {
      double o[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const long long hi = ((long long)sum[0][q] << 24) + ((long long)sum[1][q] << 16) + ((long long)sum[2][q] << 8) + sum[3][q];
        const long long lo = ((long long)sum[4][q] << 24) + ((long long)sum[5][q] << 16) + ((long long)sum[6][q] << 8) + sum[7][q];
        o[q] = (double)hi * 4294967296.0 + (double)lo;
      }
      T* out = part + (int64_t)blockIdx.y * runs * n + row;
#pragma unroll
      for (int q = 0; q < F::RUNS; ++q) {
        const int run = grp * F::RUNS + q;
        if (run >= runs) break;
        const int ex = xe[run];
        const bool bad = !ok || ea == LZ_NONFINITE || ex == LZ_NONFINITE;  // also a wait that ran out
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        const int c = F::FORMS * q;
        const double re = bad ? nan : ldexp(o[c], ea + ex - 70);
        const double im = F::FORMS == 1 ? 0.0 : bad ? nan : ldexp(o[c + F::FORMS - 1], ea + ex - 70);
        out[(int64_t)run * n] = s::make(re, im);
      }
    }
  } else if (warp < 12) {
    // ------------------------------------------------------------ digits of A
    asm volatile("setmaxnreg.inc.sync.aligned.u32 136;");
    const int g = (warp >> 2) - 1;
    const uint32_t dst = lane_addr + (uint32_t)(H_A0 + g * H_ASLOT);
    constexpr int ESZ = (int)sizeof(T), UNIT = 16 / F::FORMS;  // columns per pass (56 registers of digits)
    const uint32_t buf = smem_u32(abuf) + (uint32_t)((g * HSTEP * 128 + (warp & 3) * 32 + lane) * ESZ);
    const int count = 2 * nblk;  // this group's steps: columns jbeg + 16 (2 it + g) ...
    // rows of tiny entries (subnormal ones cannot be cut) are scaled by 2^600 first
    const bool tiny = ea < -900, any_tiny = __any_sync(0xffffffffu, tiny);
    const double up = tiny ? 4.149515568880993e180 : 1.0;
    const int c0 = 1029 + (ea == LZ_NONFINITE ? 0 : tiny ? ea + 600 : ea);
    const T* src = A + (row < n ? row : 0) + (jbeg + HSTEP * g) * lda;
    auto copy = [&](uint32_t to, const T* p, int bytes) {
      if (ESZ == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(p), "r"(bytes) : "memory");
      else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(to), "l"(p), "r"(bytes) : "memory");
    };
    auto issue = [&](int it) {
      const int64_t j = jbeg + (int64_t)HSTEP * (2 * it + g);
      const uint32_t to = buf + (uint32_t)(it % H::SLOTS * (2 * HSTEP * 128 * ESZ));
      if (j + HSTEP <= jend && row < n) {
        const T* p = src;
#pragma unroll
        for (int q = 0; q < HSTEP; ++q, p += lda) copy(to + (uint32_t)(q * 128 * ESZ), p, ESZ);
      } else if (it < count) {  // zeros outside the matrix
#pragma unroll 1
        for (int q = 0; q < HSTEP; ++q) {
          const bool in = row < n && j + q < jend;
          copy(to + (uint32_t)(q * 128 * ESZ), in ? src + q * lda : A, in ? ESZ : 0);
        }
      }
      src += 2 * HSTEP * lda;
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int it = 0; it < H::SLOTS - 1; ++it) issue(it);
    for (int it = 0; it < count; ++it) {
      issue(it + H::SLOTS - 1);
      asm volatile("cp.async.wait_group %0;" ::"n"(H::SLOTS - 1) : "memory");
      const uint32_t from = buf + (uint32_t)(it % H::SLOTS * (2 * HSTEP * 128 * ESZ));
      if (any_tiny) {  // a loop of its own: inline, its FP64 multiplications are issued for every entry and bound the kernel
#pragma unroll 1
        for (int q = 0; q < HSTEP * F::FORMS; ++q) {
          const uint32_t at = from + (uint32_t)((q / F::FORMS) * 128 * ESZ + (q % F::FORMS) * 8);
          double v;
          asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(at) : "memory");
          asm volatile("st.shared.f64 [%0], %1;" ::"r"(at), "d"(v * up) : "memory");
        }
      }
      bool ok = true;
#pragma unroll
      for (int h = 0; h < F::FORMS; ++h) {
        uint32_t dig[F::FORMS][NDIG][UNIT / 2];
#pragma unroll
        for (int c = 0; c < UNIT; c += 2) {
          double x[2][2];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const uint32_t at = from + (uint32_t)((h * UNIT + c + k) * 128 * ESZ);
            if (F::FORMS == 2)
              asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(x[k][0]), "=d"(x[k][1]) : "r"(at) : "memory");
            else
              asm volatile("ld.shared.f64 %0, [%1];" : "=d"(x[k][0]) : "r"(at) : "memory");
          }
#pragma unroll
          for (int f = 0; f < F::FORMS; ++f) {
            uint32_t d[NDIG];
            digit_pairs(x[0][f], x[1][f], c0, d);
#pragma unroll
            for (int t = 0; t < NDIG; ++t) dig[f][t][c / 2] = d[t];
          }
        }
        if (h == 0) {
          ok = __all_sync(0xffffffffu, hemv_wait(smem_u32(&aempty[g]), (it & 1) ^ 1, gave_up, wait_ns));
          if (!ok) break;
          oz::fence_after();
        }
#pragma unroll
        for (int f = 0; f < F::FORMS; ++f)
#pragma unroll
          for (int t = 0; t < NDIG; ++t) tmem_st(dst + (uint32_t)((f * NDIG + t) * 8 + h * (UNIT / 2)), dig[f][t]);
      }
      if (!ok) break;
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      oz::fence_before();
      __syncwarp();
      if (lane == 0) oz::mbar_arrive(smem_u32(&afull[g]));
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
    if (warp == 12 && lane == 0) {
      // ------------------------------------------------------------ MMA issue
      bool ok = true;
      for (int kb = 0; kb < nblk && ok; ++kb) {
        const int st = kb % H_XSTAGES;
        ok = hemv_wait(smem_u32(&xfull[st]), (kb / H_XSTAGES) & 1, gave_up, wait_ns);
        if (!ok) break;
        const uint64_t xd = oz::sw128_desc(smem_u32(smem + st * H::X_BYTES));
#pragma unroll 1
        for (int k = 0; k < HK / HSTEP; ++k) {
          // accumulator: two steps each
          const int g = k & 1, b = k >> 1, it = 2 * kb + (k >> 1);
          ok = (g != 0 || hemv_wait(smem_u32(&dempty[b]), (kb & 1) ^ 1, gave_up, wait_ns)) &&
               hemv_wait(smem_u32(&afull[g]), it & 1, gave_up, wait_ns);
          if (!ok) break;
          oz::fence_after();
#pragma unroll
          for (int f = 0; f < F::FORMS; ++f)
#pragma unroll
            for (int t = NDIG - 1; t >= 0; --t) {
              // digit t's window: levels 6 - t .. 7, in MMAs of a multiple of 16 columns
              const int first = NDIG - 1 - t, groups = NLEV - first;
              const int N = (groups * 8 + 15) / 16 * 16;
              const uint32_t idesc = (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(HEMV_ROWS >> 4) << 24);
              mma_tmem_a(tmem + (uint32_t)(b * H_ACC + first * 8), tmem + (uint32_t)(H_A0 + g * H_ASLOT + (f * NDIG + t) * 8),
                         xd + (uint64_t)(f * (FORM_HALVES * 2 >> 4) + k * (HSTEP * 2 >> 4)), idesc,
                         g == 0 && f == 0 && t == NDIG - 1 ? 0u : 1u);
            }
          oz::mma_commit(smem_u32(&aempty[g]));
          if (g == 1) oz::mma_commit(smem_u32(&dfull[b]));
        }
        if (ok) oz::mma_commit(smem_u32(&xempty[st]));
      }
      // every MMA is done before TMEM is freed
      oz::mma_commit(smem_u32(drain));
      const unsigned long long t0 = oz::globaltimer();
      while (!oz::mbar_try(smem_u32(drain), 0) && oz::globaltimer() - t0 < H_DRAIN_NS) {
      }
    } else if (warp == 13 && lane == 0) {
      // ------------------------------------------------------------ copies of X
      const int64_t nkb = (n + HK - 1) / HK;
      const __half* src = X + ((int64_t)grp * nkb + jbeg / HK) * F::BLOCK_HALVES;
      int issued = 0;
      for (; issued < nblk; ++issued) {
        const int st = issued % H_XSTAGES;
        if (!hemv_wait(smem_u32(&xempty[st]), ((issued / H_XSTAGES) & 1) ^ 1, gave_up, wait_ns)) break;
        oz::mbar_expect_tx(smem_u32(&xfull[st]), H::X_BYTES);
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         smem_u32(smem + st * H::X_BYTES)),
                     "l"(src + (int64_t)issued * F::BLOCK_HALVES), "r"(H::X_BYTES), "r"(smem_u32(&xfull[st]))
                     : "memory");
      }
      // the copies in flight land before the CTA exits
      for (int i = issued > H_XSTAGES ? issued - H_XSTAGES : 0; i < issued; ++i) {
        const unsigned long long t0 = oz::globaltimer();
        while (!oz::mbar_try(smem_u32(&xfull[i % H_XSTAGES]), (i / H_XSTAGES) & 1) && oz::globaltimer() - t0 < H_DRAIN_NS) {
        }
      }
    }
  }
  __syncwarp();
  oz::fence_before();
  __syncthreads();
  oz::fence_after();
  if (threadIdx.x == 0 && *gave_up) atomicOr(status, LZ_STATUS_WAIT);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// The same by FP64 multiply-adds on the full entries, for the native mode, whose results rest on plain FP64 arithmetic only:
// R real or complex vectors (X, ld ldx), one row per thread, X staged 128 columns at a time.  The FP64 rate bounds it: complex,
// n = 8192, 4 runs: 1.8 ms a step.
constexpr int DFMA_ROWS = 64, DFMA_COLS = 128;
template <typename T, int R>
__global__ void __launch_bounds__(DFMA_ROWS) hemv_dfma_kernel(int64_t n, const T* __restrict__ A, int64_t lda,
                                                               const T* __restrict__ X, int64_t ldx, int cols, T* part) {
  grid_dependency_wait();
  using s = S<T>;
  __shared__ T xs[DFMA_COLS][R];
  const int64_t i = (int64_t)blockIdx.x * DFMA_ROWS + threadIdx.x;
  const int64_t jbeg = (int64_t)blockIdx.y * cols, jend = jbeg + cols < n ? jbeg + cols : n;
  T acc[R];
#pragma unroll
  for (int r = 0; r < R; ++r) acc[r] = s::zero();
  for (int64_t j0 = jbeg; j0 < jend; j0 += DFMA_COLS) {
    const int nj = (int)(jend - j0 < DFMA_COLS ? jend - j0 : DFMA_COLS);
    __syncthreads();
    for (int t = threadIdx.x; t < DFMA_COLS * R; t += DFMA_ROWS)
      xs[t / R][t % R] = t / R < nj ? X[j0 + t / R + (t % R) * ldx] : s::zero();
    __syncthreads();
    if (i >= n) continue;
    const T* a = A + i + j0 * lda;
    constexpr int B = 16 / (int)(sizeof(T) / 8);  // loads in flight
    for (int j = 0; j < nj; j += B) {
      T v[B];
#pragma unroll
      for (int b = 0; b < B; ++b) v[b] = j + b < nj ? a[(j + b) * lda] : s::zero();
#pragma unroll
      for (int b = 0; b < B; ++b)
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = s::fma(v[b], xs[j + b][r], acc[r]);
    }
  }
  if (i >= n) return;
#pragma unroll
  for (int r = 0; r < R; ++r) part[((int64_t)blockIdx.y * R + r) * n + i] = acc[r];
}

template <typename T>
static void hemv_dfma(cudaStream_t st, int64_t n, const T* A, int64_t lda, const T* X, int64_t ldx, int cols, int runs, T* part) {
  const dim3 grid(ceil_div(n, DFMA_ROWS), ceil_div(n, cols));
  switch (runs) {
#define CASE(R) \
  case R: launch_pdl(hemv_dfma_kernel<T, R>, grid, DFMA_ROWS, 0, st, n, A, lda, X, ldx, cols, part); break;
    CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8)
#undef CASE
  }
  CHASE_CHECK_LAUNCH();
}

// Columns per hemv block (a multiple of 64): row blocks times column chunks in full waves of one block per SM, a block
// costing about two column blocks more than its columns (set-up, pipeline fill).  At most 64 column blocks (the
// integer sums) and, unless those need more, at most 608 blocks in all (the partial sums' space).
static int hemv_cols(int64_t n) {
  const int64_t rb = (n + HEMV_ROWS - 1) / HEMV_ROWS, kb = (n + HK - 1) / HK;
  const int64_t least = (kb + 63) / 64, most = std::max(least, std::min(kb, 608 / rb));
  int64_t best = least, cost = INT64_MAX;
  for (int64_t nc = least; nc <= most; ++nc) {
    const int64_t c = (rb * nc + 151) / 152 * ((kb + nc - 1) / nc + 2);
    if (c < cost) {
      cost = c;
      best = nc;
    }
  }
  return (int)((kb + best - 1) / best * HK);
}

// Bound of nchunk * n over all sizes up to n (the hemv partial sums of one run): 608 blocks' rows, or n rows per 4096
// columns.
static int64_t hemv_part_rows(int64_t n) { return std::max<int64_t>(608 * HEMV_ROWS, n * (n / 4096 + 1)); }

// vector fragments, row maxima, exponents
static int64_t operand_elems(int64_t n, int runs, bool cplx) {
  const int64_t scal = cplx ? 16 : 8;
  return (frag_halves(n, cplx, runs) * 2 + n * 4 + 512 + scal - 1) / scal + 16;
}

int64_t lanczos_work_elems(int64_t n, int runs, int steps, bool cplx) {
  // basis | W | hemv partial sums | operands
  return (int64_t)runs * steps * n + runs * n + runs * hemv_part_rows(n) + operand_elems(n, runs, cplx);
}

int64_t lanczos_context_elems(int64_t n, int64_t quota, bool cplx) {
  // the partial sums of n below 4464 take more than n rows per 256 columns, by 608 blocks' rows at most
  return quota + LZ_MAXR * 608ll * HEMV_ROWS + operand_elems(n, LZ_MAXR, cplx);
}

// ---------------------------------------------------------------- one step of every run
// One cluster of CTAs per run (blockIdx.y); CTA `rank` owns a contiguous block of rows.  Dots go one basis column per
// warp (one FP64 warp reduction per column and CTA); the CTAs' partial sums meet in distributed shared memory and
// every CTA adds them in rank order, so the result does not depend on scheduling.  FP64 multiply-adds bound it
// (8 per row and basis column), hence up to 16 SMs per run.
constexpr int STEP_THREADS = 512;
constexpr int STEP_MAXC = 16;

__device__ __forceinline__ unsigned cluster_ctas() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ double peer_double(const double* p, unsigned cta) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), ra;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(cta));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(ra) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long peer_bits(const unsigned long long* p, unsigned cta) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), ra;
  unsigned long long v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(cta));
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(ra) : "memory");
  return v;
}

// start: w = L0's column of the run, normalised into basis column 0 (j = -1)
template <typename T>
__global__ void __launch_bounds__(STEP_THREADS) lanczos_step_kernel(int64_t n, int runs, int steps, int j, int nchunk,
                                                                     const T* __restrict__ part,
                                                                     const T* __restrict__ L0, T* Vb, T* Wb,
                                                                     double* alpha, double* beta, __half* X, int* xe) {
  grid_dependency_wait();
  using s = S<T>;
  constexpr int NC = s::cplx ? 2 : 1;
  constexpr int NW = STEP_THREADS / 32;
  __shared__ double red[NW];
  __shared__ unsigned long long redm[NW];
  __shared__ double sh_alpha, sh_norm;           // this CTA's partial sums, read by its peers
  __shared__ unsigned long long sh_max;
  __shared__ double sh_dot[LZ_MAXS][NC];
  __shared__ T coef[LZ_MAXS];
  const unsigned nct = cluster_ctas(), rank = blockIdx.x;
  const int run = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t per = (n + nct - 1) / nct;
  const int64_t i0 = rank * per < n ? rank * per : n, i1 = i0 + per < n ? i0 + per : n;
  T* w = Wb + (int64_t)run * n;
  T* V = Vb + (int64_t)run * n * steps;
  double nrm = 0.0;
  unsigned long long mx = 0ull;
  if (j < 0) {
    for (int64_t i = i0 + tid; i < i1; i += STEP_THREADS) {
      const T v = L0[(int64_t)run * n + i];
      w[i] = v;
      nrm += s::abs2(v);
      const unsigned long long b = magnitude_bits<T>(v);
      mx = mx > b ? mx : b;
    }
  } else {
    // w = A v_j from the product's chunks; alpha = Re <v_j, w>
    double a = 0.0;
    for (int64_t i = i0 + tid; i < i1; i += STEP_THREADS) {
      T v = s::zero();
      for (int c = 0; c < nchunk; ++c) v = s::add(v, part[((int64_t)c * runs + run) * n + i]);
      w[i] = v;
      const T q = V[i + (int64_t)j * n];
      a += s::re(q) * s::re(v) + s::im(q) * s::im(v);
    }
    a = warp_sum(a);
    if (lane == 0) red[warp] = a;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int k = 0; k < NW; ++k) t += red[k];
      sh_alpha = t;
    }
    __syncthreads();
    cluster_barrier();
    double al = 0.0;
    for (unsigned c = 0; c < nct; ++c) al += peer_double(&sh_alpha, c);
    if (tid == 0 && rank == 0) alpha[run * LZ_MAXS + j] = al;
    const double bprev = j > 0 ? beta[run * LZ_MAXS + j - 1] : 0.0;
    for (int64_t i = i0 + tid; i < i1; i += STEP_THREADS) {
      T v = s::sub(w[i], s::scale(V[i + (int64_t)j * n], al));
      if (j > 0) v = s::sub(v, s::scale(V[i + (int64_t)(j - 1) * n], bprev));
      w[i] = v;
    }
    __syncthreads();
    // one full classical Gram-Schmidt pass against the run's basis
    for (int col = warp; col <= j; col += NW) {
      const T* q = V + (int64_t)col * n;
      T acc = s::zero();
#pragma unroll 4
      for (int64_t i = i0 + lane; i < i1; i += 32) acc = s::fmac(q[i], w[i], acc);
      const double re = warp_sum(s::re(acc));
      const double im = s::cplx ? warp_sum(s::im(acc)) : 0.0;
      if (lane == 0) {
        sh_dot[col][0] = re;
        if (NC == 2) sh_dot[col][NC - 1] = im;
      }
    }
    __syncthreads();
    cluster_barrier();
    for (int t = tid; t <= j; t += STEP_THREADS) {
      double re = 0.0, im = 0.0;
      for (unsigned c = 0; c < nct; ++c) {
        re += peer_double(&sh_dot[t][0], c);
        if (NC == 2) im += peer_double(&sh_dot[t][NC - 1], c);
      }
      coef[t] = s::make(re, im);
    }
    __syncthreads();
    for (int64_t i = i0 + tid; i < i1; i += STEP_THREADS) {
      T v = w[i];
#pragma unroll 4
      for (int col = 0; col <= j; ++col) v = s::sub(v, s::mul(V[i + (int64_t)col * n], coef[col]));
      w[i] = v;
      nrm += s::abs2(v);
      const unsigned long long b = magnitude_bits<T>(v);
      mx = mx > b ? mx : b;
    }
  }
  nrm = warp_sum(nrm);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = mx > b ? mx : b;
  }
  __syncthreads();
  if (lane == 0) {
    red[warp] = nrm;
    redm[warp] = mx;
  }
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    unsigned long long m = 0ull;
    for (int k = 0; k < NW; ++k) {
      t += red[k];
      m = m > redm[k] ? m : redm[k];
    }
    sh_norm = t;
    sh_max = m;
  }
  __syncthreads();
  cluster_barrier();
  double ss = 0.0;
  mx = 0ull;
  for (unsigned c = 0; c < nct; ++c) {
    ss += peer_double(&sh_norm, c);
    const unsigned long long b = peer_bits(&sh_max, c);
    mx = mx > b ? mx : b;
  }
  cluster_barrier();  // no CTA exits before its peers have read its sums
  const double bt = sqrt(ss);
  if (j >= 0 && tid == 0 && rank == 0) beta[run * LZ_MAXS + j] = bt;
  if (j + 1 >= steps) return;
  const double inv = j < 0 ? 1.0 / bt : (bt > 0.0 ? 1.0 / bt : 0.0);
  // largest magnitude of the new vector: rounding is monotone, so the scaled maximum bounds every entry
  const int e = exponent_of_bits((unsigned long long)__double_as_longlong(fabs(__longlong_as_double((long long)mx) * inv)));
  if (tid == 0 && rank == 0) xe[run] = e;
  const int es = e == LZ_NONFINITE ? 0 : e;
  T* vn = V + (int64_t)(j + 1) * n;
  for (int64_t i = i0 + tid; i < i1; i += STEP_THREADS) {
    const T v = s::scale(w[i], inv);
    vn[i] = v;
    write_frag<T>(X, (n + HK - 1) / HK, i, run, to_fixed(s::re(v), es), NC == 2 ? to_fixed(s::im(v), es) : 0ll);
  }
}

// ---------------------------------------------------------------- Ritz values
// Implicit QL with Wilkinson shifts on a tridiagonal T (diagonal d, off-diagonal e, k <= 64) by one warp: eigenvalues, and
// z, the first row of the eigenvectors' matrix (Golub and Welsch 1969).  About 1.7 sweeps per eigenvalue of at most k
// rotations, a serial chain of FP64 operations in lane 0 (0.9 ms for k = 25).
__device__ __noinline__ void ql_first_row(int k, double* d, double* e, double* z, int* status) {
  const int lane = threadIdx.x & 31;
  const double eps = 1.1102230246251565e-16;
  for (int l = 0; l < k; ++l) {
    for (int iter = 0;; ++iter) {
      // first mm >= l whose off-diagonal entry is negligible (k - 1 at the latest)
      auto small = [&](int i) {
        return i >= k - 1 || (i >= l && (fabs(e[i]) <= eps * (fabs(d[i]) + fabs(d[i + 1])) || fabs(e[i]) < 1e-150));
      };
      const unsigned lo = __ballot_sync(0xffffffffu, small(lane));
      const unsigned hi = __ballot_sync(0xffffffffu, small(lane + 32));
      const int mm = min(k - 1, lo ? __ffs((int)lo) - 1 : 31 + __ffs((int)hi));
      if (mm == l) break;
      if (iter == 60) {
        if (lane == 0) atomicOr(status, LZ_STATUS_QL);
        break;
      }
      if (lane == 0) {
        double g = (d[l + 1] - d[l]) / (2.0 * e[l]);
        const double h = sqrt(g * g + 1.0);
        g = d[mm] - d[l] + e[l] / (g + (g >= 0.0 ? h : -h));
        double sn = 1.0, cs = 1.0, p = 0.0;
        double di1 = d[mm];
        int i = mm - 1;
        for (; i >= l; --i) {
          const double ei = e[i], di = d[i], zi = z[i], zi1 = z[i + 1];
          const double f = sn * ei, b = cs * ei;
          const double q = fma(f, f, g * g);
          if (!(q > 1e-300)) {  // the rotation is undefined: the matrix splits here
            e[i + 1] = 0.0;
            d[i + 1] = di1 - p;
            e[mm] = 0.0;
            break;
          }
          const double ri = fast_rsqrt(q);
          e[i + 1] = q * ri;
          sn = f * ri;
          cs = g * ri;
          g = di1 - p;
          const double t = fma(di - g, sn, 2.0 * cs * b);
          p = sn * t;
          d[i + 1] = g + p;
          g = fma(cs, t, -b);
          z[i + 1] = fma(sn, zi, cs * zi1);
          z[i] = fma(cs, zi, -sn * zi1);
          di1 = di;
        }
        if (i < l) {
          d[l] -= p;
          e[l] = g;
          e[mm] = 0.0;
        }
      }
      __syncwarp();
    }
    __syncwarp();
  }
}

// The same in FP32 with all eigenvectors (columns of Z, ld ldz), the lanes sharing Z's rows.  False: no convergence.
__device__ __forceinline__ bool ql_fp32(int k, float* d, float* e, float* Z, int ldz) {
  const int lane = threadIdx.x & 31;
  const float eps = 5.9604645e-8f;
  for (int l = 0; l < k; ++l) {
    for (int iter = 0;; ++iter) {
      auto small = [&](int i) {
        return i >= k - 1 || (i >= l && fabsf(e[i]) <= eps * (fabsf(d[i]) + fabsf(d[i + 1]) + 1e-3f));
      };
      const unsigned lo = __ballot_sync(0xffffffffu, small(lane));
      const unsigned hi = __ballot_sync(0xffffffffu, small(lane + 32));
      const int mm = min(k - 1, lo ? __ffs((int)lo) - 1 : 31 + __ffs((int)hi));
      if (mm == l) break;
      if (iter == 60) return false;
      // every lane makes the same scalars
      float g = (d[l + 1] - d[l]) / (2.0f * e[l]);
      const float h = sqrtf(g * g + 1.0f);
      g = d[mm] - d[l] + e[l] / (g + (g >= 0.0f ? h : -h));
      float sn = 1.0f, cs = 1.0f, p = 0.0f, di1 = d[mm];
      float z0 = lane < k ? Z[lane + mm * ldz] : 0.0f, z1 = lane + 32 < k ? Z[lane + 32 + mm * ldz] : 0.0f;
      int i = mm - 1;
      for (; i >= l; --i) {
        const float f = sn * e[i], b = cs * e[i], di = d[i];
        const float q = fmaf(f, f, g * g);
        if (!(q > 1e-36f)) return false;  // the rotation is undefined: left to the FP64 version
        // every lane has made its reads of the rotation before (and of d[mm], d[l + 1], e[l]) when lane 0 stores over them
        __syncwarp();
        const float ri = rsqrtf(q);
        const float c0 = lane < k ? Z[lane + i * ldz] : 0.0f, c1 = lane + 32 < k ? Z[lane + 32 + i * ldz] : 0.0f;
        sn = f * ri;
        cs = g * ri;
        g = di1 - p;
        const float t = fmaf(di - g, sn, 2.0f * cs * b);
        p = sn * t;
        if (lane == 0) {
          e[i + 1] = q * ri;
          d[i + 1] = g + p;
        }
        g = fmaf(cs, t, -b);
        if (lane < k) Z[lane + (i + 1) * ldz] = fmaf(sn, c0, cs * z0);
        if (lane + 32 < k) Z[lane + 32 + (i + 1) * ldz] = fmaf(sn, c1, cs * z1);
        z0 = fmaf(cs, c0, -sn * z0);
        z1 = fmaf(cs, c1, -sn * z1);
        di1 = di;
      }
      if (lane < k) Z[lane + l * ldz] = z0;
      if (lane + 32 < k) Z[lane + 32 + l * ldz] = z1;
      __syncwarp();
      if (lane == 0) {
        d[l] -= p;
        e[l] = g;
        e[mm] = 0.0f;
      }
      __syncwarp();
    }
  }
  return true;
}

// Eigenvalues theta (ascending) and squared first eigenvector components tau2 of every run's tridiagonal T, one block
// per run.  An FP64 rotation chain is bound by the latency of its operations (over 100 cycles each), so QL runs in
// FP32 and its eigenvectors X are corrected in FP64 by products that all threads share (Ogita and Aishima 2018):
// R = I - X^T X, S = X^T T X, E_ij = (S_ij + l_j R_ij) / (l_j - l_i), X <- X + X E, quadratically convergent.  The step
// after max |E| <= 1e-8 ends it; a pair of eigenvalues too close for E, or no convergence, leaves T to QL in FP64.
// k = 25: 125 us, 890 by QL in FP64.  (A two-sided Jacobi over the block took 5.6 ms.)
constexpr int TRI_THREADS = 256;
__global__ void __launch_bounds__(TRI_THREADS) tridiag_kernel(int steps, const double* alpha, const double* beta, double* theta,
                                                              double* tau2, int* status) {
  const int r = blockIdx.x, k = steps, tid = threadIdx.x, ld = k + 1;
  extern __shared__ double tri_smem[];
  double *X = tri_smem, *Y = X + k * ld, *Sm = Y + k * ld, *Rm = Sm + k * ld;  // column-major, ld k + 1
  __shared__ double d[LZ_MAXS], e[LZ_MAXS], z[LZ_MAXS], lam[LZ_MAXS], red[3][TRI_THREADS / 32];
  __shared__ float df[LZ_MAXS], ef[LZ_MAXS];
  __shared__ int sc_sh, ok_sh;
  // scaled by a power of two to norm about 1, so that squares neither overflow nor vanish
  if (tid < 32) {
    double m = 0.0;
    for (int i = tid; i < k; i += 32) {
      d[i] = alpha[r * LZ_MAXS + i];
      e[i] = i + 1 < k ? beta[r * LZ_MAXS + i] : 0.0;
      z[i] = i == 0 ? 1.0 : 0.0;
      m = fmax(m, fmax(fabs(d[i]), fabs(e[i])));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    int sc = 0;
    if (m > 0.0 && isfinite(m)) frexp(m, &sc);
    for (int i = tid; i < k; i += 32) {
      d[i] = ldexp(d[i], -sc);
      e[i] = ldexp(e[i], -sc);
      df[i] = (float)d[i];
      ef[i] = (float)e[i];
    }
    if (tid == 0) sc_sh = sc;
  }
  float* Z = reinterpret_cast<float*>(Y);
  for (int q = tid; q < k * ld; q += TRI_THREADS) Z[q] = q % ld == q / ld ? 1.0f : 0.0f;
  __syncthreads();
  if (tid < 32) {
    const bool ok = ql_fp32(k, df, ef, Z, ld);
    if (tid == 0) ok_sh = ok;
  }
  __syncthreads();
  for (int q = tid; q < k * ld; q += TRI_THREADS) X[q] = Z[q];
  __syncthreads();
  bool ok = ok_sh != 0, last = false;
  auto block_max = [&](double v, int set) {  // NaN counts as infinity
    v = v == v ? v : INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((tid & 31) == 0) red[set][tid >> 5] = v;
    __syncthreads();
    v = red[set][0];
    for (int w = 1; w < TRI_THREADS / 32; ++w) v = fmax(v, red[set][w]);
    return v;
  };
  for (int it = 0; ok && !last; ++it) {
    for (int q = tid; q < k * k; q += TRI_THREADS) {
      const int j = q / k, i = q - j * k;
      const double* x = X + j * ld;
      double v = d[i] * x[i];
      if (i > 0) v += e[i - 1] * x[i - 1];
      if (i + 1 < k) v += e[i] * x[i + 1];
      Y[j * ld + i] = v;
    }
    __syncthreads();
    double off = 0.0, orth = 0.0;
    for (int q = tid; q < k * k; q += TRI_THREADS) {
      const int j = q / k, i = q - j * k;
      if (i > j) continue;  // both are symmetric
      double sa = 0.0, ra = i == j ? 1.0 : 0.0;
      for (int p = 0; p < k; ++p) {
        sa += X[i * ld + p] * Y[j * ld + p];
        ra -= X[i * ld + p] * X[j * ld + p];
      }
      Sm[j * ld + i] = Sm[i * ld + j] = sa;
      Rm[j * ld + i] = Rm[i * ld + j] = ra;
      if (i == j) lam[i] = sa / (1.0 - ra);
      else off = fmax(off, fabs(sa));
      orth = fmax(orth, fabs(ra));
    }
    off = block_max(off, 0);
    orth = block_max(orth, 1);
    // eigenvalues closer than this cannot be told apart yet
    const double close = 8.0 * (off + orth);
    double big = 0.0, open = 0.0;
    for (int q = tid; q < k * k; q += TRI_THREADS) {
      const int j = q / k, i = q - j * k;
      const double gap = lam[j] - lam[i], rij = Rm[j * ld + i];
      double ev = 0.5 * rij;
      if (i != j) {
        const double c = Sm[j * ld + i] + lam[j] * rij;
        if (fabs(gap) > close) ev = c / gap;
        else if (fabs(c) > 1e-17) open = 1.0;  // not an exactly decoupled pair
      }
      big = fmax(big, fabs(ev));
      Y[j * ld + i] = ev;
    }
    big = block_max(big, 2);
    last = __syncthreads_or(open != 0.0) == 0 && big <= 1e-8;
    ok = big < 0.1 && (last || it < 5);
    if (!ok) break;
    for (int q = tid; q < k * k; q += TRI_THREADS) {
      const int j = q / k, i = q - j * k;
      double v = X[j * ld + i];
      for (int p = 0; p < k; ++p) v += X[p * ld + i] * Y[j * ld + p];
      Sm[j * ld + i] = v;
    }
    __syncthreads();
    double* t = X;
    X = Sm;
    Sm = t;
  }
  if (ok) {
    for (int i = tid; i < k; i += TRI_THREADS) {
      d[i] = lam[i];
      z[i] = X[i * ld];
    }
  } else if (tid < 32) {
    ql_first_row(k, d, e, z, status);
  }
  __syncthreads();
  const int sc = sc_sh;
  // ascending (stable) order; a T that is not finite has no order and gives NaN throughout
  for (int i = tid; i < k; i += TRI_THREADS) {
    const double wi = d[i];
    int rank = 0;
    bool bad = false;
    for (int q = 0; q < k; ++q) {
      rank += (d[q] < wi) || (d[q] == wi && q < i);
      bad |= !isfinite(d[q]) || !isfinite(z[q]);
    }
    theta[r * LZ_MAXS + (bad ? i : rank)] = bad ? NAN : ldexp(wi, sc);
    tau2[r * LZ_MAXS + (bad ? i : rank)] = bad ? NAN : z[i] * z[i];
  }
}

// b_sup, mu_1, mu_ne (DoS quantile), theta_max: the pooled Ritz values ranked in parallel, their weights added in
// ascending order by one thread.  All four are NaN when any of the values is not finite (fmax and fmin would drop it); the
// status word follows them.
__global__ void lanczos_bounds_kernel(int runs, int steps, int64_t n, int ne, const double* theta, const double* tau2,
                                      const double* beta, const int* status, double* out5) {
  __shared__ double th[LZ_MAXR * LZ_MAXS], so[LZ_MAXR * LZ_MAXS], wt[LZ_MAXR * LZ_MAXS];
  const int total = runs * steps;
  bool bad = false;
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    const int at = (i / steps) * LZ_MAXS + i % steps;
    th[i] = theta[at];
    so[i] = wt[i] = 0.0;
    bad |= !isfinite(th[i]) || !isfinite(tau2[at]) || !isfinite(beta[at]);
  }
  bad = __syncthreads_or(bad);
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    const double t = th[i];
    int rank = 0;
    for (int q = 0; q < total; ++q) rank += (th[q] < t) || (th[q] == t && q < i);
    so[rank] = t;
    wt[rank] = tau2[(i / steps) * LZ_MAXS + i % steps] / runs;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  double b_sup = -1e308, mu1 = 1e308, tmax = -1e308;
  for (int r = 0; r < runs; ++r) {
    b_sup = fmax(b_sup, th[r * steps + steps - 1] + fabs(beta[r * LZ_MAXS + steps - 1]));
    mu1 = fmin(mu1, th[r * steps]);
    tmax = fmax(tmax, th[r * steps + steps - 1]);
  }
  const double target = (double)ne / (double)n;
  double acc = 0.0, mu_ne = -1e308;
  for (int q = 0; q < total; ++q) {
    acc += wt[q];
    mu_ne = so[q];
    if (acc >= target) break;
  }
  double span = b_sup - mu1;
  double lo = mu1 + 1e-3 * span, hi = b_sup - 1e-3 * span;
  mu_ne = fmin(fmax(mu_ne, lo), hi);
  out5[0] = bad ? NAN : b_sup;
  out5[1] = bad ? NAN : mu1;
  out5[2] = bad ? NAN : mu_ne;
  out5[3] = bad ? NAN : tmax;
  out5[4] = *status;
}

// CTAs per run: 16 where the device schedules such clusters and the vectors are long, else 8
template <typename T> static int step_ctas(int64_t n) {
  static std::once_flag once;
  static bool big = false;
  std::call_once(once, []() {
    if (cudaFuncSetAttribute(lanczos_step_kernel<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = STEP_MAXC;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(STEP_MAXC, 1, 1);
    cfg.blockDim = dim3(STEP_THREADS, 1, 1);
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, lanczos_step_kernel<T>, &cfg) == cudaSuccess && nc > 0) big = true;
    else cudaGetLastError();
  });
  return n >= 2048 && big ? STEP_MAXC : 8;
}

template <typename T> static void lanczos_attributes() {
  static std::once_flag once;
  static cudaError_t err = cudaSuccess;
  std::call_once(once, []() {
    err = cudaFuncSetAttribute(hemv_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, Hemv<T>::SMEM);
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(tridiag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 4 * LZ_MAXS * (LZ_MAXS + 1) * (int)sizeof(double));
  });
  CHASE_CUDA(err);
}

template <typename T>
void lanczos(cudaStream_t st, const T* A, int64_t n, int64_t lda, int ne, const T* L0, int runs, int steps,
             double* out5, T* work, int64_t work_elems, double* dwork, bool native) {
  CHASE_REQUIRE(runs >= 1 && runs <= LZ_MAXR, 1, "lanczos: 1 <= runs <= 8");
  CHASE_REQUIRE(steps >= 1 && steps <= LZ_MAXS && steps <= n, 1, "lanczos: 1 <= steps <= min(64, n)");
  const int cols = hemv_cols(n);
  const int nchunk = (int)ceil_div(n, cols);
  CHASE_REQUIRE(work_elems >= lanczos_work_elems(n, runs, steps, S<T>::cplx), 2, "lanczos: workspace too small");
  T* Vb = work;
  T* W = Vb + (int64_t)runs * steps * n;
  T* part = W + (int64_t)runs * n;
  // fragments are read 16 bytes at a time
  __half* X = reinterpret_cast<__half*>((reinterpret_cast<uintptr_t>(part + (int64_t)nchunk * runs * n) + 15) & ~(uintptr_t)15);
  const int64_t xhalves = frag_halves(n, S<T>::cplx, runs);
  unsigned* rmax = reinterpret_cast<unsigned*>(X + xhalves);
  int* xe = reinterpret_cast<int*>(rmax + n);
  // dwork: alpha, beta, theta, tau2 (runs*LZ_MAXS each) + status
  double* alpha = dwork;
  double* beta = alpha + LZ_MAXR * LZ_MAXS;
  double* theta = beta + LZ_MAXR * LZ_MAXS;
  double* tau2 = theta + LZ_MAXR * LZ_MAXS;
  int* status = reinterpret_cast<int*>(tau2 + LZ_MAXR * LZ_MAXS);
  CHASE_CUDA(cudaMemsetAsync(status, 0, sizeof(int), st));
  // unused vector columns and rows past n are zero digits
  CHASE_CUDA(cudaMemsetAsync(X, 0, xhalves * sizeof(__half), st));
  CHASE_CUDA(cudaMemsetAsync(rmax, 0, n * sizeof(unsigned), st));
  if (!native) {
    row_max_kernel<T><<<dim3(ceil_div(n, 128), ceil_div(n, ROWMAX_COLS)), 128, 0, st>>>(n, A, lda, rmax);
    CHASE_CHECK_LAUNCH();
  }

  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[2] = {{}, pdl_attribute()};
  const int ctas = step_ctas<T>(n);
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ctas;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(ctas, runs, 1);
  cfg.blockDim = dim3(STEP_THREADS, 1, 1);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  auto step = [&](int j) {
    CHASE_CUDA(cudaLaunchKernelEx(&cfg, lanczos_step_kernel<T>, n, runs, steps, j, nchunk, (const T*)part, L0, Vb, W,
                                  alpha, beta, X, xe));
    CHASE_CHECK_LAUNCH();
  };
  lanczos_attributes<T>();
  step(-1);
  const dim3 g1(ceil_div(n, HEMV_ROWS), nchunk, ceil_div(runs, Frag<T>::RUNS));
  for (int j = 0; j < steps; ++j) {
    if (native) {
      hemv_dfma<T>(st, n, A, lda, Vb + (int64_t)j * n, n * steps, cols, runs, part);
    } else {
      launch_pdl(hemv_kernel<T>, g1, HEMV_THREADS, Hemv<T>::SMEM, st, n, A, lda, rmax, X, xe, cols, runs, part,
                 grid_wait_limit_ns(), status);
      CHASE_CHECK_LAUNCH();
    }
    step(j);
  }
  tridiag_kernel<<<runs, TRI_THREADS, 4 * steps * (steps + 1) * (int)sizeof(double), st>>>(steps, alpha, beta, theta, tau2, status);
  CHASE_CHECK_LAUNCH();
  lanczos_bounds_kernel<<<1, 256, 0, st>>>(runs, steps, n, ne, theta, tau2, beta, status, out5);
  CHASE_CHECK_LAUNCH();
}

void check_lanczos(const double (&out5)[5]) {
  CHASE_REQUIRE(((int)out5[4] & LZ_STATUS_WAIT) == 0, 8, "a Lanczos product hit its wait limit");
  for (int i = 0; i < 4; ++i) CHASE_REQUIRE(std::isfinite(out5[i]), 5, "non-finite Lanczos bounds");
}

template void lanczos<double>(cudaStream_t, const double*, int64_t, int64_t, int, const double*, int, int, double*,
                              double*, int64_t, double*, bool);
template void lanczos<double2>(cudaStream_t, const double2*, int64_t, int64_t, int, const double2*, int, int, double*,
                               double2*, int64_t, double*, bool);

}  // namespace chase
