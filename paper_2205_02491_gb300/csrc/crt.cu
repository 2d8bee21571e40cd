// FP64-class products C = L R on the bf16 tensor cores (tcgen05, TMEM, TMA, CTA pairs) through residues: the modular form of
// Ozaki's scheme (Ozaki, Uchino and Imamura 2025).
//
// Every left row / right column x is scaled by a power of two so that its 2-norm is below 2^62 and rounded to
// integers X (at most half a unit each).  The integer product then satisfies |C_ij| <= ||X_i|| ||Y_j|| < 2^124
// (Cauchy-Schwarz), and it is determined by its residues modulo NMOD = 16 pairwise coprime moduli m_i <= 256 whose
// product is M = 2^125.6 (Chinese remainder theorem): 2^124 = 0.33 M < M / 2.  Each residue of X lies in
// [-128, 128] and is exact in bf16, a product of two residues is at most 2^14, and 1024 of them sum to at most 2^24,
// so FP32 accumulators are exact over chunks of 1024 along K.  Complex operands take three real products per modulus
// instead of four, P1 = Xr Yr, P2 = Xi Yi, P3 = (Xr + Xi)(Yr + Yi): modulo m_i nothing is lost to the sums or to
// Re = P1 - P2, Im = P3 - P1 - P2.
//
// Why residues and not digits: splitting FP64 operands into seven 8-bit digits takes 28 digit-pair products (112 for
// complex operands) and one accumulator per digit level, which caps the MMA width at 80 columns (44 cycles per MMA,
// the instruction's floor, for 40 cycles of math).  Residues take 16 (48 complex) products, each a plain bf16 GEMM
// with the widest MMA (256 x 256 x 16 on a CTA pair), and round the operands no more coarsely: an entry keeps
// 62 - log2(norm / |entry|) bits.
// Why moduli up to 256 and not 512 (residues up to 256 are exact in bf16 too, and 14 moduli suffice): chunks would
// hold 256 along K, and reading TMEM four times as often stalls the MMAs (n = 8192, 512 columns, 14 real planes:
// 863 us, against 588 us with a read per 1024), which outweighs the two planes saved.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "crt.h"
#include "tcgen05.cuh"
#include "tmap.h"

namespace chase {
namespace crt {

using oz::fence_after;
using oz::fence_before;
using oz::globaltimer;
using oz::mbar_expect_tx;
using oz::mbar_init;
using oz::mbar_try;
using oz::smem_u32;
using oz::sw128_desc;

// ---------------------------------------------------------------- moduli and reconstruction constants
typedef unsigned __int128 u128;

// The 16 pairwise coprime integers <= 256 with the largest product (exhaustive search from the top).
#define CRT_MODULI {256, 253, 251, 249, 247, 241, 239, 235, 233, 229, 227, 223, 217, 211, 199, 197}

struct Tables {
  int m[NMOD];           // moduli
  int inv[NMOD];         // round(2^38 / m): nearest-integer quotients of |t| < 2^30 by a multiply and a shift
  int c1[NMOD], c2[NMOD];  // 2^21 and 2^42 modulo m, in [-128, 128]
  uint32_t w[NMOD][4];   // (M / m_i) ((M / m_i)^-1 mod m_i): the CRT weights, 32-bit limbs
  uint32_t off[4];       // -BIAS sum_i w_i mod M
  uint64_t Mlo, Mhi;
  float q;               // 2^112 / M
};
constexpr int BIAS = 512;  // added to every residue (at most 3 * 128 in size) so that the limb products are unsigned

constexpr int sym_mod(u128 x, int m) {
  int r = (int)(x % (u128)m);
  return r > m / 2 ? r - m : r;
}

constexpr Tables make_tables() {
  Tables t{};
  const int ms[NMOD] = CRT_MODULI;
  u128 M = 1;
  for (int i = 0; i < NMOD; ++i) M *= (u128)ms[i];
  u128 wsum = 0;
  for (int i = 0; i < NMOD; ++i) {
    const int m = ms[i];
    t.m[i] = m;
    t.inv[i] = (int)((((uint64_t)1 << 38) + (uint64_t)m / 2) / (uint64_t)m);
    t.c1[i] = sym_mod((u128)1 << 21, m);
    t.c2[i] = sym_mod((u128)1 << 42, m);
    const u128 Mi = M / (u128)m;
    const int a = (int)(Mi % (u128)m);
    int iv = 1;
    while (a * iv % m != 1) ++iv;
    const u128 w = Mi * (u128)iv;  // < M: iv < m
    for (int l = 0; l < 4; ++l) t.w[i][l] = (uint32_t)(w >> (32 * l));
    wsum = (wsum + w) % M;
  }
  u128 off = 0;
  for (int i = 0; i < BIAS; ++i) off = (off + wsum) % M;
  off = M - off;
  for (int l = 0; l < 4; ++l) t.off[l] = (uint32_t)(off >> (32 * l));
  t.Mlo = (uint64_t)M;
  t.Mhi = (uint64_t)(M >> 64);
  t.q = (float)(281474976710656.0 / (double)t.Mhi);  // 2^112 / M = 2^48 / (M / 2^64)
  return t;
}

constexpr Tables kTables = make_tables();
static_assert(kTables.Mhi >> 61 == 1, "M lies in [2^125, 2^126)");
__constant__ const Tables cT = make_tables();

// ---------------------------------------------------------------- scales
// Exponent e with norm < 2^e from the sum of squares.
__device__ __forceinline__ int norm_exponent(double ss) {
  int e;
  frexp(sqrt(ss) * (1.0 + 1e-9), &e);
  return e;
}

// Column norms: one pass of plain squares; a sum outside the range where squares neither overflow nor lose
// bits to underflow (or a non-finite one) takes a second, scaled pass.  HBM/L2-bound, one block per column.
template <typename T>
__global__ void __launch_bounds__(256) col_exponent_kernel(int64_t K, const T* __restrict__ X, int64_t ldx, int* ex) {
  grid_dependency_wait();
  using s = S<T>;
  const T* x = X + (int64_t)blockIdx.x * ldx;
  __shared__ double red[8];
  __shared__ double sum_sh;
  auto block_sum = [&](double v) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < 8; ++w) t += red[w];
      sum_sh = t;
    }
    __syncthreads();
    return sum_sh;
  };
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int64_t i = threadIdx.x;
  for (; i + 768 < K; i += 1024) {
    const T v0 = x[i], v1 = x[i + 256], v2 = x[i + 512], v3 = x[i + 768];
    a0 += s::abs2(v0);
    a1 += s::abs2(v1);
    a2 += s::abs2(v2);
    a3 += s::abs2(v3);
  }
  for (; i < K; i += 256) a0 += s::abs2(x[i]);
  double ss = block_sum((a0 + a1) + (a2 + a3));
  if (ss > 1e-250 && ss < 1e250) {
    if (threadIdx.x == 0) ex[blockIdx.x] = norm_exponent(ss);
    return;
  }
  // largest magnitude (through the bit pattern, so that NaN and infinity compare largest), then scaled squares
  __shared__ unsigned long long mx;
  if (threadIdx.x == 0) mx = 0ull;
  __syncthreads();
  unsigned long long m = 0ull;
  for (int64_t j = threadIdx.x; j < K; j += 256) {
    const T v = x[j];
    const unsigned long long br = (unsigned long long)__double_as_longlong(fabs(s::re(v)));
    const unsigned long long bi = (unsigned long long)__double_as_longlong(fabs(s::im(v)));
    m = m > br ? m : br;
    m = m > bi ? m : bi;
  }
  atomicMax(&mx, m);
  __syncthreads();
  if (mx >= 0x7ff0000000000000ull) {
    if (threadIdx.x == 0) ex[blockIdx.x] = NONFINITE;
    return;
  }
  if (mx == 0ull) {
    if (threadIdx.x == 0) ex[blockIdx.x] = 0;
    return;
  }
  int em;
  frexp(__longlong_as_double((long long)mx), &em);
  double b = 0.0;
  for (int64_t j = threadIdx.x; j < K; j += 256) {
    const T v = x[j];
    const double r = ldexp(s::re(v), -em), q = ldexp(s::im(v), -em);
    b += r * r + q * q;
  }
  ss = block_sum(b);
  if (threadIdx.x == 0) ex[blockIdx.x] = em + norm_exponent(ss);
}

// Row norms of a column-major X (vector = row): 32 rows x 8 threads along K per block, so that a short and a long
// K both fill the SMs; same two-pass rule as the columns.
template <typename T>
__global__ void __launch_bounds__(256) row_exponent_kernel(int64_t nvec, int64_t K, const T* __restrict__ X, int64_t ldx,
                                                            int* ex) {
  grid_dependency_wait();
  using s = S<T>;
  const int r = threadIdx.x & 31, c = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * 32 + r;
  __shared__ double red[8][33];
  __shared__ unsigned long long redm[8][33];
  double a = 0.0;
  unsigned long long m = 0ull;
  if (i < nvec) {
#pragma unroll 4
    for (int64_t k = c; k < K; k += 8) {
      const T v = X[i + k * ldx];
      a += s::abs2(v);
      const unsigned long long br = (unsigned long long)__double_as_longlong(fabs(s::re(v)));
      const unsigned long long bi = (unsigned long long)__double_as_longlong(fabs(s::im(v)));
      m = m > br ? m : br;
      m = m > bi ? m : bi;
    }
  }
  red[c][r] = a;
  redm[c][r] = m;
  __syncthreads();
  if (c != 0 || i >= nvec) return;
  for (int w = 1; w < 8; ++w) {
    a += red[w][r];
    m = m > redm[w][r] ? m : redm[w][r];
  }
  int e;
  if (m >= 0x7ff0000000000000ull) {
    e = NONFINITE;
  } else if (m == 0ull) {
    e = 0;
  } else if (a > 1e-250 && a < 1e250) {
    e = norm_exponent(a);
  } else {
    int em;
    frexp(__longlong_as_double((long long)m), &em);
    double b = 0.0;
    for (int64_t k = 0; k < K; ++k) {
      const T v = X[i + k * ldx];
      const double p = ldexp(s::re(v), -em), q = ldexp(s::im(v), -em);
      b += p * p + q * q;
    }
    e = em + norm_exponent(b);
  }
  ex[i] = e;
}

// ---------------------------------------------------------------- residue planes
// round(x 2^(62 - e)) by integer shifts of the mantissa (GB300's FP64 conversions run at 1/64 of the integer
// rate); |result| <= 2^62 because |x| < 2^e, which also keeps any left shift of a finite vector's entries within 64 bits
// (9 for normal numbers, up to 61 where a whole vector is subnormal).  Non-finite vectors give arbitrary integers.
__device__ __forceinline__ long long scaled_int(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int be = (int)((b >> 52) & 0x7ff);
  long long m = b & 0xfffffffffffffll;
  if (be != 0) m |= 0x10000000000000ll;
  const int sh = (be != 0 ? be : 1) - 1075 + 62 - e;  // x = m 2^(exponent - 1075)
  long long r;
  if (sh >= 0) {
    r = (long long)((unsigned long long)m << (sh < 62 ? sh : 62));
  } else {
    const int rs = sh > -62 ? -sh : 62;
    r = ((m >> (rs - 1)) + 1) >> 1;
  }
  return b < 0 ? -r : r;
}

struct Limbs {
  int x0, x1, x2;
};
__device__ __forceinline__ Limbs limbs(long long x) {
  return Limbs{(int)(x & 0x1fffff), (int)((x >> 21) & 0x1fffff), (int)(x >> 42)};
}

// x mod m_i in [-128, 128]: the limbs' residue sum t (|t| < 2^30), then t - m round(t / m).  The quotient's error is
// below 2^-9 / 2, so |r| < m / 2 + 1 / 2: at most (m - 1) / 2 for odd m, at most 128 for m = 256.
__device__ __forceinline__ int residue(const Limbs& x, int i) {
  const int t = x.x0 + x.x1 * cT.c1[i] + x.x2 * cT.c2[i];
  const int q = (int)(((long long)t * cT.inv[i] + (1ll << 37)) >> 38);
  return t - q * cT.m[i];
}
// sum of two residues brought back to [-128, 128]
__device__ __forceinline__ int residue_sum(int a, int b, int i) {
  int r = a + b;
  if (r > 128) r -= cT.m[i];
  if (r < -128) r += cT.m[i];
  return r;
}
// two integers |r| <= 128 as packed bf16 (exact: the upper halves of their FP32 images)
__device__ __forceinline__ uint32_t pack_bf16(int a, int b) {
  const float fa = __int_as_float(0x4b400000 + a) - 12582912.0f;
  const float fb = __int_as_float(0x4b400000 + b) - 12582912.0f;
  return __byte_perm(__float_as_uint(fa), __float_as_uint(fb), 0x7632);
}

// Four consecutive K elements of one vector: every modulus' planes, one 8-byte store per plane.
template <typename T>
__device__ __forceinline__ void write_residues(const T (&v)[4], int e, bool conj, int mod0, int nmod, int64_t plane,
                                               __nv_bfloat16* out) {
  using s = S<T>;
  Limbs re[4], im[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    re[j] = limbs(scaled_int(s::re(v[j]), e));
    if (s::cplx) {
      const long long q = scaled_int(s::im(v[j]), e);
      im[j] = limbs(conj ? -q : q);
    }
  }
  for (int i = 0; i < nmod; ++i) {
    int rr[4], ri[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) rr[j] = residue(re[j], mod0 + i);
    *reinterpret_cast<uint2*>(out) = make_uint2(pack_bf16(rr[0], rr[1]), pack_bf16(rr[2], rr[3]));
    out += plane;
    if (s::cplx) {
#pragma unroll
      for (int j = 0; j < 4; ++j) ri[j] = residue(im[j], mod0 + i);
      *reinterpret_cast<uint2*>(out) = make_uint2(pack_bf16(ri[0], ri[1]), pack_bf16(ri[2], ri[3]));
      out += plane;
#pragma unroll
      for (int j = 0; j < 4; ++j) rr[j] = residue_sum(rr[j], ri[j], mod0 + i);
      *reinterpret_cast<uint2*>(out) = make_uint2(pack_bf16(rr[0], rr[1]), pack_bf16(rr[2], rr[3]));
      out += plane;
    }
  }
}

// vector = column of X
template <typename T>
__global__ void __launch_bounds__(128) residues_cols_kernel(int64_t K, int64_t Kp, int64_t nvec, const T* __restrict__ X,
                                                             int64_t ldx, const int* __restrict__ ex, int conj, int mod0,
                                                             int nmod, __nv_bfloat16* planes) {
  grid_dependency_wait();
  const int64_t col = blockIdx.y;
  const T* x = X + col * ldx;
  int e = ex[col];
  if (e == NONFINITE) e = 0;
  for (int64_t i = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x); i < K; i += 4 * (int64_t)gridDim.x * blockDim.x) {
    T v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = i + j < K ? x[i + j] : S<T>::zero();
    write_residues<T>(v, e, conj != 0, mod0, nmod, nvec * Kp, planes + col * Kp + i);
  }
}

// vector = row of X: 32 x 32 tiles transposed through shared memory
template <typename T>
__global__ void __launch_bounds__(256) residues_rows_kernel(int64_t nvec, int64_t K, int64_t Kp, const T* __restrict__ X,
                                                             int64_t ldx, const int* __restrict__ ex, int conj, int mod0,
                                                             int nmod, __nv_bfloat16* planes) {
  grid_dependency_wait();
  __shared__ T tile[32][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32, k0 = (int64_t)blockIdx.y * 32;
  for (int r = threadIdx.x >> 5; r < 32; r += 8) {
    const int64_t kk = k0 + r, i = i0 + (threadIdx.x & 31);
    tile[r][threadIdx.x & 31] = (kk < K && i < nvec) ? X[i + kk * ldx] : S<T>::zero();
  }
  __syncthreads();
  const int r = threadIdx.x >> 3, g = (threadIdx.x & 7) * 4;
  const int64_t i = i0 + r;
  if (i >= nvec || k0 + g >= K) return;
  T v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = tile[g + j][r];
  int e = ex[i];
  if (e == NONFINITE) e = 0;
  write_residues<T>(v, e, conj != 0, mod0, nmod, nvec * Kp, planes + i * Kp + k0 + g);
}

// ---------------------------------------------------------------- right operands: norms and planes in one launch
constexpr int MAXG = 64;  // products per launch
// shared::cluster address of this CTA-local address in the given CTA of the cluster
__device__ __forceinline__ uint32_t cluster_addr(uint32_t a, uint32_t cta) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(cta));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int G> struct RightParams {
  const void* X[G];
  int64_t ldx[G];
  int* ex[G];
  void* planes[G];
  int nvec[G], K[G];
};

// A right operand's columns, exponents and all residue planes; blockIdx.y runs over the products' columns.  A cluster
// (1 to 8 CTAs, 512 elements each while K <= 4096) takes one column: the CTAs' partial sums of squares meet in
// every CTA's shared memory, so that a short K needs one launch of a few microseconds and a few columns still spread
// over the SMs.  What bounds it: latency and launch overhead at small sizes, instruction issue at large ones.
// Complex, n = 512: 6.1 us where separate norm and plane launches took 8.0 and the gap between them; n = 8192 and 512
// columns: 87 us instead of 130.
template <typename T, int G>
__global__ void __launch_bounds__(128) right_planes_kernel(const __grid_constant__ RightParams<G> rp) {
  grid_dependency_wait();
  using s = S<T>;
  const int q = G == 1 ? 0 : blockIdx.z;
  const int col = blockIdx.y;
  if (col >= rp.nvec[q]) return;  // the whole cluster
  __shared__ double part[2][32];
  __shared__ unsigned long long partm[32];
  const int rank = (int)blockIdx.x, cs = (int)gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  const int64_t K = rp.K[q], kp = (K + 7) / 8 * 8;
  const int64_t slice = ((K + cs - 1) / cs + 3) / 4 * 4;
  const int64_t k0 = rank * slice, k1 = k0 + slice < K ? k0 + slice : K;
  const T* x = (const T*)rp.X[q] + (int64_t)col * rp.ldx[q];
  auto load4 = [&](T (&v)[4], int64_t i) {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = i + j < k1 ? x[i + j] : s::zero();
  };
  // the sum (largest bit pattern) over the cluster of one value per warp
  auto spread = [&](uint32_t slot, unsigned long long bits) {
    if (lane < cs)
      asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(cluster_addr(slot + 8 * (4 * rank + warp), lane)), "l"(bits) : "memory");
    cluster_sync();
  };
  auto cluster_sum = [&](double v, int set) {
    v = warp_sum(v);
    spread(smem_u32(part[set]), (unsigned long long)__double_as_longlong(v));
    return warp_sum(lane < 4 * cs ? part[set][lane] : 0.0);
  };
  T v[4];
  const int64_t i0 = k0 + 4 * tid;
  load4(v, i0);  // stays in registers when the slice is 512 elements
  double a = (s::abs2(v[0]) + s::abs2(v[1])) + (s::abs2(v[2]) + s::abs2(v[3]));
  for (int64_t i = i0 + 512; i < k1; i += 512) {
    T u[4];
    load4(u, i);
    a += (s::abs2(u[0]) + s::abs2(u[1])) + (s::abs2(u[2]) + s::abs2(u[3]));
  }
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");  // every CTA of the cluster runs
  const double ss = cluster_sum(a, 0);
  int e;
  if (ss > 1e-250 && ss < 1e250) {
    e = norm_exponent(ss);
  } else {
    // largest magnitude (bit patterns, so that NaN and infinity compare largest), then scaled squares
    unsigned long long m = 0ull;
    for (int64_t i = k0 + tid; i < k1; i += 128) {
      const unsigned long long br = (unsigned long long)__double_as_longlong(fabs(s::re(x[i])));
      const unsigned long long bi = (unsigned long long)__double_as_longlong(fabs(s::im(x[i])));
      m = m > br ? m : br;
      m = m > bi ? m : bi;
    }
    for (int o = 16; o; o >>= 1) {
      const unsigned long long t = __shfl_xor_sync(0xffffffffu, m, o);
      m = m > t ? m : t;
    }
    spread(smem_u32(partm), m);
    m = 0ull;
    for (int w = 0; w < 4 * cs; ++w) m = m > partm[w] ? m : partm[w];
    int em = 0;
    if (m < 0x7ff0000000000000ull) frexp(__longlong_as_double((long long)m), &em);
    double b = 0.0;
    for (int64_t i = k0 + tid; i < k1; i += 128) {
      const double r = ldexp(s::re(x[i]), -em), c = ldexp(s::im(x[i]), -em);
      b += r * r + c * c;
    }
    b = cluster_sum(b, 1);
    e = m >= 0x7ff0000000000000ull ? NONFINITE : m == 0ull ? 0 : em + norm_exponent(b);
  }
  if (rank == 0 && tid == 0) rp.ex[q][col] = e;
  if (e == NONFINITE) e = 0;
  const int64_t plane = (int64_t)rp.nvec[q] * kp;
  __nv_bfloat16* out = (__nv_bfloat16*)rp.planes[q] + (int64_t)col * kp;
  if (i0 < k1) write_residues<T>(v, e, false, 0, NMOD, plane, out + i0);
  for (int64_t i = i0 + 512; i < k1; i += 512) {
    load4(v, i);
    write_residues<T>(v, e, false, 0, NMOD, plane, out + i);
  }
}

// ---------------------------------------------------------------- product kernel
constexpr int TM = 256;           // rows of a tile: 128 per CTA of the pair
constexpr int TN = 256;           // columns of a tile at most
constexpr int TK = 64;            // K per copy: 128 bytes of bf16 (the 128-byte swizzle atom)
constexpr int SK = 2 * TK;        // K per stage
constexpr int CHUNK = 8;          // stages per exact FP32 accumulation (1024 along K)
constexpr int A_HALF = 128 * TK * 2;  // this CTA's left rows of a stage, half of its K
constexpr int MAX_STAGES = 6;
constexpr int SMEM_RING = 216 * 1024;
constexpr int SMEM_BYTES = SMEM_RING + 1024 + 256;
constexpr int NTHREADS = 384;     // warps 0-3: copies, MMA issue, TMEM; warps 4-11: accumulator reduction
constexpr int EPI_WARPS = 8;
constexpr unsigned long long TIMEOUT_NS = 2000000000ull;

template <int G> struct Params {
  CUtensorMap tmA[G];
  CUtensorMap tmB[G];
  int8_t* R[G];
  int M[G], N[G], K[G], mt[G], nt[G], ldr[G];  // mt, nt: row and column tiles
  int nblk[G];                   // 32-column blocks of the product's columns
  int box_b[G];                  // right rows per copy
  int unit_begin[G + 1];
  int nprob, mod0, np;           // np: planes per modulus
  int stages, stage_bytes;       // ring of the launch (as many stages as its widest right copy leaves room for)
};

// column blocks of tile n: the nblk 32-column blocks spread evenly over nt tiles
__device__ __forceinline__ void tile_cols(int nblk, int nt, int n, int& n0, int& width) {
  const int base = nblk / nt, rem = nblk % nt;
  n0 = 32 * (n * base + min(n, rem));
  width = 32 * (base + (n < rem ? 1 : 0));
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// whether the phase is complete, without waiting
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
// bounded wait: false on expiry (which sets the launch's error flag) or when another role set it
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err) {
  unsigned long long t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 255) == 255) {
      if (*(volatile int*)err != 0) return false;
      const unsigned long long t = globaltimer();
      if (t0 == 0) t0 = t;
      else if (t - t0 > TIMEOUT_NS) {
        atomicOr(err, 1);
        return false;
      }
    }
  }
}
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
      "%5}], [%2];" ::"r"(dst),
      "l"((unsigned long long)map), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}
__device__ __forceinline__ void mma_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
// arrives on the barrier at this offset in the mask's CTAs when every MMA issued so far has completed
__device__ __forceinline__ void commit_to(uint32_t bar, uint32_t mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"((uint16_t)mask)
      : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
// waits for this thread's loads; r: the registers read next (in and out, so that no use moves before the wait)
__device__ __forceinline__ void tmem_wait_ld(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                 "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}

// two FP32 lanes per instruction
__device__ __forceinline__ uint64_t pack2(uint32_t a, uint32_t b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t both(float x) { return pack2(__float_as_uint(x), __float_as_uint(x)); }

// v - m round(v / m) on both lanes, exact for integers |v| <= 2^24 (result at most m / 2 + 1 in size)
struct Mod2 {
  uint64_t inv, negm, magic, negmagic;
  __device__ __forceinline__ explicit Mod2(int m)
      : inv(both(1.0f / (float)m)), negm(both(-(float)m)), magic(both(12582912.0f)), negmagic(both(-12582912.0f)) {}
  __device__ __forceinline__ uint64_t operator()(uint64_t v) const {
    const uint64_t q = add2(fma2(v, inv, magic), negmagic);
    return fma2(q, negm, v);
  }
};

// One CTA pair per unit (tile of one residue plane's product), persistent over the launch's units.  Each CTA copies
// its 128 left rows and half of the right rows of a stage; the leader issues the pair's MMAs into one of two
// accumulator sets (2 x 256 TMEM columns) and the eight reduction warps of each CTA take a finished chunk modulo m
// into FP32 registers while the next chunk accumulates in the other set.  At a unit's end they write residues
// (8-bit); the copies and MMAs of the next unit run meanwhile.
// What bounds it: the issuing thread, and L2 traffic.  Without any copy, a stage of four MMAs took 720 cycles at any
// width up to 256 columns (512 cycles of math): a barrier check costs it about 200 cycles and the MMA queue is only a
// few instructions deep.  So a stage holds 128 along K (eight MMAs), and the next stage's barrier is looked at between its halves,
// while four MMAs are queued.
// Register split: 384 threads at 168 (64512 at launch); warps 0-3 give down to 40, warps 4-11 take 232.
template <int G>
__global__ void __launch_bounds__(NTHREADS, 1)
    crt_gemm_kernel(const __grid_constant__ Params<G> gp, int* err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + SMEM_RING);             // leader's: both CTAs' copies of a stage have landed
  uint64_t* empty = full + MAX_STAGES;                        // each CTA's: the stage's MMAs are done
  uint64_t* acc_full = empty + MAX_STAGES;                    // each CTA's: a chunk is complete in set b
  uint64_t* acc_empty = acc_full + 2;                         // leader's: both CTAs have read set b
  uint64_t* drain = acc_empty + 2;
  uint32_t* tmem_slot = (uint32_t*)(drain + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank(), leader = 0;
  constexpr uint32_t both_ctas = 3;
  const int cluster = blockIdx.x / 2, nclusters = gridDim.x / 2;
  const int total = gp.unit_begin[gp.nprob];
  const int stages = gp.stages, stage_bytes = gp.stage_bytes;

  if (threadIdx.x == 0) {
    for (int i = 0; i < MAX_STAGES; ++i) {
      mbar_init(smem_u32(&full[i]), 1);
      mbar_init(smem_u32(&empty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&acc_full[i]), 1);
      mbar_init(smem_u32(&acc_empty[i]), 2 * EPI_WARPS);
    }
    mbar_init(smem_u32(drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  cluster_sync();
  fence_after();
  grid_dependency_wait();
  const uint32_t tmem = *tmem_slot;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == 0 && lane == 0) {
      // ---------------------------------------------------------- copies
      int it = 0, sl = 0;  // stages so far, slot
      uint32_t ph = 0;     // parity of the slot's round
      bool ok = true;
      int prob = 0;
      auto advance = [&]() {
        ++it;
        if (++sl == stages) {
          sl = 0;
          ph ^= 1;
        }
      };
      for (int unit = cluster; unit < total && ok; unit += nclusters) {
        while (G > 1 && unit >= gp.unit_begin[prob + 1]) ++prob;
        const int tiles = gp.mt[prob] * gp.nt[prob];
        const int local = unit - gp.unit_begin[prob];
        const int plane = local / tiles, t = local - plane * tiles;
        const int m = t / gp.nt[prob], n = t - m * gp.nt[prob];
        int n0, width;
        tile_cols(gp.nblk[prob], gp.nt[prob], n, n0, width);
        const int box = gp.box_b[prob], K = gp.K[prob];
        const int y_a = m * TM + (int)rank * 128, y_b = n0 + (int)rank * (width >> 1);
        const int z_b = gp.mod0 * gp.np + plane;
        const uint32_t half_bytes = (uint32_t)(A_HALF + box * TK * 2);
        for (int k0 = 0; k0 < K; k0 += SK) {
          if (!mbar_wait(smem_u32(&empty[sl]), ph ^ 1, err)) {
            ok = false;
            break;
          }
          const bool two = k0 + TK < K;  // a second half within K
          if (rank == 0) mbar_expect_tx(smem_u32(&full[sl]), 2 * (two ? 2 * half_bytes : half_bytes));
          const uint32_t dst = smem_u32(smem + sl * stage_bytes), bar = cluster_addr(smem_u32(&full[sl]), leader);
          const uint32_t dst_b = dst + 2 * A_HALF, b_half = (uint32_t)(box * TK * 2);
          tma_load_pair(dst, &gp.tmA[prob], bar, k0, y_a, plane);
          tma_load_pair(dst_b, &gp.tmB[prob], bar, k0, y_b, z_b);
          if (two) {
            tma_load_pair(dst + A_HALF, &gp.tmA[prob], bar, k0 + TK, y_a, plane);
            tma_load_pair(dst_b + b_half, &gp.tmB[prob], bar, k0 + TK, y_b, z_b);
          }
          advance();
        }
      }
      if (ok) {
        // every stage's release has arrived in this CTA before it may exit
        for (int i = 0; i < stages && ok; ++i) {
          ok = mbar_wait(smem_u32(&empty[sl]), ph ^ 1, err);
          advance();
        }
      } else if (rank == 0) {
        // aborted: the copies in flight (this CTA's and its peer's) land before the pair exits
        for (int j = it > stages ? it - stages : 0; j < it; ++j) {
          const unsigned long long t0 = globaltimer();
          while (!mbar_try(smem_u32(&full[j % stages]), (j / stages) & 1) && globaltimer() - t0 < TIMEOUT_NS) {
          }
        }
      }
    } else if (warp == 1 && lane == 0 && rank == 0) {
      // ---------------------------------------------------------- MMA issue
      int chunk = 0, sl = 0;
      uint32_t ph = 0;
      bool ready = false;  // the slot's copies are known to have landed
      bool ok = true;
      int prob = 0;
      for (int unit = cluster; unit < total && ok; unit += nclusters) {
        while (G > 1 && unit >= gp.unit_begin[prob + 1]) ++prob;
        const int tiles = gp.mt[prob] * gp.nt[prob];
        const int local = unit - gp.unit_begin[prob];
        const int n = (local % tiles) % gp.nt[prob];
        int n0, width;
        tile_cols(gp.nblk[prob], gp.nt[prob], n, n0, width);
        const uint32_t idesc = oz::idesc_bf16(TM, width);
        const int K = gp.K[prob];
        const uint32_t b_half = (uint32_t)(gp.box_b[prob] * TK * 2);
        int in_chunk = 0;
        for (int k0 = 0; k0 < K; k0 += SK) {
          const int b = chunk & 1;
          if (in_chunk == 0) {
            if (!mbar_wait(smem_u32(&acc_empty[b]), ((chunk >> 1) & 1) ^ 1, err)) {
              ok = false;
              break;
            }
            fence_after();
          }
          if (!ready && !mbar_wait(smem_u32(&full[sl]), ph, err)) {
            ok = false;
            break;
          }
          fence_after();
          const uint32_t base = smem_u32(smem + sl * stage_bytes);
          const uint64_t ad = sw128_desc(base), bd = sw128_desc(base + 2 * A_HALF);
          const uint32_t d = tmem + (uint32_t)(b * 256);
#pragma unroll
          for (int ks = 0; ks < TK / 16; ++ks)
            mma_pair(d, ad + (uint64_t)(ks * 2), bd + (uint64_t)(ks * 2), idesc, (in_chunk != 0 || ks != 0) ? 1u : 0u);
          // the next stage's barrier, while these run
          const uint32_t slot = smem_u32(&empty[sl]);
          if (++sl == stages) {
            sl = 0;
            ph ^= 1;
          }
          ready = mbar_test(smem_u32(&full[sl]), ph);
          if (k0 + TK < K) {
            const uint64_t ad2 = ad + (uint64_t)(A_HALF >> 4), bd2 = bd + (uint64_t)(b_half >> 4);
#pragma unroll
            for (int ks = 0; ks < TK / 16; ++ks) mma_pair(d, ad2 + (uint64_t)(ks * 2), bd2 + (uint64_t)(ks * 2), idesc, 1u);
          }
          commit_to(slot, both_ctas);
          if (++in_chunk == CHUNK || k0 + SK >= K) {
            commit_to(smem_u32(&acc_full[b]), both_ctas);
            ++chunk;
            in_chunk = 0;
          }
        }
      }
      // every MMA is done before TMEM is freed
      commit_to(smem_u32(drain), both_ctas);
      const unsigned long long t0 = globaltimer();
      while (!mbar_try(smem_u32(drain), 0) && globaltimer() - t0 < TIMEOUT_NS) {
      }
    }
    __syncwarp();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
    // ------------------------------------------------------------ chunk reduction
    const int ew = warp - 4, q = ew & 3, half = ew >> 2;  // TMEM lane quadrant, column half
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    const uint32_t rel0 = cluster_addr(smem_u32(&acc_empty[0]), leader), rel1 = cluster_addr(smem_u32(&acc_empty[1]), leader);
    int chunk = 0;
    bool ok = true;
    int prob = 0;
    for (int unit = cluster; unit < total && ok; unit += nclusters) {
      while (G > 1 && unit >= gp.unit_begin[prob + 1]) ++prob;
      const int nt = gp.nt[prob];
      const int tiles = gp.mt[prob] * nt;
      const int local = unit - gp.unit_begin[prob];
      const int plane = local / tiles, t = local - plane * tiles;
      const int m = t / nt, n = t - m * nt;
      int n0, width;
      tile_cols(gp.nblk[prob], nt, n, n0, width);
      const int hc = width >> 1;  // this warp's columns: [half hc, half hc + hc)
      const Mod2 mod(cT.m[gp.mod0 + plane / gp.np]);
      const int nchunk = (gp.K[prob] + CHUNK * SK - 1) / (CHUNK * SK);
      uint64_t acc[64];
#pragma unroll
      for (int j = 0; j < 64; ++j) acc[j] = 0ull;
      for (int c = 0; c < nchunk; ++c, ++chunk) {
        const int b = chunk & 1;
        // one verdict per warp: the loads below need every lane
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&acc_full[b]), (chunk >> 1) & 1, err));
        if (!ok) break;
        fence_after();
        const uint32_t src = lane_addr + (uint32_t)(b * 256 + half * hc);
        // the next 32 columns load while these are reduced (a load's wait covers every load issued before it)
        uint32_t r[2][32];
        tmem_ld32(src, r[0]);
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          if (g * 32 >= hc) continue;
          tmem_wait_ld(r[g & 1]);
          if (g * 32 + 32 < hc) {
            tmem_ld32(src + (uint32_t)(g * 32 + 32), r[(g + 1) & 1]);
          } else {  // every read of this set is done: release it before the arithmetic
            fence_before();
            __syncwarp();
            if (lane == 0) arrive_cluster(b ? rel1 : rel0);
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const uint64_t v = pack2(r[g & 1][2 * j], r[g & 1][2 * j + 1]);
            acc[g * 16 + j] = add2(acc[g * 16 + j], mod(v));
          }
        }
      }
      if (!ok) break;
      const int row = m * TM + (int)rank * 128 + q * 32 + lane;
      if (row < gp.M[prob]) {
        const int N = gp.N[prob], ldr = gp.ldr[prob];
        const int c0 = n0 + half * hc;
        int8_t* out = gp.R[prob] + ((int64_t)(gp.mod0 * gp.np + plane) * N + c0) * ldr + row;
#pragma unroll
        for (int j = 0; j < 64; ++j) {
          // sums of at most 128 per chunk: exact in FP32; residues at most 128 in size, +128 (modulo 256 only) wraps
          const uint64_t v = mod(acc[j]);
          const float lo = __uint_as_float((uint32_t)v), hi = __uint_as_float((uint32_t)(v >> 32));
          if (2 * j < hc && c0 + 2 * j < N) out[(int64_t)(2 * j) * ldr] = (int8_t)(int)lo;
          if (2 * j + 1 < hc && c0 + 2 * j + 1 < N) out[(int64_t)(2 * j + 1) * ldr] = (int8_t)(int)hi;
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  cluster_sync();
  fence_after();
  if (threadIdx.x == 0) {
    // the leader's last commit has arrived in this CTA too
    const unsigned long long t0 = globaltimer();
    while (!mbar_try(smem_u32(drain), 0) && globaltimer() - t0 < TIMEOUT_NS) {
    }
  }
  __syncthreads();
  if (warp == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  cluster_sync();
}

// ---------------------------------------------------------------- reconstruction
// Double nearest to X 2^e for a signed 128-bit integer X (round to nearest even up to sticky bits below 2^-63 of the
// leading one), by integer operations; exponents outside the normal range go through ldexp.
__device__ __forceinline__ double to_double(__int128 x, int e) {
  const bool neg = x < 0;
  u128 u = neg ? (u128)(-x) : (u128)x;
  uint64_t hi = (uint64_t)(u >> 64), lo = (uint64_t)u;
  if ((hi | lo) == 0ull) return 0.0;
  int sh;  // u = top 2^(64 - sh)
  uint64_t top;
  if (hi) {
    sh = __clzll((long long)hi);
    top = sh ? (hi << sh) | (lo >> (64 - sh)) : hi;
  } else {
    sh = 64 + __clzll((long long)lo);
    top = lo << (sh - 64);
  }
  const uint64_t r = (top >> 11) + ((top >> 10) & 1ull & (uint64_t)(((top & 0x3ffull) != 0ull) | ((top >> 11) & 1ull)));
  // value = r 2^(75 - sh + e); r in [2^52, 2^53]
  const int ex = 75 - sh + e + 1075;  // biased exponent of r's leading bit at 2^52
  double v;
  if (ex >= 1 && ex <= 2045)
    v = __longlong_as_double((long long)(r + ((uint64_t)(ex - 1) << 52)));
  else
    v = ldexp((double)r, ex - 1075);
  return neg ? -v : v;
}

// The product entry (in units of 2^e) whose residues, each plus BIAS, have been summed against the weights' limbs.
__device__ __forceinline__ double reconstruct(const uint64_t (&a)[4], int e) {
  const uint64_t s0 = a[0] + cT.off[0];
  const uint64_t s1 = a[1] + cT.off[1] + (s0 >> 32);
  const uint64_t s2 = a[2] + cT.off[2] + (s1 >> 32);
  const uint64_t s3 = a[3] + cT.off[3] + (s2 >> 32);
  // T = s3 2^96 + ...; T / M < 2^14 lies within 0.33 of an integer; FP32 of its top 28 bits is off by 2^-9 at most
  const uint32_t q = (uint32_t)__float2int_rn((float)(uint32_t)(s3 >> 16) * cT.q);
  u128 t = ((u128)((s3 << 32) | (uint32_t)s2) << 64) | (u128)((s1 << 32) | (uint32_t)s0);
  const u128 M = ((u128)cT.Mhi << 64) | cT.Mlo;
  t -= M * (u128)q;
  return to_double((__int128)t, e);
}

// ROWS = 4: four rows per thread (one 4-byte load per plane); HBM-bound on the residues (1 byte per plane and entry), the
// weights' limb products run on the integer pipe.  ROWS = 1: one row per thread, for products too small to fill the
// SMs otherwise, with every plane's load in flight at once.
template <int G> struct CombineParams {
  const int8_t* R[G];
  const int* lex[G];
  const int* rex[G];
  Epi e[G];
  int M[G], N[G], ldr[G];
};
template <bool CPLX, int ROWS, int G>
__global__ void __launch_bounds__(64) combine_kernel(const __grid_constant__ CombineParams<G> cp) {
  grid_dependency_wait();
  constexpr int NP = CPLX ? 3 : 1, NC = CPLX ? 2 : 1;
  const int prob = G == 1 ? 0 : blockIdx.z;
  const int M = cp.M[prob], N = cp.N[prob], ldr = cp.ldr[prob];
  const int i0 = ROWS * (blockIdx.x * blockDim.x + threadIdx.x), j = blockIdx.y;
  if (i0 >= M || j >= N) return;
  const int* __restrict__ lex = cp.lex[prob];
  const Epi& ep = cp.e[prob];
  const int8_t* __restrict__ src = cp.R[prob] + (int64_t)j * ldr + i0;
  const int64_t plane = (int64_t)N * ldr;
  uint64_t acc[ROWS][NC][4];
#pragma unroll
  for (int r = 0; r < ROWS; ++r)
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
      for (int l = 0; l < 4; ++l) acc[r][c][l] = 0ull;
  constexpr int BATCH = ROWS == 1 ? NMOD : 4;  // moduli whose loads are in flight together
#pragma unroll
  for (int i0m = 0; i0m < NMOD; i0m += BATCH) {
    int8_t p[BATCH][NP][ROWS];
#pragma unroll
    for (int b = 0; b < BATCH; ++b)
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        const int8_t* q = src + (int64_t)((i0m + b) * NP + k) * plane;
        if (ROWS == 4) {
          const char4 v = *reinterpret_cast<const char4*>(q);
          p[b][k][0] = v.x;
          p[b][k][ROWS > 1 ? 1 : 0] = v.y;
          p[b][k][ROWS > 2 ? 2 : 0] = v.z;
          p[b][k][ROWS > 3 ? 3 : 0] = v.w;
        } else {
          p[b][k][0] = *q;
        }
      }
#pragma unroll
    for (int b = 0; b < BATCH; ++b)
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        const int p0 = p[b][0][r];
        uint32_t v[NC];
        if (CPLX) {
          const int p1 = p[b][NP - 2][r], p2 = p[b][NP - 1][r];
          v[0] = (uint32_t)(p0 - p1 + BIAS);
          v[NC - 1] = (uint32_t)(p2 - p0 - p1 + BIAS);
        } else {
          v[0] = (uint32_t)(p0 + BIAS);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
          for (int l = 0; l < 4; ++l) acc[r][c][l] += (uint64_t)v[c] * cT.w[i0m + b][l];
      }
  }
  const int ej = cp.rex[prob][j];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const int i = i0 + r;
    if (i >= M) return;
    const int ei = lex[i];
    const bool bad = ei == NONFINITE || ej == NONFINITE;
    double* C = (double*)ep.C + (i + (int64_t)j * ep.ldc) * NC;
    const double g = ep.Y ? ep.gamma * (ep.ycol ? ep.ycol[j] : 1.0) : 0.0;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      double v = bad ? __longlong_as_double(0x7ff8000000000000ll) : reconstruct(acc[r][c], ei + ej - 124);
      double out = ep.alpha * v;
      if (ep.Y) out += g * ((const double*)ep.Y)[(i + (int64_t)j * ep.ldy) * NC + c];
      if (ep.Z) out += ep.beta * ((const double*)ep.Z)[(i + (int64_t)j * ep.ldz) * NC + c];
      C[c] = out;
    }
  }
}

// ---------------------------------------------------------------- host side
template <typename T>
void scales(cudaStream_t st, bool by_rows, int64_t nvec, int64_t K, const T* X, int64_t ldx, int* ex) {
  if (by_rows)
    launch_pdl(row_exponent_kernel<T>, ceil_div(nvec, 32), 256, 0, st, nvec, K, X, ldx, ex);
  else
    launch_pdl(col_exponent_kernel<T>, (unsigned)nvec, 256, 0, st, K, X, ldx, ex);
  CHASE_CHECK_LAUNCH();
}

template <typename T>
void residues(cudaStream_t st, bool by_rows, bool conj, int64_t nvec, int64_t K, const T* X, int64_t ldx, const int* ex,
              int mod0, int nmod, void* planes) {
  const int64_t kp = kpad(K);
  if (by_rows) {
    const dim3 grid(ceil_div(nvec, 32), ceil_div(K, 32));
    CHASE_REQUIRE(grid.y <= 65535, 1, "residues: vectors too long");
    launch_pdl(residues_rows_kernel<T>, grid, 256, 0, st, nvec, K, kp, X, ldx, ex, conj ? 1 : 0, mod0, nmod,
                                                  (__nv_bfloat16*)planes);
  } else {
    CHASE_REQUIRE(nvec <= 65535, 1, "residues: too many vectors");
    const dim3 grid(ceil_div(K, 512), (unsigned)nvec);
    launch_pdl(residues_cols_kernel<T>, grid, 128, 0, st, K, kp, nvec, X, ldx, ex, conj ? 1 : 0, mod0, nmod,
                                                  (__nv_bfloat16*)planes);
  }
  CHASE_CHECK_LAUNCH();
}

// CTA pairs the device keeps resident (0: none)
template <int G> static int max_pairs() {
  static std::once_flag once;
  static cudaError_t err = cudaSuccess;
  static int got = 0;
  std::call_once(once, []() {
    err = cudaFuncSetAttribute(crt_gemm_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (err != cudaSuccess) return;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 2;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(2, 1, 1);
    cfg.blockDim = dim3(NTHREADS, 1, 1);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    err = cudaOccupancyMaxActiveClusters(&got, crt_gemm_kernel<G>, &cfg);
  });
  CHASE_CUDA(err);
  return got;
}

template <int G> static void launch(cudaStream_t st, const Product* ops, int nops, bool cplx, int mod0, int nmod, int* err) {
  static thread_local Params<G> gp;  // large for G > 1: built in thread-local host memory
  const int np = planes(cplx);
  int64_t units = 0;
  int box_max = 0;
  for (int p = 0; p < nops; ++p) {
    const Product& o = ops[p];
    const int64_t kp = kpad(o.K);
    const int nblk = (int)ceil_div(o.N, 32), nt = (int)ceil_div(nblk, TN / 32);
    const int box = 16 * (int)ceil_div(nblk, nt);
    gp.tmA[p] = make_tmap_bf16(o.lpl, o.K, kp, o.M, nmod * np, TK, 128, 1, CU_TENSOR_MAP_SWIZZLE_128B);
    gp.tmB[p] = make_tmap_bf16(o.rpl, o.K, kp, o.N, NMOD * np, TK, box, 1, CU_TENSOR_MAP_SWIZZLE_128B);
    gp.R[p] = (int8_t*)o.res;
    gp.M[p] = (int)o.M;
    gp.N[p] = (int)o.N;
    gp.K[p] = (int)o.K;
    box_max = std::max(box_max, box);
    gp.mt[p] = (int)ceil_div(o.M, TM);
    gp.nt[p] = nt;
    gp.nblk[p] = nblk;
    gp.box_b[p] = box;
    gp.ldr[p] = (int)rpad(o.M);
    gp.unit_begin[p] = (int)units;
    units += (int64_t)gp.mt[p] * nt * np * nmod;
    CHASE_REQUIRE(units <= 0x7fffffff, 1, "residue product: too many tiles");
  }
  gp.unit_begin[nops] = (int)units;
  gp.nprob = nops;
  gp.mod0 = mod0;
  gp.np = np;
  gp.stage_bytes = 2 * (A_HALF + box_max * TK * 2);
  gp.stages = std::min(MAX_STAGES, SMEM_RING / gp.stage_bytes);
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[2] = {{}, pdl_attribute()};
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(2 * std::min<int64_t>(units, std::max(1, max_pairs<G>()))), 1, 1);
  cfg.blockDim = dim3(NTHREADS, 1, 1);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  CHASE_CUDA(cudaLaunchKernelEx(&cfg, crt_gemm_kernel<G>, gp, err));
  CHASE_CHECK_LAUNCH();
}

template <bool CPLX>
void multiply(cudaStream_t st, const Product* ops, int nops, int mod0, int nmod, int* err) {
  for (int q0 = 0; q0 < nops; q0 += MAXG) {
    const int cnt = std::min(MAXG, nops - q0);
    if (cnt == 1)
      launch<1>(st, ops + q0, 1, CPLX, mod0, nmod, err);
    else
      launch<MAXG>(st, ops + q0, cnt, CPLX, mod0, nmod, err);
  }
}

template <bool CPLX, int ROWS, int G> static void launch_combine(cudaStream_t st, const Product* ops, int nops) {
  static thread_local CombineParams<G> cp;
  int64_t M = 0, N = 0;
  for (int p = 0; p < nops; ++p) {
    const Product& o = ops[p];
    CHASE_REQUIRE(o.N <= 65535, 1, "residue product: too many columns");
    cp.R[p] = (const int8_t*)o.res;
    cp.lex[p] = o.lex;
    cp.rex[p] = o.rex;
    cp.e[p] = o.e;
    cp.M[p] = (int)o.M;
    cp.N[p] = (int)o.N;
    cp.ldr[p] = (int)rpad(o.M);
    M = std::max(M, o.M);
    N = std::max(N, o.N);
  }
  launch_pdl(combine_kernel<CPLX, ROWS, G>, dim3(ceil_div(M, 64 * ROWS), (unsigned)N, (unsigned)nops), 64, 0, st, cp);
  CHASE_CHECK_LAUNCH();
}

template <bool CPLX> void combine(cudaStream_t st, const Product* ops, int nops) {
  for (int q0 = 0; q0 < nops; q0 += MAXG) {
    const int cnt = std::min(MAXG, nops - q0);
    int64_t entries = 0;
    for (int q = q0; q < q0 + cnt; ++q) entries += ops[q].M * ops[q].N;
    // One row per thread up to 2^19 entries (four rows make about 8 two-warp blocks per SM there): complex,
    // 512 x 40 entries 4.3 us instead of 12, 3001 x 100 7.5 instead of 14; four rows read the planes in wider loads
    // and win above.
    const bool small = entries <= (1 << 19);
    if (cnt == 1 && small) launch_combine<CPLX, 1, 1>(st, ops + q0, 1);
    else if (cnt == 1) launch_combine<CPLX, 4, 1>(st, ops + q0, 1);
    else if (small) launch_combine<CPLX, 1, MAXG>(st, ops + q0, cnt);
    else launch_combine<CPLX, 4, MAXG>(st, ops + q0, cnt);
  }
}

template <typename T, int G> static void launch_right(cudaStream_t st, const Product* ops, int nops) {
  static thread_local RightParams<G> rp;
  int64_t K = 0, N = 0;
  for (int p = 0; p < nops; ++p) {
    const Product& o = ops[p];
    CHASE_REQUIRE(o.N <= 65535, 1, "residues: too many vectors");
    rp.X[p] = o.X;
    rp.ldx[p] = o.ldx;
    rp.ex[p] = o.rex;
    rp.planes[p] = o.rpl;
    rp.nvec[p] = (int)o.N;
    rp.K[p] = (int)o.K;
    K = std::max(K, o.K);
    N = std::max(N, o.N);
  }
  int cs = 1;
  while (cs < 8 && 512 * cs < K) cs *= 2;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[2] = {{}, pdl_attribute()};
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(cs, (unsigned)N, (unsigned)nops);
  cfg.blockDim = dim3(128, 1, 1);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  CHASE_CUDA(cudaLaunchKernelEx(&cfg, right_planes_kernel<T, G>, rp));
  CHASE_CHECK_LAUNCH();
}

template <typename T> void right_planes(cudaStream_t st, const Product* ops, int nops) {
  for (int q0 = 0; q0 < nops; q0 += MAXG) {
    const int cnt = std::min(MAXG, nops - q0);
    if (cnt == 1) launch_right<T, 1>(st, ops + q0, 1);
    else launch_right<T, MAXG>(st, ops + q0, cnt);
  }
}

#define INST(T)                                                                                                  \
  template void scales<T>(cudaStream_t, bool, int64_t, int64_t, const T*, int64_t, int*);                         \
  template void residues<T>(cudaStream_t, bool, bool, int64_t, int64_t, const T*, int64_t, const int*, int, int, void*); \
  template void right_planes<T>(cudaStream_t, const Product*, int);
INST(double)
INST(double2)
#undef INST
template void multiply<false>(cudaStream_t, const Product*, int, int, int, int*);
template void multiply<true>(cudaStream_t, const Product*, int, int, int, int*);
template void combine<false>(cudaStream_t, const Product*, int);
template void combine<true>(cudaStream_t, const Product*, int);

}  // namespace crt
}  // namespace chase
