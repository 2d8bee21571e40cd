// Lanczos spectral-bound estimation (Algorithm 1, line 2) on the device.
//
// All runs advance together, two launches per step: the product of A with one vector per run (hemv_mma_kernel, A
// streamed once per step), and the rest of the step (lanczos_step_kernel, one cluster of CTAs per run): three-term
// update, one classical Gram-Schmidt reorthogonalisation against the run's basis, normalisation.  The tridiagonal T
// of each run is diagonalised by implicit QL, and one block computes b_sup = max(theta_max + |beta_last|),
// mu_1 = min theta_min, theta_max and the density-of-states quantile mu_ne = smallest pooled Ritz value whose
// cumulative weight (1/runs) sum tau_j^2 reaches ne/n, clamped into (mu_1, b_sup) by 1e-3 of the spectral span.
#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "kernels.h"

namespace chase {

constexpr int LZ_MAXR = 8;      // runs
constexpr int LZ_MAXS = 64;     // steps

// ---------------------------------------------------------------- fixed-point operands
// A value x with |x| < 2^e is held as r = round(x 2^(54 - e)), |r| <= 2^54, in balanced base-256 digits
// r = sum_t d_t 256^t, t = 0..6, d_t in [-128, 127]: adding 128 to every digit makes them the bytes of an integer.
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

// part[c][r][i] = sum_{j in chunk c} A[i,j] X[j,r] for up to 8 real columns (4 complex runs, re and im interleaved).
// FP64 multiply-adds bound a plain version (GB300: 2 per SM and clock; four complex vectors take 16 per element of A,
// 1.78 ms at n = 8192 where reading A takes 0.16 ms), and 64-bit integer ones are only 8 times faster (1.03 ms).
// Here A (per row) and X (per run) are 55-bit fixed-point numbers in seven 8-bit digits; the digits of A are made in
// registers, straight into the fragments of mma.sync m16n8k16 (f16 digits, FP32 sums), whose 8 columns are the
// vectors.  Digit pairs up to level 7 (34 of 49; the rest is below 2^-56 of the scales' product) go to one accumulator
// per level, exact over 64 columns (at most 8 pairs x 2 planes x 64 products of 2^14 < 2^24), then to integers.
constexpr int HEMV_ROWS = 64;    // 16 per warp
constexpr int HEMV_FOLD = 4;     // 16-column steps between folds
constexpr int NLEV = 8;

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// digits t = 0..6 of two fixed-point numbers as f16 pairs (exact: 1024 + byte - 1152)
__device__ __forceinline__ void digit_pairs(long long r0, long long r1, uint32_t (&out)[NDIG]) {
  const unsigned long long w0 = (unsigned long long)r0 + DIGIT_BIAS, w1 = (unsigned long long)r1 + DIGIT_BIAS;
  const uint32_t l0 = (uint32_t)w0, l1 = (uint32_t)w1, h0 = (uint32_t)(w0 >> 32), h1 = (uint32_t)(w1 >> 32);
  const uint32_t b[4] = {__byte_perm(l0, l1, 0x5140), __byte_perm(l0, l1, 0x7362), __byte_perm(h0, h1, 0x5140),
                         __byte_perm(h0, h1, 0x7362)};
  const __half2 off = __half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));  // 1152
#pragma unroll
  for (int t = 0; t < NDIG; ++t) {
    const uint32_t v = __byte_perm(b[t >> 1], 0x64646464u, (t & 1) ? 0x4342 : 0x4140);
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&v), off);
    out[t] = *reinterpret_cast<const uint32_t*>(&h);
  }
}

// Vectors as B fragments: for every 16 columns of A (rows of X), digit and lane the lane's registers
// (k = 2t, 2t + 1 | 2t + 8, 2t + 9 of vector column g; lane = 4 g + t).  Complex: form 0 multiplies Re A
// (columns re, im of each run), form 1 multiplies Im A (columns -im, re).
template <typename T> struct Frag {
  static constexpr int FORMS = S<T>::cplx ? 2 : 1;
  static constexpr int RUNS = S<T>::cplx ? 4 : 8;       // runs per group of 8 columns
  static constexpr int LANE_HALVES = FORMS * 4;         // halves per lane and digit
  static constexpr int STEP_HALVES = NDIG * 32 * LANE_HALVES;
};
inline int64_t frag_halves(int64_t n, bool cplx, int runs) {
  const int per = cplx ? 4 : 8;
  return (n + 15) / 16 * ((runs + per - 1) / per) * (NDIG * 32 * (cplx ? 8 : 4));
}
// writes digit t = 0..6 of entry j of a run's vector
template <typename T>
__device__ __forceinline__ void write_frag(__half* X, int64_t nk16, int64_t j, int run, long long re, long long im) {
  using F = Frag<T>;
  const int grp = run / F::RUNS, r = run % F::RUNS, kk = (int)(j & 15);
  __half* base = X + ((int64_t)grp * nk16 + (j >> 4)) * F::STEP_HALVES;
  const int reg = kk >> 3, t4 = (kk & 7) >> 1, half = kk & 1;
  unsigned long long wr = (unsigned long long)re + DIGIT_BIAS, wi = (unsigned long long)im + DIGIT_BIAS;
  for (int t = 0; t < NDIG; ++t, wr >>= 8, wi >>= 8) {
    const __half dr = __int2half_rn((int)(wr & 0xff) - 128);
    __half* o = base + (int64_t)t * 32 * F::LANE_HALVES;
    if (F::FORMS == 2) {
      const __half di = __int2half_rn((int)(wi & 0xff) - 128);
      __half* c0 = o + ((2 * r) * 4 + t4) * F::LANE_HALVES + reg * 2 + half;
      __half* c1 = o + ((2 * r + 1) * 4 + t4) * F::LANE_HALVES + reg * 2 + half;
      c0[0] = dr;
      c1[0] = di;
      c0[4] = __hneg(di);
      c1[4] = dr;
    } else {
      o[(r * 4 + t4) * F::LANE_HALVES + reg * 2 + half] = dr;
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(2 * HEMV_ROWS) hemv_mma_kernel(int64_t n, const T* __restrict__ A, int64_t lda,
                                                                  const unsigned* __restrict__ rmax,
                                                                  const __half* __restrict__ X,
                                                                  const int* __restrict__ xe, int cols, int runs,
                                                                  T* part) {
  using s = S<T>;
  using F = Frag<T>;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
  const int64_t row0 = (int64_t)blockIdx.x * HEMV_ROWS + warp * 16 + g, row1 = row0 + 8;
  const int64_t jbeg = (int64_t)blockIdx.y * cols, jend = jbeg + cols < n ? jbeg + cols : n;
  const int grp = blockIdx.z;
  const int64_t nk16 = (n + 15) / 16;
  const bool l0 = row0 < n, l1 = row1 < n;
  const int e0 = l0 ? exponent_of_bits((unsigned long long)rmax[row0] << 32 | 0xffffffffull) : 0;
  const int e1 = l1 ? exponent_of_bits((unsigned long long)rmax[row1] << 32 | 0xffffffffull) : 0;
  const int s0 = e0 == LZ_NONFINITE ? 0 : e0, s1 = e1 == LZ_NONFINITE ? 0 : e1;
  float acc[NLEV][4];
  int sum[NLEV][4];
#pragma unroll
  for (int l = 0; l < NLEV; ++l)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      acc[l][q] = 0.0f;
      sum[l][q] = 0;
    }
  const __half* xb = X + ((int64_t)grp * nk16 + jbeg / 16) * F::STEP_HALVES + lane * F::LANE_HALVES;
  const T* a0 = A + row0 + (jbeg + 2 * t4) * lda;
  int fold = 0;
  // this lane's 2 x 4 entries of the step: rows row0, row1; columns 2t, 2t + 1, 2t + 8, 2t + 9
  T v[2][4], w[2][4];
  auto load = [&](int64_t j, const T* a, T (&o)[2][4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int dj = (q & 1) + 8 * (q >> 1);
      const bool in = j + 2 * t4 + dj < jend;
      o[0][q] = in && l0 ? a[dj * lda] : s::zero();
      o[1][q] = in && l1 ? a[dj * lda + 8] : s::zero();
    }
  };
  load(jbeg, a0, v);
  for (int64_t j = jbeg; j < jend; j += 16) {
    a0 += 16 * lda;
    load(j + 16, a0, w);  // past the end: zeros, no access
    uint32_t bf[NDIG][F::FORMS][2];
#pragma unroll
    for (int u = 0; u < NDIG; ++u) {
      const __half* p = xb + u * 32 * F::LANE_HALVES;
      if (F::FORMS == 2) {
        const uint4 q = *reinterpret_cast<const uint4*>(p);
        bf[u][0][0] = q.x;
        bf[u][0][1] = q.y;
        bf[u][F::FORMS - 1][0] = q.z;
        bf[u][F::FORMS - 1][1] = q.w;
      } else {
        const uint2 q = *reinterpret_cast<const uint2*>(p);
        bf[u][0][0] = q.x;
        bf[u][0][1] = q.y;
      }
    }
    xb += F::STEP_HALVES;
#pragma unroll
    for (int f = 0; f < F::FORMS; ++f) {
      uint32_t ad[4][NDIG];  // A registers 0..3 (row0 | row1, then columns + 8) by digit
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int rr = r & 1, c = (r >> 1) * 2, sc = rr ? s1 : s0;
        const double x0 = f ? s::im(v[rr][c]) : s::re(v[rr][c]), x1 = f ? s::im(v[rr][c + 1]) : s::re(v[rr][c + 1]);
        digit_pairs(to_fixed(x0, sc), to_fixed(x1, sc), ad[r]);
      }
#pragma unroll
      for (int t = NDIG - 1; t >= 0; --t) {
        const uint32_t a[4] = {ad[0][t], ad[1][t], ad[2][t], ad[3][t]};
#pragma unroll
        for (int u = NDIG - 1; u >= 0; --u) {
          const int lev = 2 * (NDIG - 1) - t - u;
          if (lev < NLEV) mma_16816(acc[lev], a, bf[u][f][0], bf[u][f][1]);
        }
      }
    }
    if (++fold == HEMV_FOLD || j + 16 >= jend) {
      fold = 0;
#pragma unroll
      for (int l = 0; l < NLEV; ++l)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          sum[l][q] += __float2int_rn(acc[l][q]);
          acc[l][q] = 0.0f;
        }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) v[r][q] = w[r][q];
  }
  // levels 0-3 and 4-7 as two integers; value = (hi 2^32 + lo) 2^40, in units of 2^(ea + ex - 108)
  double o[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const long long hi = ((long long)sum[0][q] << 24) + ((long long)sum[1][q] << 16) + ((long long)sum[2][q] << 8) + sum[3][q];
    const long long lo = ((long long)sum[4][q] << 24) + ((long long)sum[5][q] << 16) + ((long long)sum[6][q] << 8) + sum[7][q];
    o[q] = (double)hi * 4294967296.0 + (double)lo;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    // accumulator columns 2t, 2t + 1: complex, one run's re and im; real, two runs
    const int run = F::FORMS == 2 ? grp * F::RUNS + t4 : grp * F::RUNS + 2 * t4 + (q & 1);
    const int ea = q < 2 ? e0 : e1;
    if (run >= runs) continue;
    const int ex = xe[run];
    o[q] = ea == LZ_NONFINITE || ex == LZ_NONFINITE ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(o[q], ea + ex - 68);
  }
  T* out = part + (int64_t)blockIdx.y * runs * n;
  if (F::FORMS == 2) {
    const int run = grp * F::RUNS + t4;
    if (run < runs) {
      if (l0) out[(int64_t)run * n + row0] = s::make(o[0], o[1]);
      if (l1) out[(int64_t)run * n + row1] = s::make(o[2], o[3]);
    }
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int run = grp * F::RUNS + 2 * t4 + (q & 1);
      const bool in = q < 2 ? l0 : l1;
      if (run < runs && in) out[(int64_t)run * n + (q < 2 ? row0 : row1)] = s::make(o[q], 0.0);
    }
  }
}

// Columns per hemv block (a multiple of 64): enough blocks for a few waves on small problems, at most 512 columns
static int hemv_cols(int64_t n) {
  const int64_t row_blocks = (n + HEMV_ROWS - 1) / HEMV_ROWS;
  const int64_t want = std::max<int64_t>(1, 152 * 8 / row_blocks);
  const int64_t c = ((n + want - 1) / want + 63) / 64 * 64;
  return (int)std::min<int64_t>(512, std::max<int64_t>(64, c));
}

// Bound of nchunk * n over all sizes up to n (the hemv partial sums of one run): the wanted blocks' rows, or n rows
// per 512 columns.
static int64_t hemv_part_rows(int64_t n) { return std::max<int64_t>(152 * 8 * HEMV_ROWS, n * (n / 512 + 1)); }

int64_t lanczos_work_elems(int64_t n, int runs, int steps, bool cplx) {
  // basis | W | hemv partial sums | vector fragments | row maxima | exponents
  const int64_t scal = cplx ? 16 : 8;
  const int64_t extra = (frag_halves(n, cplx, runs) * 2 + n * 4 + 512 + scal - 1) / scal;
  return (int64_t)runs * steps * n + runs * n + runs * hemv_part_rows(n) + extra + 16;
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
    write_frag<T>(X, (n + 15) / 16, i, run, to_fixed(s::re(v), es), NC == 2 ? to_fixed(s::im(v), es) : 0ll);
  }
}

// ---------------------------------------------------------------- Ritz values
// Implicit QL with Wilkinson shifts on the run's tridiagonal T (steps <= 64), one warp per run: eigenvalues, and the
// first row of the eigenvectors' matrix, which is all the density of states needs (Golub and Welsch 1969).  About
// 1.7 QL sweeps per eigenvalue of at most `steps` rotations, a serial chain in lane 0; the search for a negligible
// off-diagonal before each sweep is one step of the whole warp.  Output theta ascending and tau2 = squared first
// components.  (A two-sided Jacobi over the block took 5.6 ms for 25 steps.)
__global__ void tridiag_ql_kernel(int steps, const double* alpha, const double* beta, double* theta, double* tau2,
                                  int* status) {
  const int r = blockIdx.x, k = steps, lane = threadIdx.x;
  __shared__ double d[LZ_MAXS], e[LZ_MAXS], z[LZ_MAXS];
  // scaled by a power of two to norm about 1, so that squares neither overflow nor vanish
  double m = 0.0;
  for (int i = lane; i < k; i += 32) {
    d[i] = alpha[r * LZ_MAXS + i];
    e[i] = i + 1 < k ? beta[r * LZ_MAXS + i] : 0.0;
    z[i] = i == 0 ? 1.0 : 0.0;
    m = fmax(m, fmax(fabs(d[i]), fabs(e[i])));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  int sc = 0;
  if (m > 0.0 && isfinite(m)) frexp(m, &sc);
  for (int i = lane; i < k; i += 32) {
    d[i] = ldexp(d[i], -sc);
    e[i] = ldexp(e[i], -sc);
  }
  __syncwarp();
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
        if (lane == 0) atomicMax(status, 1);
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
  // ascending (stable) order
  for (int i = lane; i < k; i += 32) {
    const double wi = d[i];
    int rank = 0;
    for (int q = 0; q < k; ++q) rank += (d[q] < wi) || (d[q] == wi && q < i);
    theta[r * LZ_MAXS + rank] = ldexp(wi, sc);
    tau2[r * LZ_MAXS + rank] = z[i] * z[i];
  }
}

// b_sup, mu_1, mu_ne (DoS quantile), theta_max: the pooled Ritz values ranked in parallel, their weights added in
// ascending order by one thread.
__global__ void lanczos_bounds_kernel(int runs, int steps, int64_t n, int ne, const double* theta, const double* tau2,
                                      const double* beta, double* out4) {
  __shared__ double th[LZ_MAXR * LZ_MAXS], so[LZ_MAXR * LZ_MAXS], wt[LZ_MAXR * LZ_MAXS];
  const int total = runs * steps;
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    th[i] = theta[(i / steps) * LZ_MAXS + i % steps];
    so[i] = wt[i] = 0.0;
  }
  __syncthreads();
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
  out4[0] = b_sup;
  out4[1] = mu1;
  out4[2] = mu_ne;
  out4[3] = tmax;
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

template <typename T>
void lanczos(cudaStream_t st, const T* A, int64_t n, int64_t lda, int ne, const T* L0, int runs, int steps,
             double* out4, T* work, int64_t work_elems, double* dwork) {
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
  row_max_kernel<T><<<dim3(ceil_div(n, 128), ceil_div(n, ROWMAX_COLS)), 128, 0, st>>>(n, A, lda, rmax);
  CHASE_CHECK_LAUNCH();

  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  const int ctas = step_ctas<T>(n);
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ctas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.gridDim = dim3(ctas, runs, 1);
  cfg.blockDim = dim3(STEP_THREADS, 1, 1);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  auto step = [&](int j) {
    CHASE_CUDA(cudaLaunchKernelEx(&cfg, lanczos_step_kernel<T>, n, runs, steps, j, nchunk, (const T*)part, L0, Vb, W,
                                  alpha, beta, X, xe));
    CHASE_CHECK_LAUNCH();
  };
  step(-1);
  const dim3 g1(ceil_div(n, HEMV_ROWS), nchunk, ceil_div(runs, Frag<T>::RUNS));
  for (int j = 0; j < steps; ++j) {
    hemv_mma_kernel<T><<<g1, 2 * HEMV_ROWS, 0, st>>>(n, A, lda, rmax, X, xe, cols, runs, part);
    CHASE_CHECK_LAUNCH();
    step(j);
  }
  tridiag_ql_kernel<<<runs, 32, 0, st>>>(steps, alpha, beta, theta, tau2, status);
  CHASE_CHECK_LAUNCH();
  lanczos_bounds_kernel<<<1, 256, 0, st>>>(runs, steps, n, ne, theta, tau2, beta, out4);
  CHASE_CHECK_LAUNCH();
}

template void lanczos<double>(cudaStream_t, const double*, int64_t, int64_t, int, const double*, int, int, double*,
                              double*, int64_t, double*);
template void lanczos<double2>(cudaStream_t, const double2*, int64_t, int64_t, int, const double2*, int, int, double*,
                               double2*, int64_t, double*);

}  // namespace chase
