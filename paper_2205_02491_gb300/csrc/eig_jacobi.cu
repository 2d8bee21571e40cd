// Dense Hermitian eigensolver of the Rayleigh-Ritz quotient (Algorithm 1,
// line 6) on the device: parallel cyclic two-sided Jacobi in FP64.
//
// Ordering: round-robin tournament on kp = k rounded up to even indices; each
// of the kp-1 rounds of a sweep rotates kp/2 disjoint pairs at once.  A round
// is two launches: rotation parameters for every pair (from the 2x2 blocks of
// the current G), then an in-place update of G (2x2 blocks of J^H G J) and of
// Z (Z J).  For each pair the 2x2 block [[a, g], [conj g, b]] is made real by
// the phase D = diag(1, conj(g)/|g|) and zeroed by the real rotation with
// t = sign(z)/(|z| + sqrt(1+z^2)), z = (b-a)/(2|g|).
#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "kernels.h"

namespace chase {

template <typename T> struct Rot {
  int partner;  // index paired with this one in the current round (-1: none)
  T self;       // J[x][x]
  T other;      // J[partner][x]
};

__device__ inline void round_pair(int r, int idx, int kp, int& a, int& b) {
  int m = kp - 1;
  if (idx == 0) {
    a = r;
    b = kp - 1;
  } else {
    a = (r + idx) % m;
    b = (r - idx + m) % m;
  }
}

// rotation parameters of pair idx of round r.  The device functions take plain (not __restrict__)
// pointers: inside the persistent sweep kernel G and the rotations are written by other blocks
// between barriers, so their loads must not go through the non-coherent read-only path.
template <typename T>
__device__ __forceinline__ void jacobi_params(int k, int kp, int r, int idx, const T* G, int64_t ldg, Rot<T>* rot) {
  using s = S<T>;
  int a, b;
  round_pair(r, idx, kp, a, b);
  int p = min(a, b), q = max(a, b);
  if (q >= k) {  // dummy index for odd k
    if (p < k) rot[p] = Rot<T>{-1, s::one(), s::zero()};
    return;
  }
  T g = G[p + (int64_t)q * ldg];
  double ag = magnitude(g);
  if (!(ag > 1e-300)) {
    rot[p] = Rot<T>{q, s::one(), s::zero()};
    rot[q] = Rot<T>{p, s::one(), s::zero()};
    return;
  }
  double ap = s::re(G[p + (int64_t)p * ldg]), bq = s::re(G[q + (int64_t)q * ldg]);
  double z = (bq - ap) / (2.0 * ag);
  double t = (z >= 0.0 ? 1.0 : -1.0) / (fabs(z) + sqrt(1.0 + z * z));
  double c = 1.0 / sqrt(1.0 + t * t);
  double sn = t * c;
  T ph = s::scale(s::conj(g), 1.0 / ag);  // conj(g)/|g|
  // J = [[c, sn], [-sn*ph, c*ph]] on columns (p, q)
  rot[p] = Rot<T>{q, s::make(c, 0.0), s::scale(ph, -sn)};  // J[p][p], J[q][p]
  rot[q] = Rot<T>{p, s::scale(ph, c), s::make(sn, 0.0)};   // J[q][q], J[p][q]
}

template <typename T>
__global__ void jacobi_params_kernel(int k, int kp, int r, const T* __restrict__ G, int64_t ldg, Rot<T>* rot) {
  int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= kp / 2) return;
  jacobi_params<T>(k, kp, r, idx, G, ldg, rot);
}

// G <- J^H G J, one thread per (row pair, column pair) 2x2 block (in place).  Split into a load
// and a compute/store half so that the persistent sweep can keep several blocks' loads in flight.
template <typename T> struct GItem {
  int rows[2], cols[2];
  bool diag;  // i1 == i2: the rotated pair's own 2x2 block
  T in[2][2], js[2], jo[2], ks[2], ko[2];
};

template <typename T>
__device__ __forceinline__ void g_load(int k, int kp, int r, int i1, int i2, const T* G, int64_t ldg,
                                       const Rot<T>* rot, GItem<T>& it) {
  using s = S<T>;
  round_pair(r, i1, kp, it.rows[0], it.rows[1]);
  round_pair(r, i2, kp, it.cols[0], it.cols[1]);
  it.diag = i1 == i2;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v)
      it.in[u][v] = (it.rows[u] < k && it.cols[v] < k) ? G[it.rows[u] + (int64_t)it.cols[v] * ldg] : s::zero();
  // coefficients: J[x][x] and J[partner(x)][x]
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (it.rows[u] < k) {
      Rot<T> rr = rot[it.rows[u]];
      it.js[u] = rr.self;
      it.jo[u] = rr.partner >= 0 ? rr.other : s::zero();
    } else {
      it.js[u] = s::one();
      it.jo[u] = s::zero();
    }
    if (it.cols[u] < k) {
      Rot<T> rc = rot[it.cols[u]];
      it.ks[u] = rc.self;
      it.ko[u] = rc.partner >= 0 ? rc.other : s::zero();
    } else {
      it.ks[u] = s::one();
      it.ko[u] = s::zero();
    }
  }
}

template <typename T>
__device__ __forceinline__ void g_store(int k, T* G, int64_t ldg, const GItem<T>& it) {
  using s = S<T>;
  // column update: C[u][v] = in[u][v] J[v][v] + in[u][v'] J[v'][v]
  T cu[2][2];
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) cu[u][v] = s::add(s::mul(it.in[u][v], it.ks[v]), s::mul(it.in[u][1 - v], it.ko[v]));
  // row update: out[u][v] = conj(J[u][u]) C[u][v] + conj(J[u'][u]) C[u'][v]
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      if (it.rows[u] >= k || it.cols[v] >= k) continue;
      T o = s::add(s::mul(s::conj(it.js[u]), cu[u][v]), s::mul(s::conj(it.jo[u]), cu[1 - u][v]));
      if (it.rows[u] == it.cols[v]) o = s::make(s::re(o), 0.0);
      if (it.diag && u != v) o = s::zero();  // the rotated pair's off-diagonal entry
      G[it.rows[u] + (int64_t)it.cols[v] * ldg] = o;
    }
}

template <typename T>
__device__ __forceinline__ void jacobi_apply_g(int k, int kp, int r, int i1, int i2, T* G, int64_t ldg,
                                               const Rot<T>* rot) {
  GItem<T> it;
  g_load<T>(k, kp, r, i1, i2, G, ldg, rot, it);
  g_store<T>(k, G, ldg, it);
}

template <typename T>
__global__ void jacobi_apply_g_kernel(int k, int kp, int r, T* G, int64_t ldg, const Rot<T>* __restrict__ rot) {
  int i1 = blockIdx.x * blockDim.x + threadIdx.x;  // row pair index
  int i2 = blockIdx.y * blockDim.y + threadIdx.y;  // column pair index
  int half = kp / 2;
  if (i1 >= half || i2 >= half) return;
  jacobi_apply_g<T>(k, kp, r, i1, i2, G, ldg, rot);
}

// Z <- Z J (rows i, column pairs), in place; load / compute-store halves as for G.
template <typename T> struct ZItem {
  int a, b;
  T za, zb, as, ao, bs, bo;
};

template <typename T>
__device__ __forceinline__ bool z_load(int k, int kp, int r, int i, int pi, const T* Z, int64_t ldz,
                                       const Rot<T>* rot, ZItem<T>& it) {
  round_pair(r, pi, kp, it.a, it.b);
  if (it.a >= k || it.b >= k) return false;
  const Rot<T> ra = rot[it.a], rb = rot[it.b];
  it.as = ra.self;
  it.ao = ra.other;
  it.bs = rb.self;
  it.bo = rb.other;
  it.za = Z[i + (int64_t)it.a * ldz];
  it.zb = Z[i + (int64_t)it.b * ldz];
  return true;
}

template <typename T> __device__ __forceinline__ void z_store(int i, T* Z, int64_t ldz, const ZItem<T>& it) {
  using s = S<T>;
  Z[i + (int64_t)it.a * ldz] = s::add(s::mul(it.za, it.as), s::mul(it.zb, it.ao));
  Z[i + (int64_t)it.b * ldz] = s::add(s::mul(it.zb, it.bs), s::mul(it.za, it.bo));
}

template <typename T>
__device__ __forceinline__ void jacobi_apply_z(int k, int kp, int r, int i, int pi, T* Z, int64_t ldz,
                                               const Rot<T>* rot) {
  ZItem<T> it;
  if (z_load<T>(k, kp, r, i, pi, Z, ldz, rot, it)) z_store<T>(i, Z, ldz, it);
}

template <typename T>
__global__ void jacobi_apply_z_kernel(int k, int kp, int r, T* Z, int64_t ldz, const Rot<T>* __restrict__ rot) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int pi = blockIdx.y;
  if (i >= k) return;
  jacobi_apply_z<T>(k, kp, r, i, pi, Z, ldz, rot);
}

template <typename T> __global__ void set_identity_kernel(int k, T* Z, int64_t ldz) {
  int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i < k) Z[i + (int64_t)j * ldz] = (i == j) ? S<T>::one() : S<T>::zero();
}

// off^2 and fro^2 of G: per-column partials then an ordered sum (deterministic)
template <typename T> __global__ void offdiag_partial_kernel(int k, const T* __restrict__ G, int64_t ldg, double* part) {
  using s = S<T>;
  int j = blockIdx.x;
  double off = 0.0, tot = 0.0;
  for (int i = threadIdx.x; i < k; i += blockDim.x) {
    double v = s::abs2(G[i + (int64_t)j * ldg]);
    tot += v;
    if (i != j) off += v;
  }
  __shared__ double r1[32], r2[32];
  off = warp_sum(off);
  tot = warp_sum(tot);
  if ((threadIdx.x & 31) == 0) {
    r1[threadIdx.x >> 5] = off;
    r2[threadIdx.x >> 5] = tot;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    double a = threadIdx.x < (blockDim.x >> 5) ? r1[threadIdx.x] : 0.0;
    double b = threadIdx.x < (blockDim.x >> 5) ? r2[threadIdx.x] : 0.0;
    a = warp_sum(a);
    b = warp_sum(b);
    if (threadIdx.x == 0) {
      part[2 * j] = a;
      part[2 * j + 1] = b;
    }
  }
}

__global__ void offdiag_sum_kernel(int k, const double* part, double* out) {
  double a = 0.0, b = 0.0;
  for (int j = threadIdx.x; j < k; j += 32) {
    a += part[2 * j];
    b += part[2 * j + 1];
  }
  a = warp_sum(a);
  b = warp_sum(b);
  if (threadIdx.x == 0) {
    out[0] = a;
    out[1] = b;
  }
}

// eigenvalues from the diagonal, ascending rank (stable), permutation
template <typename T>
__global__ void diag_rank_kernel(int k, const T* __restrict__ G, int64_t ldg, double* w, int* perm) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= k) return;
  double wi = S<T>::re(G[i + (int64_t)i * ldg]);
  int rank = 0;
  for (int j = 0; j < k; ++j) {
    double wj = S<T>::re(G[j + (int64_t)j * ldg]);
    rank += (wj < wi) || (wj == wi && j < i);
  }
  w[rank] = wi;
  perm[rank] = i;
}

template <typename T>
int heev_jacobi(cudaStream_t st, int k, T* G, int64_t ldg, double* w, T* Z, int64_t ldz, T* work, int64_t work_elems,
                double* dwork, int* iwork, double tol, int max_sweeps) {
  // work: k*k scalars for the unsorted Z plus Rot array; dwork: 2k+2 doubles; iwork: k ints
  CHASE_REQUIRE(work_elems >= (int64_t)k * k + 3 * (int64_t)k + 8, 2, "heev_jacobi: workspace too small");
  if (k <= 0) return 0;
  T* Zu = work;
  Rot<T>* rot = reinterpret_cast<Rot<T>*>(work + (int64_t)k * k);
  int kp = k + (k & 1);
  set_identity_kernel<T><<<dim3(ceil_div(k, 256), k), 256, 0, st>>>(k, Zu, k);
  CHASE_CHECK_LAUNCH();
  double* part = dwork + 2;
  double hstat[2];
  int sweeps = 0;
  bool done = false;
  for (; sweeps <= max_sweeps; ++sweeps) {
    offdiag_partial_kernel<T><<<k, 128, 0, st>>>(k, G, ldg, part);
    CHASE_CHECK_LAUNCH();
    offdiag_sum_kernel<<<1, 32, 0, st>>>(k, part, dwork);
    CHASE_CHECK_LAUNCH();
    CHASE_CUDA(cudaMemcpyAsync(hstat, dwork, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
    CHASE_CUDA(cudaStreamSynchronize(st));
    CHASE_REQUIRE(isfinite(hstat[0]) && isfinite(hstat[1]), 5, "heev_jacobi: non-finite matrix");
    if (sqrt(hstat[0]) <= tol * sqrt(hstat[1]) || k == 1) {
      done = true;
      break;
    }
    if (sweeps == max_sweeps) break;
    int half = kp / 2;
    dim3 gblk(16, 16), ggrid(ceil_div(half, 16), ceil_div(half, 16));
    dim3 zgrid(ceil_div(k, 128), half);
    for (int r = 0; r < kp - 1; ++r) {
      jacobi_params_kernel<T><<<ceil_div(half, 128), 128, 0, st>>>(k, kp, r, G, ldg, rot);
      CHASE_CHECK_LAUNCH();
      jacobi_apply_g_kernel<T><<<ggrid, gblk, 0, st>>>(k, kp, r, G, ldg, rot);
      CHASE_CHECK_LAUNCH();
      jacobi_apply_z_kernel<T><<<zgrid, 128, 0, st>>>(k, kp, r, Zu, k, rot);
      CHASE_CHECK_LAUNCH();
    }
  }
  CHASE_REQUIRE(done, 8, "heev_jacobi: sweep cap reached without convergence");
  diag_rank_kernel<T><<<ceil_div(k, 128), 128, 0, st>>>(k, G, ldg, w, iwork);
  CHASE_CHECK_LAUNCH();
  permute_cols<T>(st, k, k, Zu, k, Z, ldz, iwork);
  return sweeps;
}

// ---------------------------------------------------------------- FP32 rotations
// realness of a diagonal entry without a round trip through double
__device__ __forceinline__ void bj_real(float& a) {}
__device__ __forceinline__ void bj_real(float2& a) { a.y = 0.0f; }

// Rotation that zeroes g in [[a, g], [conj g, b]]: phase ph = conj(g)/|g|, then c, sn.  All in FP32 (GB300's FP64 runs
// at 1/64 of it, and this is the serial part of a round), but each pair is brought back to unit length by one Newton
// step on a residual computed without cancellation, so c^2 + sn^2 and |ph| are off by their own rounding only, as if
// rounded from FP64 (plain FP32 parameters raise the pass's rounding floor above what the FP64 corrections that follow
// can absorb for close eigenvalues).
template <typename F> struct Givens {
  float c, sn;
  F ph;
};
__device__ __forceinline__ float phase_of(float g, float& ag) {
  ag = fabsf(g);
  return g < 0.0f ? -1.0f : 1.0f;
}
__device__ __forceinline__ float2 phase_of(float2 g, float& ag) {
  const float x = fabsf(g.x), y = fabsf(g.y), m = fmaxf(x, y), r = __fdividef(fminf(x, y), m);
  ag = m * sqrtf(fmaf(r, r, 1.0f));
  const float inv = 1.0f / ag;
  float2 ph = make_float2(g.x * inv, -g.y * inv);
  const float d = 0.5f * fmaf(-ph.y, ph.y, fmaf(-ph.x, ph.x, 1.0f));
  return make_float2(fmaf(ph.x, d, ph.x), fmaf(ph.y, d, ph.y));
}
__device__ __forceinline__ float largest(float g) { return fabsf(g); }
__device__ __forceinline__ float largest(float2 g) { return fmaxf(fabsf(g.x), fabsf(g.y)); }
__device__ __forceinline__ float real_of(float g) { return g; }
__device__ __forceinline__ float real_of(float2 g) { return g.x; }

template <typename F> __device__ __forceinline__ Givens<F> givens(F a, F b, F g) {
  Givens<F> o;
  o.c = 1.0f;
  o.sn = 0.0f;
  o.ph = S<F>::one();
  if (!(largest(g) > 1e-30f)) return o;
  float ag;
  o.ph = phase_of(g, ag);
  const float z = (real_of(b) - real_of(a)) / (2.0f * ag);
  const float az = fabsf(z);
  // t = sign(z) / (|z| + sqrt(1 + z^2)); from |z| = 1e4 on the square root is |z| to FP32
  const float t = copysignf(1.0f / (az + (az < 1e4f ? sqrtf(fmaf(z, z, 1.0f)) : az)), z);
  const float c = rsqrtf(fmaf(t, t, 1.0f)), sn = t * c;
  const float d = 0.5f * fmaf(-sn, sn, fmaf(-c, c, 1.0f));
  o.c = fmaf(c, d, c);
  o.sn = fmaf(sn, d, sn);
  return o;
}

// (p, q) <- (c p - sn ph q, sn p + c ph q): columns p, q of a row times J = [[c, sn], [-sn ph, c ph]]; rows take conj(ph)
__device__ __forceinline__ void rotate(float& p, float& q, float c, float sn, float ph) {
  const float y = q * ph, x = p;
  p = fmaf(c, x, -sn * y);
  q = fmaf(sn, x, c * y);
}
__device__ __forceinline__ void rotate(float2& p, float2& q, float c, float sn, float2 ph) {
  const float2 y = make_float2(fmaf(q.x, ph.x, -q.y * ph.y), fmaf(q.x, ph.y, q.y * ph.x)), x = p;
  p = make_float2(fmaf(c, x.x, -sn * y.x), fmaf(c, x.y, -sn * y.y));
  q = make_float2(fmaf(sn, x.x, c * y.x), fmaf(sn, x.y, c * y.y));
}

// ---------------------------------------------------------------- persistent sweep
// FP32 first pass of quotients of 65 to 127 columns: one cooperative launch runs all kp-1 rounds of a sweep.  A round is
// one phase and one grid-wide barrier (all blocks are co-resident under a cooperative launch): every item works
// out the rotations it needs from the old G (FP32, a few tens of instructions) and writes the other of two copies, so
// nothing waits for a parameter pass; Z items own their entries.  With a parameter phase in FP64 and two barriers a
// round took 10 us.  Every barrier wait is bounded by a wall-clock limit; on expiry, or when another block has flagged an
// error, the block sets/keeps the error flag and returns.
constexpr int SWEEP_THREADS = 256;  // up to four blocks per SM (measured faster than one 1024-thread block)
// barrier words, each in its own 32-byte sector
constexpr int BAR_COUNT = 0, BAR_ERR = 16, BAR_WORDS = 17;

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// bar[BAR_COUNT]: arrivals since the launch, bar[BAR_ERR]: error flag (both zero at launch); target: the arrivals that
// complete this barrier, (rounds so far) x blocks; wait_ns: wall-clock limit of one wait.  Everyone polls the arrival
// count itself, an arrival is one release operation and a poll one acquire: with a generation word that the last block
// to arrive sets (three more serial trips to L2), a sleep between polls and separate fences a round took 5.6 us, and
// 4.7 without them; with G's and Z's items on different threads 3.9 (96 columns).
__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ bool grid_barrier(unsigned* bar, unsigned target, unsigned long long wait_ns) {
  __shared__ int ok_sh;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* vb = bar;
    int ok = vb[BAR_ERR] == 0u;
    if (ok) {
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&bar[BAR_COUNT]) : "memory");
      unsigned long long t0 = 0;
      while (load_acquire(&bar[BAR_COUNT]) < target) {
        const unsigned long long t = gtimer();
        if (t0 == 0) t0 = t;
        if (vb[BAR_ERR] != 0u) {
          ok = 0;
          break;
        }
        if (t - t0 > wait_ns) {
          atomicOr(&bar[BAR_ERR], 1u);
          ok = 0;
          break;
        }
      }
    }
    ok_sh = ok;
  }
  __syncthreads();
  return ok_sh != 0;
}

template <typename F>
__device__ __forceinline__ Givens<F> pair_rotation(int k, int p, int q, const F* G, int64_t ldg) {
  // the dummy index of an odd k rotates nothing
  if (p >= k || q >= k) return givens<F>(S<F>::zero(), S<F>::zero(), S<F>::zero());
  return givens<F>(G[p + (int64_t)p * ldg], G[q + (int64_t)q * ldg], G[p + (int64_t)q * ldg]);
}

// Starts from Ga; the result of the kp - 1 (odd) rounds is in Gb.  Plain loads: other blocks write between barriers.
template <typename F>
__global__ void __launch_bounds__(SWEEP_THREADS, 4) jacobi_sweep_kernel(int k, int kp, F* Ga, F* Gb, F* Z, unsigned* bar,
                                                                        unsigned long long wait_ns) {
  using s = S<F>;
  const int half = kp / 2;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nthr = gridDim.x * blockDim.x;
  const int ng = half * half, nz = k * half;
  const int64_t ld = k;
  for (int r = 0; r < kp - 1; ++r) {
    const F* Go = (r & 1) ? Gb : Ga;
    F* Gn = (r & 1) ? Ga : Gb;
    // G's items, then Z's: one per thread
    for (int x = tid; x < ng; x += nthr) {
      const int i1 = x % half, i2 = x / half;
      int p1, q1, p2, q2;
      round_pair(r, i1, kp, p1, q1);
      round_pair(r, i2, kp, p2, q2);
      const Givens<F> jr = pair_rotation<F>(k, p1, q1, Go, ld), jc = pair_rotation<F>(k, p2, q2, Go, ld);
      const bool a = p1 < k, b = q1 < k, c = p2 < k, d = q2 < k;
      F tt = a && c ? Go[p1 + p2 * ld] : s::zero(), tb = a && d ? Go[p1 + q2 * ld] : s::zero();
      F bt = b && c ? Go[q1 + p2 * ld] : s::zero(), bb = b && d ? Go[q1 + q2 * ld] : s::zero();
      rotate(tt, tb, jc.c, jc.sn, jc.ph);
      rotate(bt, bb, jc.c, jc.sn, jc.ph);
      rotate(tt, bt, jr.c, jr.sn, s::conj(jr.ph));
      rotate(tb, bb, jr.c, jr.sn, s::conj(jr.ph));
      if (i1 == i2) {
        bj_real(tt);
        bj_real(bb);
        tb = bt = s::zero();
      }
      if (a && c) Gn[p1 + p2 * ld] = tt;
      if (a && d) Gn[p1 + q2 * ld] = tb;
      if (b && c) Gn[q1 + p2 * ld] = bt;
      if (b && d) Gn[q1 + q2 * ld] = bb;
    }
    for (int x = tid < ng ? tid + (ng - tid + nthr - 1) / nthr * nthr - ng : tid - ng; x < nz; x += nthr) {
      const int i = x % k;
      int p, q;
      round_pair(r, x / k, kp, p, q);
      if (p >= k || q >= k) continue;
      const Givens<F> j = pair_rotation<F>(k, p, q, Go, ld);
      F zp = Z[i + p * ld], zq = Z[i + q * ld];
      rotate(zp, zq, j.c, j.sn, j.ph);
      Z[i + p * ld] = zp;
      Z[i + q * ld] = zq;
    }
    if (!grid_barrier(bar, (unsigned)(r + 1) * gridDim.x, wait_ns)) return;
  }
}

// co-resident blocks of SWEEP_THREADS threads for the sweep kernel (0: no cooperative launch)
template <typename F> static int sweep_grid() {
  static const int nb = []() {
    int dev = 0, sms = 0, per = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, jacobi_sweep_kernel<F>, SWEEP_THREADS, 0) != cudaSuccess)
      return 0;
    return sms * std::min(per, 4);
  }();
  return nb;
}

template <typename F>
int heev_sweep(cudaStream_t st, int k, F* G, double* w, F* Z, int64_t ldz, F* work, int64_t work_elems, double* dwork,
               int* iwork, double tol, int max_sweeps) {
  CHASE_REQUIRE(k >= BAR_WORDS && work_elems >= 2 * (int64_t)k * k, 2, "heev_sweep: workspace too small");
  F* Zu = work;
  F* buf[2] = {G, work + (int64_t)k * k};
  const int kp = k + (k & 1);
  set_identity_kernel<F><<<dim3(ceil_div(k, 256), k), 256, 0, st>>>(k, Zu, k);
  CHASE_CHECK_LAUNCH();
  double* part = dwork + 2;
  double hstat[2];
  // grid sized by the work of a round (one item per thread), at most the co-resident maximum: small quotients take
  // few SMs, which leaves room for other streams' kernels.  The barrier words live in iwork (k ints; overwritten by
  // the final ranking only after the sweeps).
  const int items = (kp / 2) * (kp / 2) + k * (kp / 2);
  const int grid = std::min<int>(sweep_grid<F>(), (int)ceil_div(items, SWEEP_THREADS));
  CHASE_REQUIRE(grid > 0, 9, "heev_sweep: no cooperative launch on this device");
  unsigned* bar = reinterpret_cast<unsigned*>(iwork);
  unsigned bar_err = 0;
  int sweeps = 0;
  for (; sweeps <= max_sweeps; ++sweeps) {
    offdiag_partial_kernel<F><<<k, 128, 0, st>>>(k, buf[0], k, part);
    CHASE_CHECK_LAUNCH();
    offdiag_sum_kernel<<<1, 32, 0, st>>>(k, part, dwork);
    CHASE_CHECK_LAUNCH();
    CHASE_CUDA(cudaMemcpyAsync(hstat, dwork, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
    if (sweeps > 0)
      CHASE_CUDA(cudaMemcpyAsync(&bar_err, bar + BAR_ERR, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
    CHASE_CUDA(cudaStreamSynchronize(st));
    CHASE_REQUIRE(bar_err == 0, 8, "heev_sweep: a grid barrier of the sweep kernel hit its wait limit");
    CHASE_REQUIRE(isfinite(hstat[0]) && isfinite(hstat[1]), 5, "heev_sweep: non-finite matrix");
    // the cap is not an error: the FP64 refinement follows
    if (sqrt(hstat[0]) <= tol * sqrt(hstat[1]) || sweeps == max_sweeps) break;
    CHASE_CUDA(cudaMemsetAsync(bar, 0, BAR_WORDS * sizeof(unsigned), st));
    int kk = k, kpp = kp;
    unsigned long long wait_ns = grid_wait_limit_ns();
    void* args[] = {&kk, &kpp, &buf[0], &buf[1], &Zu, &bar, &wait_ns};
    CHASE_CUDA(cudaLaunchCooperativeKernel((const void*)jacobi_sweep_kernel<F>, dim3(grid), dim3(SWEEP_THREADS), args, 0,
                                           st));
    CHASE_CHECK_LAUNCH();
    std::swap(buf[0], buf[1]);
  }
  diag_rank_kernel<F><<<ceil_div(k, 128), 128, 0, st>>>(k, buf[0], k, w, iwork);
  CHASE_CHECK_LAUNCH();
  permute_cols<F>(st, k, k, Zu, k, Z, ldz, iwork);
  return sweeps;
}

// ---------------------------------------------------------------- one-block Jacobi (FP32 first pass, k <= 64)
// The whole solve in one launch of one CTA: G and Z in shared memory by position (the tournament of bj_solve_kernel
// below, M = 32 or 64 indices, zero rows and columns past k), sweeps until the off-diagonal norm is below tol or stops
// falling at FP32's floor.  A launch per round phase and a host check per sweep took about 2 ms for 24 columns.
// out: sweeps used, or -1 for a non-finite matrix.
template <typename F, int M>
__global__ void __launch_bounds__(M * M / 4) jacobi_block_kernel(int k, const F* __restrict__ G, int64_t ldg, float tol,
                                                                  int max_sweeps, double* w, F* Z, int64_t ldz, int* out) {
  using s = S<F>;
  constexpr int H = M / 2, NT = M * M / 4;
  extern __shared__ __align__(16) unsigned char bj_smem[];
  F* Sm = reinterpret_cast<F*>(bj_smem);  // [2][M][M]
  F* Um = Sm + 2 * M * M;                 // [2][M][M]
  __shared__ Givens<F> prm[2][H];
  __shared__ double red_off[NT / 32], red_tot[NT / 32];
  __shared__ float dg[M];
  const int tid = threadIdx.x, i1 = tid / H, i2 = tid % H;
  for (int e = tid; e < M * M; e += NT) {
    const int l = e % M, m = e / M;
    Sm[m * M + l] = (l < k && m < k) ? s::conj(G[l + (int64_t)m * ldg]) : s::zero();
    Um[m * M + l] = (l == m) ? s::one() : s::zero();
  }
  auto next_top = [](int i) { return i == 0 ? 0 : (i == H - 1 ? M - 1 : i + 1); };
  auto next_bot = [](int i) { return i == 0 ? 1 : H + i - 1; };
  const int rt = next_top(i1) * M, rb = next_bot(i1) * M, ct = next_top(i2), cb = next_bot(i2);
  int cur = 0, sweeps = 0;
  double prev = 0.0;
  __syncthreads();
  for (;; ++sweeps) {
    const F* Sc = Sm + cur * M * M;
    double off = 0.0, tot = 0.0;
    for (int e = tid; e < M * M; e += NT) {
      const double v = s::abs2(Sc[e]);
      tot += v;
      if (e % M != e / M) off += v;
    }
    off = warp_sum(off);
    tot = warp_sum(tot);
    if ((tid & 31) == 0) {
      red_off[tid >> 5] = off;
      red_tot[tid >> 5] = tot;
    }
    __syncthreads();
    off = tot = 0.0;
    for (int i = 0; i < NT / 32; ++i) {
      off += red_off[i];
      tot += red_tot[i];
    }
    if (!isfinite(tot)) {
      if (tid == 0) out[0] = -1;
      return;
    }
    // FP32 floor as in heev_block_jacobi
    if (off <= (double)tol * tol * tot || sweeps == max_sweeps || (sweeps >= 2 && off > 0.0625 * prev && off <= 1e-10 * tot))
      break;
    prev = off;
    if (tid < H) prm[0][tid] = givens<F>(Sc[tid * (M + 1)], Sc[(H + tid) * (M + 1)], Sc[tid * M + H + tid]);
    __syncthreads();
    for (int rr = 0; rr < M - 1; ++rr, cur ^= 1) {
      const int pb = rr & 1;
      const F* S0 = Sm + cur * M * M;
      F* S1 = Sm + (cur ^ 1) * M * M;
      const F* U0 = Um + cur * M * M;
      F* U1 = Um + (cur ^ 1) * M * M;
      const Givens<F> pc = prm[pb][i2], pr = prm[pb][i1];
      {
        F tt = S0[i1 * M + i2], tb = S0[i1 * M + H + i2], bt = S0[(H + i1) * M + i2], bb = S0[(H + i1) * M + H + i2];
        rotate(tt, tb, pc.c, pc.sn, pc.ph);
        rotate(bt, bb, pc.c, pc.sn, pc.ph);
        rotate(tt, bt, pr.c, pr.sn, s::conj(pr.ph));
        rotate(tb, bb, pr.c, pr.sn, s::conj(pr.ph));
        if (i1 == i2) {
          bj_real(tt);
          bj_real(bb);
          tb = bt = s::zero();
        }
        S1[rt + ct] = tt;
        S1[rt + cb] = tb;
        S1[rb + ct] = bt;
        S1[rb + cb] = bb;
      }
      __syncthreads();
      if (tid < H && rr + 1 < M - 1)
        prm[pb ^ 1][tid] = givens<F>(S1[tid * (M + 1)], S1[(H + tid) * (M + 1)], S1[tid * M + H + tid]);
      if (tid >= 32) {
        for (int x = tid - 32; x < M * H; x += NT - 32) {
          const int l = x / H, c = x % H;
          const Givens<F> pz = prm[pb][c];
          F ut = U0[l * M + c], ub = U0[l * M + H + c];
          rotate(ut, ub, pz.c, pz.sn, pz.ph);
          U1[l * M + next_top(c)] = ut;
          U1[l * M + next_bot(c)] = ub;
        }
      }
      __syncthreads();
    }
  }
  // ascending (stable) order of the first k diagonal entries
  const F* Sf = Sm + cur * M * M;
  const F* Uf = Um + cur * M * M;
  if (tid < M) dg[tid] = real_of(Sf[tid * (M + 1)]);
  __syncthreads();
  for (int c = tid >> 5; c < k; c += NT / 32) {
    int rank = 0;
    for (int j = 0; j < k; ++j) rank += (dg[j] < dg[c]) || (dg[j] == dg[c] && j < c);
    if ((tid & 31) == 0) w[rank] = dg[c];
    for (int l = tid & 31; l < k; l += 32) Z[l + (int64_t)rank * ldz] = Uf[l * M + c];
  }
  if (tid == 0) out[0] = sweeps;
}

template <typename F>
void heev_block(cudaStream_t st, int k, const F* G, int64_t ldg, double* w, F* Z, int64_t ldz, int* out, float tol,
                int max_sweeps) {
  CHASE_REQUIRE(k >= 1 && k <= 64, 1, "heev_block: 1 <= k <= 64");
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, []() {
    attr = cudaFuncSetAttribute(jacobi_block_kernel<F, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(4 * 64 * 64 * sizeof(F)));
  });
  CHASE_CUDA(attr);
  if (k <= 32)
    jacobi_block_kernel<F, 32><<<1, 256, 4 * 32 * 32 * sizeof(F), st>>>(k, G, ldg, tol, max_sweeps, w, Z, ldz, out);
  else
    jacobi_block_kernel<F, 64><<<1, 1024, 4 * 64 * 64 * sizeof(F), st>>>(k, G, ldg, tol, max_sweeps, w, Z, ldz, out);
  CHASE_CHECK_LAUNCH();
}

// ---------------------------------------------------------------- block Jacobi (FP32 first pass)
// Two-sided block Jacobi: the indices are cut into blocks of BJ_B; a round-robin tournament over the
// blocks pairs them, and each round reduces every pair's 2 BJ_B x 2 BJ_B principal submatrix
// S = G[IJ, IJ] in shared memory (one sweep of parallel cyclic Jacobi, one CTA per pair, accumulating the
// rotations in U), then applies U to the whole matrix: G[:, IJ] <- G[:, IJ] U and Z[:, IJ] <- Z[:, IJ] U,
// then G[IJ, :] <- U^H G[IJ, :].
// A sweep has (blocks - 1) rounds instead of the scalar method's (k - 1), each doing dense
// (k x 64) x (64 x 64) updates, so the round count (and its launch and synchronisation cost) falls by
// the block width while the arithmetic per sweep stays 4 k^3 multiply-adds.
constexpr int BJ_B = 32;          // block width
constexpr int BJ_M = 2 * BJ_B;    // subproblem order
constexpr int BJ_SOLVE_THREADS = 1024;
constexpr int BJ_UPD_THREADS = 256;
constexpr int BJ_TILE = 16;       // rows (columns) of G or Z per update CTA

// global index of local index l of block pair (I, J)
__device__ __forceinline__ int bj_global(int I, int J, int l) {
  return l < BJ_B ? I * BJ_B + l : J * BJ_B + (l - BJ_B);
}

// A block paired with the padding block has nothing to do, except in a sweep's first round, which annihilates the
// entries inside the blocks too (the padding's rows and columns read as zero).
__device__ __forceinline__ bool bj_idle(int I, int J, int nb, int r) {
  return (I >= nb && J >= nb) || (r != 0 && (I >= nb || J >= nb));
}

// One block pair's subproblem.  Pair i of a round is (top i, bottom i): rows and columns of S, and columns of U, are
// stored by position, top i at i and bottom i at 32 + i, and every round writes them to the positions of the next one
// (two buffers), so that addresses are the same in all rounds, lanes touch consecutive words, and a thread's 2 x 2
// block of S is its row pair (warp) by its column pair (lane).
// full: all 63 rounds of the 64 indices' tournament (top 0 fixed, the others move one position around the circle top
// 1 .. 31, bottom 31 .. 0).  Else only the 32 rounds that pair a top with a bottom index (bottoms move by one): within
// the two blocks the entries were annihilated in the sweep's first round, and each cross pair is rotated once a sweep.
// While one warp works out the next round's rotations from the new S, the others apply the current ones to U: a round
// is bound by its shared-memory traffic (S and U read and written once), about 1250 cycles.
template <typename F>
__global__ void __launch_bounds__(BJ_SOLVE_THREADS) bj_solve_kernel(int k, int nbp, int r, const F* G, int64_t ldg,
                                                                     F* Ubuf, int full) {
  grid_dependency_wait();
  using s = S<F>;
  extern __shared__ __align__(16) unsigned char bj_smem[];
  F* Sm = reinterpret_cast<F*>(bj_smem);    // [2][64][64], row-major by position
  F* Um = Sm + 2 * BJ_M * BJ_M;             // [2][64][64]: row l, column by position
  __shared__ Givens<F> prm[2][BJ_B];
  const int nb = (k + BJ_B - 1) / BJ_B;
  int I, J;
  round_pair(r, blockIdx.x, nbp, I, J);
  if (bj_idle(I, J, nb, r)) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int e = tid; e < BJ_M * BJ_M; e += BJ_SOLVE_THREADS) {
    const int l = e % BJ_M, m = e / BJ_M;
    const int gl = bj_global(I, J, l), gm = bj_global(I, J, m);
    // row m, column l: the conjugate of the Hermitian matrix's entry (l, m), so that lanes store consecutive words
    Sm[m * BJ_M + l] = (gl < k && gm < k) ? s::conj(G[gl + (int64_t)gm * ldg]) : s::zero();
    Um[m * BJ_M + l] = (l == m) ? s::one() : s::zero();
  }
  // next position of (top | bottom) index i
  auto next_top = [&](int i) { return !full || i == 0 ? i : (i == BJ_B - 1 ? BJ_M - 1 : i + 1); };
  auto next_bot = [&](int i) { return full ? (i == 0 ? 1 : BJ_B + i - 1) : BJ_B + ((i + BJ_B - 1) & (BJ_B - 1)); };
  const int rt = next_top(warp) * BJ_M, rb = next_bot(warp) * BJ_M, ct = next_top(lane), cb = next_bot(lane);
  const int rounds = full ? BJ_M - 1 : BJ_B;
  __syncthreads();
  if (warp == 0) prm[0][lane] = givens<F>(Sm[lane * BJ_M + lane], Sm[(BJ_B + lane) * (BJ_M + 1)], Sm[lane * BJ_M + BJ_B + lane]);
  __syncthreads();
  for (int rr = 0; rr < rounds; ++rr) {
    const int cur = rr & 1;
    const F* S0 = Sm + cur * BJ_M * BJ_M;
    F* S1 = Sm + (cur ^ 1) * BJ_M * BJ_M;
    const F* U0 = Um + cur * BJ_M * BJ_M;
    F* U1 = Um + (cur ^ 1) * BJ_M * BJ_M;
    const Givens<F> pc = prm[cur][lane], pr = prm[cur][warp];
    {
      F tt = S0[warp * BJ_M + lane], tb = S0[warp * BJ_M + BJ_B + lane];
      F bt = S0[(BJ_B + warp) * BJ_M + lane], bb = S0[(BJ_B + warp) * BJ_M + BJ_B + lane];
      rotate(tt, tb, pc.c, pc.sn, pc.ph);
      rotate(bt, bb, pc.c, pc.sn, pc.ph);
      rotate(tt, bt, pr.c, pr.sn, s::conj(pr.ph));
      rotate(tb, bb, pr.c, pr.sn, s::conj(pr.ph));
      if (warp == lane) {
        bj_real(tt);
        bj_real(bb);
        tb = bt = s::zero();
      }
      S1[rt + ct] = tt;
      S1[rt + cb] = tb;
      S1[rb + ct] = bt;
      S1[rb + cb] = bb;
    }
    __syncthreads();
    if (warp == 0) {
      if (rr + 1 < rounds)
        prm[cur ^ 1][lane] =
            givens<F>(S1[lane * BJ_M + lane], S1[(BJ_B + lane) * (BJ_M + 1)], S1[lane * BJ_M + BJ_B + lane]);
    } else {
      for (int l = warp - 1; l < BJ_M; l += BJ_SOLVE_THREADS / 32 - 1) {
        F ut = U0[l * BJ_M + lane], ub = U0[l * BJ_M + BJ_B + lane];
        rotate(ut, ub, pc.c, pc.sn, pc.ph);
        U1[l * BJ_M + ct] = ut;
        U1[l * BJ_M + cb] = ub;
      }
    }
    __syncthreads();
  }
  // after all rounds every index is back at its position
  const F* Uf = Um + (rounds & 1) * BJ_M * BJ_M;
  F* U = Ubuf + (int64_t)blockIdx.x * BJ_M * BJ_M;  // row-major
  for (int e = tid; e < BJ_M * BJ_M; e += BJ_SOLVE_THREADS) U[e] = Uf[e];
}

// The updates: 64 x 64 times 64 x 16 products, 4 outputs per thread.  Their arithmetic is 2 to 3 us for 437 complex
// columns; what they cost is latency, so tiles are small (several CTAs per SM).  Doubled operands for packed FP32
// multiply-adds and 64 x 64 tiles with 4 x 4 outputs per thread took 20 us a launch, one CTA per SM.
// X[:, IJ] <- X[:, IJ] U for a tile of BJ_TILE rows (X = G for blockIdx.z == 0, Z for 1)
template <typename F>
__global__ void __launch_bounds__(BJ_UPD_THREADS) bj_cols_kernel(int k, int nbp, int r, F* G, int64_t ldg, F* Z,
                                                                  int64_t ldz, const F* __restrict__ Ubuf) {
  grid_dependency_wait();
  using s = S<F>;
  __shared__ __align__(16) F Us[BJ_M][BJ_M];    // U[m][c]
  __shared__ F Xs[BJ_M][BJ_TILE];               // X[row][m] at Xs[m][row]
  const int nb = (k + BJ_B - 1) / BJ_B;
  int I, J;
  round_pair(r, blockIdx.y, nbp, I, J);
  if (bj_idle(I, J, nb, r)) return;
  F* X = blockIdx.z == 0 ? G : Z;
  const int64_t ldx = blockIdx.z == 0 ? ldg : ldz;
  const int tid = threadIdx.x, i = tid % BJ_TILE, q = tid / BJ_TILE;
  const int gi = blockIdx.x * BJ_TILE + i;
  const F* U = Ubuf + (int64_t)blockIdx.y * BJ_M * BJ_M;
#pragma unroll
  for (int e = 0; e < BJ_M * BJ_M / BJ_UPD_THREADS; ++e) (&Us[0][0])[tid + e * BJ_UPD_THREADS] = U[tid + e * BJ_UPD_THREADS];
#pragma unroll
  for (int e = 0; e < BJ_M * BJ_TILE / BJ_UPD_THREADS; ++e) {
    const int l = q + e * (BJ_UPD_THREADS / BJ_TILE), gl = bj_global(I, J, l);
    Xs[l][i] = (gi < k && gl < k) ? X[gi + (int64_t)gl * ldx] : s::zero();
  }
  __syncthreads();
  F acc[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) acc[c] = s::zero();
#pragma unroll 8
  for (int m = 0; m < BJ_M; ++m) {
    const F x = Xs[m][i];
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] = s::fma(x, Us[m][4 * q + c], acc[c]);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int gl = bj_global(I, J, 4 * q + c);
    if (gi < k && gl < k) X[gi + (int64_t)gl * ldx] = acc[c];
  }
}

// G[IJ, :] <- U^H G[IJ, :] for a tile of BJ_TILE columns
template <typename F>
__global__ void __launch_bounds__(BJ_UPD_THREADS) bj_rows_kernel(int k, int nbp, int r, F* G, int64_t ldg,
                                                                  const F* __restrict__ Ubuf) {
  grid_dependency_wait();
  using s = S<F>;
  __shared__ F Us[BJ_M][BJ_M + 1];      // U[m][l]
  __shared__ F Xs[BJ_TILE][BJ_M];       // X[m][column] at Xs[column][m]
  const int nb = (k + BJ_B - 1) / BJ_B;
  int I, J;
  round_pair(r, blockIdx.y, nbp, I, J);
  if (bj_idle(I, J, nb, r)) return;
  const int tid = threadIdx.x, l = tid % BJ_M, q = tid / BJ_M;
  const int c0 = blockIdx.x * BJ_TILE, gl = bj_global(I, J, l);
  const F* U = Ubuf + (int64_t)blockIdx.y * BJ_M * BJ_M;
#pragma unroll
  for (int e = 0; e < BJ_M * BJ_M / BJ_UPD_THREADS; ++e) Us[q + e * (BJ_UPD_THREADS / BJ_M)][l] = U[tid + e * BJ_UPD_THREADS];
#pragma unroll
  for (int e = 0; e < BJ_M * BJ_TILE / BJ_UPD_THREADS; ++e) {
    const int j = q + e * (BJ_UPD_THREADS / BJ_M);
    Xs[j][l] = (gl < k && c0 + j < k) ? G[gl + (int64_t)(c0 + j) * ldg] : s::zero();
  }
  __syncthreads();
  // thread: row l of the pair, columns 4 q .. 4 q + 3; out[l][j] = sum_m conj(U[m][l]) X[m][j]
  F acc[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) acc[j] = s::zero();
#pragma unroll 8
  for (int m = 0; m < BJ_M; ++m) {
    const F u = s::conj(Us[m][l]);
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j] = s::fma(u, Xs[4 * q + j][m], acc[j]);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (gl < k && c0 + 4 * q + j < k) G[gl + (int64_t)(c0 + 4 * q + j) * ldg] = acc[j];
}

template <typename F> static size_t bj_solve_smem_bytes() { return (size_t)4 * BJ_M * BJ_M * sizeof(F); }

int heev_block_workspace(int k) {
  const int nb = (k + BJ_B - 1) / BJ_B;
  const int nbp = nb + (nb & 1);
  return nbp / 2 * BJ_M * BJ_M;
}

template <typename F>
int heev_block_jacobi(cudaStream_t st, int k, F* G, int64_t ldg, double* w, F* Z, int64_t ldz, F* work,
                      int64_t work_elems, double* dwork, int* iwork, double tol, int max_sweeps) {
  const int nb = (k + BJ_B - 1) / BJ_B;
  const int nbp = nb + (nb & 1);
  const int npairs = nbp / 2;
  CHASE_REQUIRE(k >= 1 && work_elems >= (int64_t)k * k + heev_block_workspace(k), 2,
                "heev_block_jacobi: workspace too small");
  F* Zu = work;
  F* Ubuf = work + (int64_t)k * k;
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, []() {
    attr = cudaFuncSetAttribute(bj_solve_kernel<F>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)bj_solve_smem_bytes<F>());
  });
  CHASE_CUDA(attr);
  set_identity_kernel<F><<<dim3(ceil_div(k, 256), k), 256, 0, st>>>(k, Zu, k);
  CHASE_CHECK_LAUNCH();
  double* part = dwork + 2;
  double hstat[2];
  double prev_off = 0.0;
  int sweeps = 0;
  const int tiles = ceil_div(k, BJ_TILE);
  for (; sweeps <= max_sweeps; ++sweeps) {
    offdiag_partial_kernel<F><<<k, 128, 0, st>>>(k, G, ldg, part);
    CHASE_CHECK_LAUNCH();
    offdiag_sum_kernel<<<1, 32, 0, st>>>(k, part, dwork);
    CHASE_CHECK_LAUNCH();
    CHASE_CUDA(cudaMemcpyAsync(hstat, dwork, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
    CHASE_CUDA(cudaStreamSynchronize(st));
    CHASE_REQUIRE(isfinite(hstat[0]) && isfinite(hstat[1]), 5, "heev_block_jacobi: non-finite matrix");
    if (sqrt(hstat[0]) <= tol * sqrt(hstat[1]) || k == 1 || sweeps == max_sweeps) break;
    // FP32 floor: the 64-term updates leave off-diagonal rounding that can exceed tol for large k; once a sweep
    // no longer quarters the off-diagonal norm below 1e-5 relative, the FP64 refinement takes over.  Its
    // first-order corrections converge quadratically in (off-diagonal / gap): 1e-5 keeps that ratio near 0.05
    // for relative gaps of 2e-4 (the Table 2 Geometric spectrum), where three corrections reach FP64 level
    if (sweeps >= 2 && hstat[0] > 0.0625 * prev_off && sqrt(hstat[0]) <= 1e-5 * sqrt(hstat[1])) break;
    prev_off = hstat[0];
    for (int r = 0; r < nbp - 1; ++r) {
      launch_pdl(bj_solve_kernel<F>, npairs, BJ_SOLVE_THREADS, bj_solve_smem_bytes<F>(), st, k, nbp, r, G, ldg, Ubuf, r == 0);
      CHASE_CHECK_LAUNCH();
      launch_pdl(bj_cols_kernel<F>, dim3(tiles, npairs, 2), BJ_UPD_THREADS, 0, st, k, nbp, r, G, ldg, Zu, k,
                                                                                          Ubuf);
      CHASE_CHECK_LAUNCH();
      launch_pdl(bj_rows_kernel<F>, dim3(tiles, npairs), BJ_UPD_THREADS, 0, st, k, nbp, r, G, ldg, Ubuf);
      CHASE_CHECK_LAUNCH();
    }
  }
  diag_rank_kernel<F><<<ceil_div(k, 128), 128, 0, st>>>(k, G, ldg, w, iwork);
  CHASE_CHECK_LAUNCH();
  permute_cols<F>(st, k, k, Zu, k, Z, ldz, iwork);
  return sweeps;
}

template int heev_block_jacobi<float>(cudaStream_t, int, float*, int64_t, double*, float*, int64_t, float*, int64_t,
                                      double*, int*, double, int);
template int heev_block_jacobi<float2>(cudaStream_t, int, float2*, int64_t, double*, float2*, int64_t, float2*,
                                       int64_t, double*, int*, double, int);

template int heev_jacobi<double>(cudaStream_t, int, double*, int64_t, double*, double*, int64_t, double*, int64_t,
                                 double*, int*, double, int);
template int heev_jacobi<double2>(cudaStream_t, int, double2*, int64_t, double*, double2*, int64_t, double2*, int64_t,
                                  double*, int*, double, int);
template int heev_sweep<float>(cudaStream_t, int, float*, double*, float*, int64_t, float*, int64_t, double*, int*, double,
                               int);
template int heev_sweep<float2>(cudaStream_t, int, float2*, double*, float2*, int64_t, float2*, int64_t, double*, int*,
                                double, int);
template void heev_block<float>(cudaStream_t, int, const float*, int64_t, double*, float*, int64_t, int*, float, int);
template void heev_block<float2>(cudaStream_t, int, const float2*, int64_t, double*, float2*, int64_t, int*, float, int);

}  // namespace chase
