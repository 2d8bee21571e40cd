// Adjoint of the partial eigendecomposition (lambda, V) = lowest eigenpairs of a real
// symmetric A (the differentiation form beside Algorithm 1; the paper has no
// backward).  With S the set of converged (locked) pairs, gbar and Vbar padded by
// zeros outside the returned nev pairs:
//   Abar = V_S (diag(gbar_S) + F o (V_S^T Vbar_S)) V_S^T + X V^T,
//   F_ij = 1/(lambda_j - lambda_i) (i != j, 0 on the diagonal),
// and column x_j of X solves P (A - lambda_j I) P x_j = -P vbar_j on range(P),
// P = I - V_S V_S^T, by MINRES (Paige & Saunders), all nev columns at once: one
// A-times-block product per iteration (split tensor-core products) and one block
// per column for the recurrences.  Abar is symmetrised at the end.
#include "common.cuh"
#include "kernels.h"

namespace chase {

// inner(i, j) for i < l, j < nev: (i == j ? gl_j : 0) + F_ij M_ij
__global__ void adj_inner_kernel(int l, int nev, const double* lam, const double* M, int64_t ldm, const double* gl,
                                 double* inner, int64_t ldi) {
  int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i >= l || j >= nev) return;
  double v = 0.0;
  if (i == j) {
    v = gl ? gl[j] : 0.0;
  } else if (M) {
    v = M[i + (int64_t)j * ldm] / (lam[j] - lam[i]);
  }
  inner[i + (int64_t)j * ldi] = v;
}

struct MinresState {
  double beta1, beta, ib, kr, dbar, epsln, phibar, cs, sn;  // ib = 1 / beta; kr = beta / the one before it (0: none)
  int done, itn;
};

// y = b (stored in R1 and R2), v = b / ||b||, scalars; one block per column
__global__ void minres_init_kernel(int64_t n, const double* B, int64_t ldb, double* R1, double* R2, double* Vv,
                                   double* X, double* W, double* W2, MinresState* st, double tol) {
  int j = blockIdx.x;
  const double* b = B + (int64_t)j * ldb;
  double acc = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) acc += b[i] * b[i];
  __shared__ double red[32];
  __shared__ double nb;
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    nb = sqrt(s);
    MinresState m;
    m.beta1 = nb;
    m.beta = nb;
    m.ib = nb > 0.0 ? 1.0 / nb : 0.0;
    m.kr = 0.0;
    m.dbar = 0.0;
    m.epsln = 0.0;
    m.phibar = nb;
    m.cs = -1.0;
    m.sn = 0.0;
    m.done = (nb == 0.0) ? 1 : 0;
    m.itn = 0;
    st[j] = m;
  }
  __syncthreads();
  const double inv = nb > 0.0 ? 1.0 / nb : 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    const int64_t o = i + (int64_t)j * n;
    R1[o] = b[i];
    R2[o] = b[i];
    Vv[o] = b[i] * inv;
    X[o] = 0.0;
    W[o] = 0.0;
    W2[o] = 0.0;
  }
}

// One MINRES iteration after Y = P (A - lambda_j I) v, a cluster of CTAs per column: three dependent passes with two
// sums over the column between them.  FP64 issue and latency bound it (a warp's FP64 instruction takes 16 cycles of an
// SM, and about 100 to its result), so the scalar recurrence is left to one warp per CTA, a CTA's sum goes through
// shared memory to that warp, reciprocals come from fast_rsqrt, and a thread's entries stay in registers (n <= 4096).
// n = 4096, 64 columns: 12 us; 27 with one block of 1024 threads per column.
// In place: R1 <- new r2 (= y), Wold1 <- new w, Vv <- next v; the host rotates buffer roles.
constexpr int MR_CTAS = 4, MR_THREADS = 256, MR_KEEP = 4;  // entries per thread in registers
__global__ void __launch_bounds__(MR_THREADS) __cluster_dims__(MR_CTAS, 1, 1)
    minres_update_kernel(int64_t n, const double* __restrict__ Y, double* R1, const double* __restrict__ R2, double* Vv,
                         double* Wn /* in: w1, out: new w */, const double* __restrict__ Wc /* w */, double* X,
                         MinresState* st, double tol) {
  constexpr int NW = MR_THREADS / 32;
  __shared__ double red[MR_THREADS], part[2][MR_CTAS], sh[5];
  const int j = blockIdx.y, rank = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  grid_dependency_wait();
  const MinresState m0 = st[j];
  const int64_t off = (int64_t)j * n;
  const int64_t per = (n + MR_CTAS - 1) / MR_CTAS, i0 = rank * per, i1 = i0 + per < n ? i0 + per : n;
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");  // every CTA of the cluster runs
  if (m0.done) return;  // the whole cluster
  // the column's sum, in the first warp
  auto cluster_sum = [&](double v, int set) {
    red[tid] = v;
    __syncthreads();
    if (tid < 32) {
      v = red[lane];
#pragma unroll
      for (int w = 1; w < NW; ++w) v += red[lane + 32 * w];
      v = warp_sum(v);
      if (lane < MR_CTAS) {
        uint32_t to;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                     : "=r"(to)
                     : "r"((uint32_t)__cvta_generic_to_shared(&part[set][rank])), "r"(lane));
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(to), "d"(v) : "memory");
      }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    double t = 0.0;
    if (tid < 32)
#pragma unroll
      for (int c = 0; c < MR_CTAS; ++c) t += part[set][c];
    return t;
  };
  const double kr1 = m0.kr;  // y -= (beta/oldb) r1 from the 2nd iteration on
  // pass 1: alfa = v . (Y - kr1 r1)
  double v[MR_KEEP], y[MR_KEEP];
  double d = 0.0;
#pragma unroll
  for (int k = 0; k < MR_KEEP; ++k) {
    const int64_t i = i0 + tid + k * MR_THREADS;
    const bool in = i < i1;
    v[k] = in ? Vv[off + i] : 0.0;
    y[k] = in ? Y[off + i] - kr1 * R1[off + i] : 0.0;
    d += v[k] * y[k];
  }
  for (int64_t i = i0 + tid + MR_KEEP * MR_THREADS; i < i1; i += MR_THREADS) d += Vv[off + i] * (Y[off + i] - kr1 * R1[off + i]);
  const double alfa = cluster_sum(d, 0);
  if (tid == 0) sh[0] = alfa * m0.ib;
  __syncthreads();
  const double ka = sh[0];
  // pass 2: y = Y - kr1 r1 - ka r2 (written over r1), ||y||^2
  double q = 0.0;
#pragma unroll
  for (int k = 0; k < MR_KEEP; ++k) {
    const int64_t i = i0 + tid + k * MR_THREADS;
    if (i < i1) y[k] -= ka * R2[off + i];
    q += y[k] * y[k];
  }
  for (int64_t i = i0 + tid + MR_KEEP * MR_THREADS; i < i1; i += MR_THREADS) {
    const double t = Y[off + i] - kr1 * R1[off + i] - ka * R2[off + i];
    R1[off + i] = t;
    q += t * t;
  }
  const double yy = cluster_sum(q, 1);
  if (tid < 32) {
    MinresState m = m0;
    const double binv = yy > 0.0 ? fast_rsqrt(yy) : 0.0;
    m.beta = yy * binv;
    m.ib = binv;
    const double delta = m.cs * m.dbar + m.sn * alfa;
    const double gbar = m.sn * m.dbar - m.cs * alfa;
    m.epsln = m.sn * m.beta;
    m.dbar = -m.cs * m.beta;
    const double g2 = fma(gbar, gbar, yy);
    double ginv;
    if (g2 > 1e-280 && g2 < 1e280) ginv = fast_rsqrt(g2);
    else ginv = 1.0 / fmax(hypot(gbar, m.beta), 1e-300);
    m.cs = gbar * ginv;
    m.sn = m.beta * ginv;
    const double phi = m.cs * m.phibar;
    if (tid == 0) {
      sh[1] = m0.epsln;
      sh[2] = delta;
      sh[3] = ginv;
      sh[4] = phi;
      sh[0] = binv;
      if (rank == 0) {  // every CTA has read the old state before the sums met
        m.phibar = m.sn * m.phibar;
        m.kr = m.beta * m0.ib;
        m.itn += 1;
        if (m.phibar <= tol * m.beta1 || m.beta == 0.0) m.done = 1;
        st[j] = m;
      }
    }
  }
  __syncthreads();
  const double oldeps = sh[1], delta = sh[2], ginv = sh[3], phi = sh[4], binv = sh[0];
  // pass 3: w = (v - oldeps w1 - delta w2)/gamma over w1; x += phi w; v <- y / beta
#pragma unroll
  for (int k = 0; k < MR_KEEP; ++k) {
    const int64_t i = i0 + tid + k * MR_THREADS;
    if (i < i1) {
      const double w = (v[k] - oldeps * Wn[off + i] - delta * Wc[off + i]) * ginv;
      Wn[off + i] = w;
      X[off + i] += phi * w;
      R1[off + i] = y[k];
      Vv[off + i] = y[k] * binv;
    }
  }
  for (int64_t i = i0 + tid + MR_KEEP * MR_THREADS; i < i1; i += MR_THREADS) {
    const double w = (Vv[off + i] - oldeps * Wn[off + i] - delta * Wc[off + i]) * ginv;
    Wn[off + i] = w;
    X[off + i] += phi * w;
    Vv[off + i] = R1[off + i] * binv;
  }
}

__global__ void count_done_kernel(int nev, const MinresState* st, int* out) {
  grid_dependency_wait();
  int c = 0;
  for (int j = threadIdx.x; j < nev; j += 32) c += st[j].done;
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (threadIdx.x == 0) *out = c;
}

__global__ void add_kernel(int64_t count, double* a, const double* b) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) a[i] += b[i];
}

void adj_inner(cudaStream_t st, int l, int nev, const double* lam, const double* M, int64_t ldm, const double* gl,
               double* inner, int64_t ldi) {
  adj_inner_kernel<<<dim3(ceil_div(l, 128), nev), 128, 0, st>>>(l, nev, lam, M, ldm, gl, inner, ldi);
  CHASE_CHECK_LAUNCH();
}

void minres_init(cudaStream_t st, int64_t n, int nev, const double* B, int64_t ldb, double* R1, double* R2,
                 double* Vv, double* X, double* W, double* W2, void* state, double tol) {
  minres_init_kernel<<<nev, 256, 0, st>>>(n, B, ldb, R1, R2, Vv, X, W, W2, (MinresState*)state, tol);
  CHASE_CHECK_LAUNCH();
}

void minres_update(cudaStream_t st, int64_t n, int nev, const double* Y, double* R1, const double* R2, double* Vv,
                   double* Wn, const double* Wc, double* X, void* state, double tol) {
  launch_pdl(minres_update_kernel, dim3(MR_CTAS, nev), MR_THREADS, 0, st, n, Y, R1, R2, Vv, Wn, Wc, X, (MinresState*)state, tol);
  CHASE_CHECK_LAUNCH();
}

void minres_count_done(cudaStream_t st, int nev, const void* state, int* out) {
  launch_pdl(count_done_kernel, 1, 32, 0, st, nev, (const MinresState*)state, out);
  CHASE_CHECK_LAUNCH();
}

void add_inplace(cudaStream_t st, int64_t count, double* a, const double* b) {
  add_kernel<<<ceil_div(count, 256), 256, 0, st>>>(count, a, b);
  CHASE_CHECK_LAUNCH();
}

size_t minres_state_bytes(int nev) { return (size_t)nev * sizeof(MinresState); }

}  // namespace chase
