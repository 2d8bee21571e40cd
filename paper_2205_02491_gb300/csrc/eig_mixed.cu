// Helpers of the mixed-precision Rayleigh-Ritz eigensolve (Algorithm 1, line 6).
//
// The quotient G is first diagonalised by the parallel Jacobi solver in FP32 (58x
// the FP64 rate on GB300).  Its eigenvectors Z are then refined in FP64-class products (Ogita and Aishima 2018): with
// N = Z^H Z, S = Z^H G Z, R = I - N and l_p = S_pp / N_pp,
//   Z <- Z (I + E),  E_pq = (S_pq + l_q R_pq) / (l_q - l_p),
// converges quadratically.  R's term is what close eigenvalues need: a normalisation Z (I - R / 2) in its place leaves
// 3/8 R^2 in S, which a gap of 1e-5 amplifies (three eigenvalues 1e-5 apart: residuals up to 1e-3).
// Pairs of one cluster take E_pq = R_pq / 2, which only keeps them orthonormal, and an exact FP64 Jacobi on the
// cluster's block of the quotient, one block per cluster.
#include "common.cuh"
#include "kernels.h"

namespace chase {

template <typename A, typename B> __device__ inline B cvt(A a);
template <> __device__ inline float cvt<double, float>(double a) { return (float)a; }
template <> __device__ inline double cvt<float, double>(float a) { return (double)a; }
template <> __device__ inline float2 cvt<double2, float2>(double2 a) { return make_float2((float)a.x, (float)a.y); }
template <> __device__ inline double2 cvt<float2, double2>(float2 a) { return make_double2(a.x, a.y); }

template <typename T, typename F>
__global__ void convert_kernel(int k, const T* in, int64_t ldi, F* out, int64_t ldo) {
  int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i < k) out[i + (int64_t)j * ldo] = cvt<T, F>(in[i + (int64_t)j * ldi]);
}

template <typename T, typename F> void convert_mat(cudaStream_t st, int k, const T* in, int64_t ldi, F* out, int64_t ldo) {
  convert_kernel<T, F><<<dim3(ceil_div(k, 256), k), 256, 0, st>>>(k, in, ldi, out, ldo);
  CHASE_CHECK_LAUNCH();
}

// l_p = S_pp / N_pp; zeroes the word that receives the largest entry of E
template <typename T>
__global__ void quotients_kernel(int k, const T* S_, const T* N, double* lam, unsigned* emax) {
  grid_dependency_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *emax = 0u;
  if (i < k) lam[i] = S<T>::re(S_[i + (int64_t)i * k]) / S<T>::re(N[i + (int64_t)i * k]);
}

template <typename T>
void eig_quotients(cudaStream_t st, int k, const T* S_, const T* N, double* lam, unsigned* emax) {
  launch_pdl(quotients_kernel<T>, ceil_div(k, 128), 128, 0, st, k, S_, N, lam, emax);
  CHASE_CHECK_LAUNCH();
}

// id: the columns' clusters.  emax: the bits of the largest |re| + |im| (NaN stays largest).  S and N are Hermitian up to
// rounding, which a small gap would amplify into a loss of orthonormality: their Hermitian parts are taken.
template <typename T>
__global__ void __launch_bounds__(128) correction_kernel(int k, const T* __restrict__ S_, const T* __restrict__ N,
                                                          const double* __restrict__ lam, const int* __restrict__ id, T* E,
                                                          unsigned* emax) {
  grid_dependency_wait();
  using s = S<T>;
  const int p = blockIdx.x * blockDim.x + threadIdx.x, q = blockIdx.y;
  unsigned bits = 0u;
  if (p < k) {
    const int64_t pq = p + (int64_t)q * k, qp = q + (int64_t)p * k;
    T r = s::scale(s::add(N[pq], s::conj(N[qp])), -0.5);
    T v;
    if (p == q) {
      v = s::make(0.5 + 0.5 * s::re(r), 0.0);
    } else if (id[p] == id[q]) {
      v = s::scale(r, 0.5);
    } else {
      const T sv = s::scale(s::add(S_[pq], s::conj(S_[qp])), 0.5);
      v = s::scale(s::add(sv, s::scale(r, lam[q])), 1.0 / (lam[q] - lam[p]));
    }
    E[pq] = v;
    bits = __float_as_uint(fabsf((float)s::re(v)) + fabsf((float)s::im(v)));
  }
  bits = __reduce_max_sync(0xffffffffu, bits);
  if ((threadIdx.x & 31) == 0) atomicMax(emax, bits);
}

template <typename T>
void eig_correction(cudaStream_t st, int k, const T* S_, const T* N, const double* lam, const int* id, T* E, unsigned* emax) {
  launch_pdl(correction_kernel<T>, dim3(ceil_div(k, 128), k), 128, 0, st, k, S_, N, lam, id, E, emax);
  CHASE_CHECK_LAUNCH();
}

// One CTA per cluster [s, s+c), c <= CMAX, after Z <- Z (I + E): the block of the new quotient is S_pq + (l_p + l_q) E_pq up
// to the square of E (E = R / 2 inside a cluster).  Cyclic Jacobi on it, eigenvalues to w[s..s+c) (l before), then
// Z[:, s:s+c] <- Z[:, s:s+c] U in place, row by row, both in ascending order.
constexpr int CMAX = CLUSTER_MAX;
template <typename T>
__global__ void cluster_kernel(int k, const int* cl, const T* S_, const T* E, T* Z, int64_t ldz, double* w,
                               int* status) {
  using s = S<T>;
  const int start = cl[2 * blockIdx.x], c = cl[2 * blockIdx.x + 1];
  __shared__ T B[CMAX][CMAX + 1];
  __shared__ T U[CMAX][CMAX + 1];
  __shared__ T jpp, jpq, jqp, jqq;
  __shared__ int cont, rank[CMAX];
  for (int t = threadIdx.x; t < c * c; t += blockDim.x) {
    int i = t % c, j = t / c;
    const int64_t ij = (start + i) + (int64_t)(start + j) * k, ji = (start + j) + (int64_t)(start + i) * k;
    const T h = s::scale(s::add(S_[ij], s::conj(S_[ji])), 0.5);
    B[i][j] = s::add(h, s::scale(E[ij], w[start + i] + w[start + j]));
    U[i][j] = (i == j) ? s::one() : s::zero();
  }
  __syncthreads();
  int sweep = 0;
  for (; sweep < 40; ++sweep) {
    if (threadIdx.x == 0) {
      double fro = 0.0, off = 0.0;
      for (int i = 0; i < c; ++i)
        for (int j = 0; j < c; ++j) {
          double a = s::abs2(B[i][j]);
          fro += a;
          if (i != j) off += a;
        }
      cont = (sqrt(off) > 1e-15 * sqrt(fro)) && fro > 0.0;
    }
    __syncthreads();
    if (!cont) break;
    for (int p = 0; p < c - 1; ++p)
      for (int q = p + 1; q < c; ++q) {
        if (threadIdx.x == 0) {
          T g = B[p][q];
          double ag = magnitude(g);
          if (!(ag > 1e-300)) {
            jpp = s::one();
            jpq = s::zero();
            jqp = s::zero();
            jqq = s::one();
          } else {
            double z = (s::re(B[q][q]) - s::re(B[p][p])) / (2.0 * ag);
            double t = (z >= 0.0 ? 1.0 : -1.0) / (fabs(z) + sqrt(1.0 + z * z));
            double cc = 1.0 / sqrt(1.0 + t * t), sn = t * cc;
            T ph = s::scale(s::conj(g), 1.0 / ag);
            jpp = s::make(cc, 0.0);
            jpq = s::make(sn, 0.0);
            jqp = s::scale(ph, -sn);
            jqq = s::scale(ph, cc);
          }
        }
        __syncthreads();
        int i = threadIdx.x;
        if (i < c) {  // columns p, q of B and U
          T bp = B[i][p], bq = B[i][q];
          B[i][p] = s::add(s::mul(bp, jpp), s::mul(bq, jqp));
          B[i][q] = s::add(s::mul(bp, jpq), s::mul(bq, jqq));
          T up = U[i][p], uq = U[i][q];
          U[i][p] = s::add(s::mul(up, jpp), s::mul(uq, jqp));
          U[i][q] = s::add(s::mul(up, jpq), s::mul(uq, jqq));
        }
        __syncthreads();
        if (i < c) {  // rows p, q of B
          T rp = B[p][i], rq = B[q][i];
          B[p][i] = s::add(s::mul(s::conj(jpp), rp), s::mul(s::conj(jqp), rq));
          B[q][i] = s::add(s::mul(s::conj(jpq), rp), s::mul(s::conj(jqq), rq));
        }
        __syncthreads();
        if (i == 0) {
          B[p][q] = s::zero();
          B[q][p] = s::zero();
          B[p][p] = s::make(s::re(B[p][p]), 0.0);
          B[q][q] = s::make(s::re(B[q][q]), 0.0);
        }
        __syncthreads();
      }
  }
  if (threadIdx.x == 0 && sweep >= 40) atomicMax(status, 1);
  // ascending (stable) order: the next pass tells clusters by the distance between neighbours
  for (int i = threadIdx.x; i < c; i += blockDim.x) {
    const double wi = s::re(B[i][i]);
    int r = 0;
    for (int j = 0; j < c; ++j) r += (s::re(B[j][j]) < wi) || (s::re(B[j][j]) == wi && j < i);
    w[start + r] = wi;
    rank[i] = r;
  }
  __syncthreads();
  // Z[:, start:start+c] <- Z[:, start:start+c] U
  for (int r = threadIdx.x; r < k; r += blockDim.x) {
    T row[CMAX];
#pragma unroll
    for (int j = 0; j < CMAX; ++j)
      if (j < c) row[j] = Z[r + (int64_t)(start + j) * ldz];
#pragma unroll
    for (int j = 0; j < CMAX; ++j) {
      if (j >= c) continue;
      T acc = s::zero();
#pragma unroll
      for (int m = 0; m < CMAX; ++m)
        if (m < c) acc = s::fma(row[m], U[m][j], acc);
      Z[r + (int64_t)(start + rank[j]) * ldz] = acc;
    }
  }
}

template <typename T>
void cluster_eig(cudaStream_t st, int k, int nclusters, const int* cl, const T* S_, const T* E, T* Z, int64_t ldz,
                 double* w, int* status) {
  if (nclusters <= 0) return;
  cluster_kernel<T><<<nclusters, 128, 0, st>>>(k, cl, S_, E, Z, ldz, w, status);
  CHASE_CHECK_LAUNCH();
}

template <typename T> __global__ void rank_kernel(int k, const double* w, double* wout, int* perm) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= k) return;
  double wi = w[i];
  int rank = 0;
  for (int j = 0; j < k; ++j) rank += (w[j] < wi) || (w[j] == wi && j < i);
  wout[rank] = wi;
  perm[rank] = i;
}

template <typename T>
void sort_pairs(cudaStream_t st, int k, double* w, const T* Z, int64_t ldz, T* out, int64_t ldo, double* wtmp, int* perm) {
  rank_kernel<T><<<ceil_div(k, 128), 128, 0, st>>>(k, w, wtmp, perm);
  CHASE_CHECK_LAUNCH();
  permute_cols<T>(st, k, k, Z, ldz, out, ldo, perm);
  CHASE_CUDA(cudaMemcpyAsync(w, wtmp, k * sizeof(double), cudaMemcpyDeviceToDevice, st));
}

#define INST(T)                                                                                                  \
  template void eig_quotients<T>(cudaStream_t, int, const T*, const T*, double*, unsigned*);                      \
  template void eig_correction<T>(cudaStream_t, int, const T*, const T*, const double*, const int*, T*, unsigned*); \
  template void cluster_eig<T>(cudaStream_t, int, int, const int*, const T*, const T*, T*, int64_t, double*, int*); \
  template void sort_pairs<T>(cudaStream_t, int, double*, const T*, int64_t, T*, int64_t, double*, int*);
INST(double)
INST(double2)
#undef INST
template void convert_mat<double, float>(cudaStream_t, int, const double*, int64_t, float*, int64_t);
template void convert_mat<float, double>(cudaStream_t, int, const float*, int64_t, double*, int64_t);
template void convert_mat<double2, float2>(cudaStream_t, int, const double2*, int64_t, float2*, int64_t);
template void convert_mat<float2, double2>(cudaStream_t, int, const float2*, int64_t, double2*, int64_t);

}  // namespace chase
