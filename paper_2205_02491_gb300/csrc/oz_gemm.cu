// Split tensor-core products, host side: the workspace, the FP64-class products (residue planes, crt.cu) in passes
// over A's moduli and panels of columns, and the mixed modes' digit planes, launch-configuration tuner, K-split
// planning and dispatch to the tcgen05 kernel of oz_kernel.cuh, whose instantiations live in the oz_inst_*.cu units.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "crt.h"
#include "oz.h"
#include "oz_kernel.cuh"

namespace chase {
namespace oz {
// ---------------------------------------------------------------- split kernels
// Digits of one value x with |x| < s = 2^e: d_t = rint(r_t), r_0 = x/s * 2^7, r_{t+1} = (r_t - d_t) 2^8; a plane stores
// d_t 2^-8t.  Rounding to nearest even is symmetric and looks no further than 2^-16 of r_0, so the digits come exactly
// from |r_0| in 32-bit fixed point (23 fraction bits, the last one also set by anything below it): FP64 instructions
// (nine per digit) bound this kernel otherwise (n = 5003 real: A 786 us).
template <int NS> __device__ __forceinline__ void digits(double x, int e, float (&out)[NS]) {
  const uint32_t hi = (uint32_t)__double2hiint(x);
  const int be = (int)((hi >> 20) & 0x7ff);
  if (be == 2047 || e < -1000 || e > 1000) {  // non-finite, or a scale near the ends of the range
    double r = ldexp(x, 7 - e);  // exact; 1 / 2^e overflows for a subnormal column
#pragma unroll
    for (int t = 0; t < NS; ++t) {
      const double d = rint(r);
      out[t] = (float)d;
      r = (r - d) * 256.0;
    }
    return;
  }
  const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | (be ? 0x100000u : 0u)) << 32) | (uint32_t)__double2loint(x);
  const int n = min(1045 + e - (be ? be : 1), 63);  // x = m 2^(be - 1075); at least 23
  const uint32_t q = (uint32_t)(m >> n);
  int v = (int)(q | (((unsigned long long)q << n) != m ? 1u : 0u));
#pragma unroll
  for (int t = 0; t < NS; ++t) {
    const int sh = 23 - 8 * t;
    const int d = (v + ((1 << (sh - 1)) - 1) + ((v >> sh) & 1)) >> sh;
    v -= d << sh;
    const int sd = (int)hi < 0 ? -d : d;
    out[t] = __int_as_float(0x4b400000 + sd) - 12582912.0f;
  }
}
__device__ __forceinline__ uint32_t pack_planes(float a, float b, float sc) {  // exact: at most 8 significant bits
  return __byte_perm(__float_as_uint(a * sc), __float_as_uint(b * sc), 0x7632);
}

// Scales and digit planes of the columns of X (conjugated when conj), a cluster of CTAs per column (512 elements each while
// K <= 4096): the column's largest magnitude f 2^e, f in [0.5, 1), gives its scale 2^e (1 for a zero column or a
// non-finite one).  Left-operand planes (KIND 0): (t, p), p in {re, im}; right-operand planes: p in {-im, re, im}; real:
// one plane per slice.  Layout planes[(t*P + p) * ncols + col][Kpad].
// n = 5003 real: A 88 us (scales and digits by separate FP64 kernels: 860), 300 right columns 14 us (39).
template <typename T, int NS, int KIND>
__global__ void __launch_bounds__(128) split_kernel(int64_t K, int64_t Kpad, int ncols, const T* __restrict__ X, int64_t ldx,
                                                    double* scale, int conj, __nv_bfloat16* planes) {
  using s = S<T>;
  __shared__ uint32_t part[32];
  __shared__ double slow[4];
  const int rank = (int)blockIdx.x, cs = (int)gridDim.x, col = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  grid_dependency_wait();
  const int64_t slice = ((K + cs - 1) / cs + 3) / 4 * 4;
  const int64_t k0 = rank * slice, k1 = k0 + slice < K ? k0 + slice : K;
  const T* x = X + (int64_t)col * ldx;
  auto load4 = [&](T (&v)[4], int64_t i) {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = i + j < k1 ? x[i + j] : s::zero();
  };
  auto top = [&](const T& v) {
    return max((uint32_t)__double2hiint(s::re(v)) & 0x7fffffffu, (uint32_t)__double2hiint(s::im(v)) & 0x7fffffffu);
  };
  T v[4];
  const int64_t i0 = k0 + 4 * tid;
  load4(v, i0);  // stays in registers when the slice is 512 elements
  uint32_t m = max(max(top(v[0]), top(v[1])), max(top(v[2]), top(v[3])));
  for (int64_t i = i0 + 512; i < k1; i += 512) {
    T u[4];
    load4(u, i);
    m = max(m, max(max(top(u[0]), top(u[1])), max(top(u[2]), top(u[3]))));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");  // every CTA of the cluster runs
  if (lane < cs) {
    uint32_t to;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(to)
                 : "r"((uint32_t)__cvta_generic_to_shared(&part[4 * rank + warp])), "r"(lane));
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(to), "r"(m) : "memory");
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  m = __reduce_max_sync(0xffffffffu, lane < 4 * cs ? part[lane] : 0u);
  int e = 0;
  double sc = 1.0;
  if (m < 0x00100000u) {  // a zero column, or subnormal throughout
    double w = 0.0;
    for (int64_t i = tid; i < K; i += 128) w = fmax(w, fmax(fabs(s::re(x[i])), fabs(s::im(x[i]))));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w = fmax(w, __shfl_xor_sync(0xffffffffu, w, o));
    if (lane == 0) slow[warp] = w;
    __syncthreads();
    w = fmax(fmax(slow[0], slow[1]), fmax(slow[2], slow[3]));
    if (w > 0.0) {
      frexp(w, &e);
      sc = ldexp(1.0, e);
    }
  } else if (m < 0x7ff00000u) {
    e = (int)(m >> 20) - 1022;
    sc = ldexp(1.0, e);
  }
  if (rank == 0 && tid == 0) scale[col] = sc;
  auto write4 = [&](const T (&u)[4], int64_t i) {
    float dr[4][NS], di[4][NS];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      digits<NS>(s::re(u[j]), e, dr[j]);
      if (s::cplx) digits<NS>(conj ? -s::im(u[j]) : s::im(u[j]), e, di[j]);
    }
    float f = 1.0f;
#pragma unroll
    for (int t = 0; t < NS; ++t, f *= 0.00390625f) {
      constexpr int P = s::cplx ? (KIND == 0 ? 2 : 3) : 1;
      auto put = [&](int p, const float (&d)[4][NS], float g) {
        *reinterpret_cast<uint2*>(planes + ((int64_t)(t * P + p) * ncols + col) * Kpad + i) =
            make_uint2(pack_planes(d[0][t], d[1][t], g), pack_planes(d[2][t], d[3][t], g));
      };
      if (!s::cplx) {
        put(0, dr, f);
      } else if (KIND == 0) {
        put(0, dr, f);
        put(1, di, f);
      } else {
        put(0, di, -f);
        put(1, dr, f);
        put(2, di, f);
      }
    }
  };
  if (i0 < k1) write4(v, i0);
  for (int64_t i = i0 + 512; i < k1; i += 512) {
    load4(v, i);
    write4(v, i);
  }
}

// ---------------------------------------------------------------- host side
static int slices_for(int mode) { return mode == 2 ? 2 : MIXED_SLICES; }  // BF16x3, BF16x6

bool available() {
  // thread-safe one-time probe (batched solves call this from several host threads)
  static const bool ok = []() {
    int dev = 0, major = 0, minor = 0;
    return cudaGetDevice(&dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) == cudaSuccess && major == 10 &&
           minor == 3 && encode_fn() != nullptr;
  }();
  return ok;
}

// ---------------------------------------------------------------- workspace
// Residues of a product are kept for panels of its columns: at most this many bytes, but at least 256 columns.
// 6 GB hold the n = 30000, 1600-column block (2.3 GB) whole.
constexpr int64_t RESIDUE_PANEL_BYTES = 6ll << 30;

// The fewest moduli of A's residue planes a workspace holds at a time: with the mixed modes' three digit slices
// their memory is 24 bytes per complex element of A (14 for real); all 16 moduli take 96 bytes beside those digits
// (32 for real).
static int fewest_mods(bool complex_) { return complex_ ? 2 : 4; }

static int panel_cols(int64_t n_max, int ne_max, bool complex_) {
  const int64_t per = crt::residue_bytes(n_max, 1, complex_);
  const int64_t fit = RESIDUE_PANEL_BYTES / per / 256 * 256;
  return (int)std::min<int64_t>(ne_max, std::max<int64_t>(256, fit));
}

static int64_t left_bytes(int64_t n_max, int ne_max, bool complex_) {
  return std::max(crt::plane_bytes(n_max, ne_max, complex_, crt::NMOD), crt::plane_bytes(ne_max, n_max, complex_, crt::NMOD));
}

static int64_t right_bytes(int64_t n_max, int ne_max, bool complex_) {
  const int64_t digits = (int64_t)MIXED_SLICES * (complex_ ? 3 : 1) * ne_max * kpad(n_max) * 2;
  return std::max(digits, crt::plane_bytes(panel_cols(n_max, ne_max, complex_), n_max, complex_, crt::NMOD));
}

static int64_t digit_bytes(int64_t n_max, bool complex_) {
  return (int64_t)MIXED_SLICES * (complex_ ? 2 : 1) * n_max * kpad(n_max) * 2;
}

// partial sums of K-split mixed products: up to about 4 waves of 128 x 64 complex tiles
constexpr int64_t PARTIAL_ELEMS = 8ll << 20;

int a_mods_within(int64_t n_max, bool complex_, int64_t budget) {
  const int64_t fit = budget / crt::plane_bytes(n_max, n_max, complex_, 1);
  return (int)std::max<int64_t>(fewest_mods(complex_), std::min<int64_t>(fit, crt::NMOD));
}

int64_t workspace_bytes(int64_t n_max, int ne_max, bool complex_, int a_mods) {
  if (a_mods == 0) a_mods = fewest_mods(complex_);
  return crt::plane_bytes(n_max, n_max, complex_, a_mods) + left_bytes(n_max, ne_max, complex_) +
         right_bytes(n_max, ne_max, complex_) +
         crt::residue_bytes(n_max, panel_cols(n_max, ne_max, complex_), complex_) + digit_bytes(n_max, complex_) +
         (2 * n_max + 2 * (int64_t)ne_max) * 8 + 64 + PARTIAL_ELEMS * 8;
}

void create(Workspace& w, int64_t n_max, int ne_max, bool complex_, int a_mods) {
  w.n_max = n_max;
  w.ne_max = ne_max;
  w.complex_ = complex_;
  if (!available()) return;
  w.b_bytes = right_bytes(n_max, ne_max, complex_);
  w.residue_bytes = crt::residue_bytes(n_max, panel_cols(n_max, ne_max, complex_), complex_);
  CHASE_CUDA(cudaMalloc(&w.l_res, left_bytes(n_max, ne_max, complex_)));
  CHASE_CUDA(cudaMalloc(&w.b_planes, w.b_bytes));
  CHASE_CUDA(cudaMalloc(&w.residue, w.residue_bytes));
  CHASE_CUDA(cudaMalloc(&w.a_planes, digit_bytes(n_max, complex_)));
  CHASE_CUDA(cudaMalloc(&w.a_ex, n_max * sizeof(int)));
  CHASE_CUDA(cudaMalloc(&w.l_ex, std::max<int64_t>(n_max, ne_max) * sizeof(int)));
  CHASE_CUDA(cudaMalloc(&w.b_ex, std::max<int64_t>(n_max, ne_max) * sizeof(int)));
  CHASE_CUDA(cudaMalloc(&w.a_scale, n_max * sizeof(double)));
  CHASE_CUDA(cudaMalloc(&w.b_scale, ne_max * sizeof(double)));
  CHASE_CUDA(cudaMalloc(&w.flags, 16 * sizeof(int)));
  CHASE_CUDA(cudaMemset(w.flags, 0, 16 * sizeof(int)));
  w.partial_elems = PARTIAL_ELEMS;
  CHASE_CUDA(cudaMalloc(&w.partial, (size_t)w.partial_elems * sizeof(double)));
  // A's planes last, and fewer where the memory that was free when a_mods was chosen has gone to someone else since
  for (w.a_mods = a_mods;; w.a_mods = std::max(fewest_mods(complex_), w.a_mods / 2)) {
    const cudaError_t err = cudaMalloc(&w.a_res, crt::plane_bytes(n_max, n_max, complex_, w.a_mods));
    if (err == cudaSuccess) break;
    w.a_res = nullptr;
    cudaGetLastError();
    CHASE_REQUIRE(err == cudaErrorMemoryAllocation && w.a_mods > fewest_mods(complex_),
                  err == cudaErrorMemoryAllocation ? 2 : 6, std::string("residue planes: ") + cudaGetErrorString(err));
  }
  w.ready = true;
}

int64_t shrink(Workspace& w) {
  const int fewest = fewest_mods(w.complex_), had = w.a_mods;
  if (!w.ready || had <= fewest) return 0;
  const int64_t bytes = crt::plane_bytes(w.n_max, w.n_max, w.complex_, fewest);
  void* kept = nullptr;
  if (cudaMalloc(&kept, bytes) != cudaSuccess) {  // no room beside the old planes
    cudaGetLastError();
    CHASE_CUDA(cudaFree(w.a_res));
    w.a_res = nullptr;
    w.ready = false;  // should the allocation fail
    CHASE_CUDA(cudaMalloc(&kept, bytes));
    w.ready = true;
  } else {
    CHASE_CUDA(cudaFree(w.a_res));
  }
  w.a_res = kept;
  w.a_mods = fewest;
  w.a_src = nullptr;
  return crt::plane_bytes(w.n_max, w.n_max, w.complex_, had - fewest);
}

void destroy(Workspace& w) {
  void* ps[] = {w.a_res,   w.l_res,   w.b_planes, w.residue, w.a_planes, w.a_ex,
                w.l_ex,    w.b_ex,    w.a_scale,  w.b_scale, w.flags,    w.partial};
  for (void* p : ps)
    if (p) cudaFree(p);
  for (auto& e : w.ev) cudaEventDestroy(e);
  for (auto& kv : w.tune)
    for (auto& e : kv.second.ev)
      if (e) cudaEventDestroy(e);
  w = Workspace{};
}

// Digit planes of nvec columns of length K of a column-major X (optionally conjugated).
// kind 0: left-operand planes (re, im); kind 1: right-operand planes (-im, re, im).
template <typename T>
static void split(cudaStream_t st, int S_, int kind, bool conj, const T* X, int64_t ld, int64_t nvec, int64_t K,
                  void* planes, double* scale) {
  // a cluster only as far as it fills the SMs (16 blocks each)
  int cs = 1;
  while (cs < 8 && 512 * cs < K && nvec * cs < 152 * 16) cs *= 2;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[2] = {{}, pdl_attribute()};
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(128, 1, 1);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  const int64_t kp = kpad(K);
  CHASE_REQUIRE(nvec <= 65535, 1, "split: too many vectors");
  cfg.gridDim = dim3(cs, (unsigned)nvec, 1);
  auto go = [&](auto kernel) {
    CHASE_CUDA(cudaLaunchKernelEx(&cfg, kernel, K, kp, (int)nvec, X, ld, scale, conj ? 1 : 0, (__nv_bfloat16*)planes));
  };
  if (S_ == 2 && kind == 1) go(split_kernel<T, 2, 1>);
  else if (S_ == 3 && kind == 1) go(split_kernel<T, 3, 1>);
  else if (S_ == 3 && kind == 0) go(split_kernel<T, 3, 0>);
  else CHASE_REQUIRE(false, 1, "unsupported slice count");
  CHASE_CHECK_LAUNCH();
}

template <typename T>
void prepare_A(cudaStream_t st, Workspace& w, const T* A, int64_t n, int64_t lda, int mode) {
  CHASE_REQUIRE(w.ready, 9, "split products not initialised");
  // A Hermitian: K-major row i of A = conjugate of column i of its column-major storage
  if (mode == 2 || mode == 3) {
    // the three-slice split's first slices are the two-slice split
    if (w.d_src == (const void*)A && w.d_n == n) return;
    split<T>(st, MIXED_SLICES, 0, true, A, lda, n, n, w.a_planes, w.a_scale);
    w.d_src = A;
    w.d_n = n;
    return;
  }
  if (w.a_src == (const void*)A && w.a_n == n) return;
  crt::scales<T>(st, false, n, n, A, lda, w.a_ex);
  if (w.a_mods == crt::NMOD) crt::residues<T>(st, false, true, n, n, A, lda, w.a_ex, 0, crt::NMOD, w.a_res);
  w.a_src = A;
  w.a_n = n;
}

void timing_begin(Workspace& w) {
  if (w.ev.empty()) {
    w.ev.resize(256);
    for (auto& e : w.ev) CHASE_CUDA(cudaEventCreate(&e));
  }
  w.ev_used = w.timed = 0;
  w.span_open = false;
  w.timing = true;
}

double timing_collect(cudaStream_t st, Workspace& w, int* launches) {
  ProductTimer::close(st, w);
  double ms = 0.0;
  for (int i = 0; i + 1 < w.ev_used; i += 2) {
    CHASE_CUDA(cudaEventSynchronize(w.ev[i + 1]));
    float t = 0.f;
    CHASE_CUDA(cudaEventElapsedTime(&t, w.ev[i], w.ev[i + 1]));
    ms += t;
  }
  if (launches) *launches = w.timed;
  w.ev_used = 0;
  w.timing = false;
  return ms;
}

void invalidate(Workspace& w) {
  w.a_src = w.d_src = nullptr;
  w.a_n = w.d_n = 0;
  if (w.flags) CHASE_CUDA(cudaMemset(w.flags, 0, 16 * sizeof(int)));  // a new call starts clean
}

// ---------------------------------------------------------------- FP64-class products
// columns of a product (M rows, inner length K) whose right planes and residues fit the workspace
static int64_t panel_fit(const Workspace& w, int64_t M, int64_t K) {
  const int64_t by_res = w.residue_bytes / crt::residue_bytes(M, 1, w.complex_);
  const int64_t by_rhs = w.b_bytes / crt::plane_bytes(1, K, w.complex_, crt::NMOD);
  return std::min(by_res, by_rhs);
}

static Epi at_column(const Epi& e, int64_t j, size_t esz) {
  Epi o = e;
  o.C = (char*)e.C + (size_t)(j * e.ldc) * esz;
  if (e.Y) o.Y = (const char*)e.Y + (size_t)(j * e.ldy) * esz;
  if (e.Z) o.Z = (const char*)e.Z + (size_t)(j * e.ldz) * esz;
  if (e.ycol) o.ycol = e.ycol + j;
  return o;
}

// C = L R by panels of columns.  lconv(mod0, nmod): makes the left planes of those moduli current (called for passes
// of `mods` moduli); the right operand's columns (rows when by_rows) are converted per panel.
template <typename T, typename LeftConv>
static void product(cudaStream_t st, Workspace& w, const void* lpl, const int* lex, int mods, LeftConv lconv, bool by_rows,
                    const T* B, int64_t ldb, int64_t M, int64_t N, int64_t K, const Epi& e) {
  const int64_t fit = panel_fit(w, M, K);
  CHASE_REQUIRE(fit >= 1, 1, "split product exceeds the workspace");
  for (int64_t j = 0; j < N; j += fit) {
    const int64_t nc = std::min(fit, N - j);
    const T* Bj = by_rows ? B + j : B + j * ldb;
    const crt::Product op{lpl, lex, w.b_planes, w.b_ex, w.residue, M, nc, K, at_column(e, j, sizeof(T)), Bj, ldb};
    if (by_rows) {
      crt::scales<T>(st, true, nc, K, Bj, ldb, w.b_ex);
      crt::residues<T>(st, true, true, nc, K, Bj, ldb, w.b_ex, 0, crt::NMOD, w.b_planes);
    } else {
      crt::right_planes<T>(st, &op, 1);
    }
    ProductTimer t(st, w, 2.0 * crt::NMOD * crt::planes(S<T>::cplx) * (double)M * (double)nc * (double)K);
    for (int m0 = 0; m0 < crt::NMOD; m0 += mods) {
      const int nm = std::min(mods, crt::NMOD - m0);
      lconv(m0, nm);
      crt::multiply<S<T>::cplx>(st, &op, 1, m0, nm, w.flags);
    }
    crt::combine<S<T>::cplx>(st, &op, 1);
    t.stop();
  }
}

// ---------------------------------------------------------------- launch-configuration tuner
// Candidates of the mixed kernels: the tile-order group size and the tile width (256 columns halve the instructions
// per unit of tensor work).
static const LaunchCfg kCand[] = {{128, 4}, {128, 16}, {256, 4}, {256, 16}};

static int log2_bucket(int64_t x) {
  int b = 0;
  while (x > 1) {
    x >>= 1;
    ++b;
  }
  return b;
}

// Size class of a launch: arithmetic, element type, grouped or not, and the log2 buckets of the shape.
static uint64_t tune_key(int S_, bool cplx, bool grouped, int64_t M, int64_t N, int64_t K) {
  return ((uint64_t)S_ << 56) | ((uint64_t)cplx << 55) | ((uint64_t)grouped << 54) |
         ((uint64_t)log2_bucket(M) << 36) | ((uint64_t)log2_bucket(N) << 18) | (uint64_t)log2_bucket(K);
}

// The configuration for the next launch of a size class.  Until every candidate has been timed, each
// launch takes the next candidate and gets an event pair (*ev_out); the first launch after that reads
// the times (one event synchronisation per size class and context) and keeps the fastest.
static LaunchCfg tune_pick(Workspace& w, uint64_t key, cudaEvent_t** ev_out) {
  const LaunchCfg* cand = kCand;
  const int nc = (int)(sizeof(kCand) / sizeof(kCand[0]));
  *ev_out = nullptr;
  if (!w.autotune) return LaunchCfg{128, w.group_m};
  TuneEntry& t = w.tune[key];
  if (t.best >= 0) return cand[t.best];
  if (t.ev.empty()) {
    t.ev.resize(2 * nc, nullptr);
    for (auto& e : t.ev) CHASE_CUDA(cudaEventCreate(&e));
  }
  if (t.next < nc) {
    *ev_out = &t.ev[2 * t.next];
    return cand[t.next++];
  }
  float best_ms = 0.f;
  int best = 0;
  for (int i = 0; i < nc; ++i) {
    CHASE_CUDA(cudaEventSynchronize(t.ev[2 * i + 1]));
    float ms = 0.f;
    CHASE_CUDA(cudaEventElapsedTime(&ms, t.ev[2 * i], t.ev[2 * i + 1]));
    if (i == 0 || ms < best_ms) {
      best_ms = ms;
      best = i;
    }
  }
  t.best = best;
  return cand[best];
}

std::vector<std::pair<uint64_t, int>> tuned(const Workspace& w) {
  std::vector<std::pair<uint64_t, int>> out;
  for (const auto& kv : w.tune)
    if (kv.second.best >= 0) out.emplace_back(kv.first, kv.second.best);
  return out;
}

static int sm_count() {
  static const int n = []() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return 148;
    return sms;
  }();
  return n;
}

// A product with fewer output tiles than two per SM is split along K (slices of at least 384, multiples of
// 96, at most 16 of them, within the partial-sum buffer) so that its launch covers the GPU.
static void plan_ksplit(Workspace& w, ProductOp& op, int ncols_tile, bool cplx) {
  const int64_t tiles = (int64_t)ceil_div(op.N, ncols_tile) * (int64_t)ceil_div(op.M, BM);
  const int64_t want = 2 * (int64_t)sm_count();
  if (tiles >= want || op.K < 2 * 384 || !w.partial) return;
  int64_t ks = std::min<int64_t>({16, ceil_div(want, tiles), op.K / 384});
  const int64_t per = op.M * op.N * (cplx ? 2 : 1);
  ks = std::min<int64_t>(ks, w.partial_elems / std::max<int64_t>(1, per));
  if (ks <= 1) return;
  const int64_t klen = ((op.K + ks - 1) / ks + 95) / 96 * 96;
  op.klen = (int)klen;
  op.ksplit = (int)ceil_div(op.K, klen);
  op.part = w.partial;
  if (op.ksplit <= 1) {
    op.ksplit = 1;
    op.part = nullptr;
  }
}

template <int S, bool CPLX, int NTT>
static void launch(cudaStream_t st, Workspace& w, int64_t M, int64_t N, int64_t K, const Epi& e, int group_m,
                   cudaEvent_t* tune_ev) {
  ProductOp op{w.a_planes, w.a_scale, MIXED_SLICES, w.b_planes, w.b_scale, M, N, K, e, group_m};
  plan_ksplit(w, op, Cfg<S, CPLX, NTT>::NCOLS, CPLX);
  launch_ops<S, CPLX, NTT, 1>(st, w, &op, 1, tune_ev);
}

template <typename T>
void split_right(cudaStream_t st, Workspace& w, int mode, const T* B, int64_t ldb, int k, int64_t n) {
  CHASE_REQUIRE(w.ready, 9, "split products not initialised");
  CHASE_REQUIRE(k <= w.ne_max && n <= w.n_max, 1, "split_right: size exceeds the workspace");
  split<T>(st, slices_for(mode), 1, false, B, ldb, k, n, w.b_planes, w.b_scale);
}

template <bool CPLX>
void launch_group(cudaStream_t st, Workspace& w, int mode, const ProductOp* ops, int nops) {
  constexpr int G = 64;
  const int S_ = slices_for(mode);
  std::vector<ProductOp> chunk;
  for (int q0 = 0; q0 < nops; q0 += G) {
    const int cnt = std::min(G, nops - q0);
    // size class of a grouped launch: its total work in row blocks x columns x K
    int64_t rows = 0, cols = 0, kk = 0;
    for (int q = q0; q < q0 + cnt; ++q) {
      rows += ops[q].M;
      cols = std::max(cols, ops[q].N);
      kk = std::max(kk, ops[q].K);
    }
    cudaEvent_t* ev = nullptr;
    const LaunchCfg cfg = tune_pick(w, tune_key(S_, CPLX, true, rows, cols, kk), &ev);
    chunk.assign(ops + q0, ops + q0 + cnt);
    for (auto& o : chunk) o.group_m = cfg.group_m;
    const ProductOp* cp = chunk.data();
    if (S_ == 3 && cfg.nt == 256) launch_ops<3, CPLX, 256, G>(st, w, cp, cnt, ev);
    else if (S_ == 3) launch_ops<3, CPLX, 128, G>(st, w, cp, cnt, ev);
    else if (cfg.nt == 256) launch_ops<2, CPLX, 256, G>(st, w, cp, cnt, ev);
    else launch_ops<2, CPLX, 128, G>(st, w, cp, cnt, ev);
  }
}

bool groupable(const Workspace& w, int64_t n, int k) { return w.a_mods == crt::NMOD && k <= panel_fit(w, n, n); }

template <typename T>
crt::Product group_product(Workspace& w, const T* B, int64_t ldb, int k, int64_t n, const Epi& e) {
  CHASE_REQUIRE(w.ready, 9, "split products not initialised");
  return crt::Product{w.a_res, w.a_ex, w.b_planes, w.b_ex, w.residue, n, k, n, e, B, ldb};
}

template <typename T> void multiply_group(cudaStream_t st, Workspace& w, const crt::Product* ops, int nops) {
  crt::right_planes<T>(st, ops, nops);
  crt::multiply<S<T>::cplx>(st, ops, nops, 0, crt::NMOD, w.flags);
  crt::combine<S<T>::cplx>(st, ops, nops);
}

template <typename T>
void hemm(cudaStream_t st, Workspace& w, const T* A, int64_t n, int64_t lda, const T* B, int64_t ldb, int k,
          const Epi& e, int mode) {
  constexpr bool CPLX = S<T>::cplx;
  CHASE_REQUIRE(w.ready, 9, "split products not initialised");
  CHASE_REQUIRE(k <= w.ne_max && n <= w.n_max, 1, "hemm size exceeds the workspace");
  CHASE_REQUIRE(n <= 65472, 1, "split products support K <= 65472");
  if (mode != 2 && mode != 3) {
    CHASE_REQUIRE(w.a_src == (const void*)A && w.a_n == n, 7, "prepare_A must precede hemm");
    auto conv = [&](int m0, int nm) {
      if (w.a_mods < crt::NMOD) crt::residues<T>(st, false, true, n, n, A, lda, w.a_ex, m0, nm, w.a_res);
    };
    product<T>(st, w, w.a_res, w.a_ex, w.a_mods, conv, false, B, ldb, n, k, n, e);
    return;
  }
  CHASE_REQUIRE(w.d_src == (const void*)A && w.d_n == n, 7, "prepare_A must precede hemm");
  const int S_ = slices_for(mode);
  split<T>(st, S_, 1, false, B, ldb, k, n, w.b_planes, w.b_scale);
  cudaEvent_t* ev = nullptr;
  const LaunchCfg cfg = tune_pick(w, tune_key(S_, CPLX, false, n, k, n), &ev);
  if (S_ == 3 && cfg.nt == 256) launch<3, CPLX, 256>(st, w, n, k, n, e, cfg.group_m, ev);
  else if (S_ == 3) launch<3, CPLX, 128>(st, w, n, k, n, e, cfg.group_m, ev);
  else if (cfg.nt == 256) launch<2, CPLX, 256>(st, w, n, k, n, e, cfg.group_m, ev);
  else launch<2, CPLX, 128>(st, w, n, k, n, e, cfg.group_m, ev);
}

// left operand: OP_N rows of A (M x K), OP_C conjugated columns of A (K x M)
template <typename T>
void left_planes(cudaStream_t st, Op opA, const T* A, int64_t lda, int64_t M, int64_t K, void* planes, int* ex) {
  crt::scales<T>(st, opA == OP_N, M, K, A, lda, ex);
  crt::residues<T>(st, opA == OP_N, opA == OP_C, M, K, A, lda, ex, 0, crt::NMOD, planes);
}

template <typename T>
void gemm_planes(cudaStream_t st, Workspace& w, const void* planes, const int* ex, const T* B, int64_t ldb, int64_t M,
                 int64_t N, int64_t K, const Epi& e) {
  CHASE_REQUIRE(w.ready, 9, "split products not initialised");
  if (M <= 0 || N <= 0) return;
  product<T>(st, w, planes, ex, crt::NMOD, [](int, int) {}, false, B, ldb, M, N, K, e);
}

template <typename T>
void gemm(cudaStream_t st, Workspace& w, Op opA, const T* A, int64_t lda, Op opB, const T* B, int64_t ldb, int64_t M,
          int64_t N, int64_t K, const Epi& e) {
  constexpr bool CPLX = S<T>::cplx;
  CHASE_REQUIRE(w.ready, 9, "split products not initialised");
  if (M <= 0 || N <= 0) return;
  CHASE_REQUIRE(N <= w.n_max && M <= w.n_max &&
                    crt::plane_bytes(M, K, CPLX, crt::NMOD) <= left_bytes(w.n_max, w.ne_max, CPLX),
                1, "split product exceeds the workspace");
  // right operand: OP_N columns of B (K x N), OP_C conjugated rows of B (N x K).  The left planes of all moduli are
  // made first, so C may overwrite A.
  left_planes<T>(st, opA, A, lda, M, K, w.l_res, w.l_ex);
  product<T>(st, w, w.l_res, w.l_ex, crt::NMOD, [](int, int) {}, opB == OP_C, B, ldb, M, N, K, e);
}

int read_flags(cudaStream_t st, Workspace& w) {
  if (!w.ready) return 0;
  int f = 0;
  CHASE_CUDA(cudaMemcpyAsync(&f, w.flags, sizeof(int), cudaMemcpyDeviceToHost, st));
  CHASE_CUDA(cudaStreamSynchronize(st));
  return f;
}

template void prepare_A<double>(cudaStream_t, Workspace&, const double*, int64_t, int64_t, int);
template void prepare_A<double2>(cudaStream_t, Workspace&, const double2*, int64_t, int64_t, int);
template void hemm<double>(cudaStream_t, Workspace&, const double*, int64_t, int64_t, const double*, int64_t, int,
                           const Epi&, int);
template void gemm<double>(cudaStream_t, Workspace&, Op, const double*, int64_t, Op, const double*, int64_t, int64_t,
                           int64_t, int64_t, const Epi&);
template void gemm<double2>(cudaStream_t, Workspace&, Op, const double2*, int64_t, Op, const double2*, int64_t, int64_t,
                            int64_t, int64_t, const Epi&);
template void left_planes<double>(cudaStream_t, Op, const double*, int64_t, int64_t, int64_t, void*, int*);
template void left_planes<double2>(cudaStream_t, Op, const double2*, int64_t, int64_t, int64_t, void*, int*);
template void gemm_planes<double>(cudaStream_t, Workspace&, const void*, const int*, const double*, int64_t, int64_t,
                                  int64_t, int64_t, const Epi&);
template void gemm_planes<double2>(cudaStream_t, Workspace&, const void*, const int*, const double2*, int64_t, int64_t,
                                   int64_t, int64_t, const Epi&);
template crt::Product group_product<double>(Workspace&, const double*, int64_t, int, int64_t, const Epi&);
template crt::Product group_product<double2>(Workspace&, const double2*, int64_t, int, int64_t, const Epi&);
template void multiply_group<double>(cudaStream_t, Workspace&, const crt::Product*, int);
template void multiply_group<double2>(cudaStream_t, Workspace&, const crt::Product*, int);
template void hemm<double2>(cudaStream_t, Workspace&, const double2*, int64_t, int64_t, const double2*, int64_t, int,
                            const Epi&, int);
template void split_right<double>(cudaStream_t, Workspace&, int, const double*, int64_t, int, int64_t);
template void split_right<double2>(cudaStream_t, Workspace&, int, const double2*, int64_t, int, int64_t);
template void launch_group<false>(cudaStream_t, Workspace&, int, const ProductOp*, int);
template void launch_group<true>(cudaStream_t, Workspace&, int, const ProductOp*, int);

}  // namespace oz
}  // namespace chase
