// Split tensor-core products (tcgen05) of the eigensolver: FP64-class products through residues (crt.cu) and the
// mixed-precision filter products through digit planes (oz_kernel.cuh), with their workspace.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <map>
#include <vector>

#include "crt.h"
#include "kernels.h"

namespace chase {
namespace oz {

// Launch configuration of the mixed-precision product kernel chosen by measurement (see tune_pick in oz_gemm.cu):
// the tile width NT (128 or 256 columns) and the tile-order group size.
struct LaunchCfg {
  int nt = 128;
  int group_m = 8;
};

// One size class of the tuner: candidates are timed on consecutive launches of that class (the degree
// steps of a filter repeat one shape), then the fastest is kept for the context's lifetime.
struct TuneEntry {
  int next = 0;          // candidates launched so far
  int best = -1;         // index of the chosen candidate once every one has been timed
  std::vector<cudaEvent_t> ev;  // start/stop pair per candidate
};

constexpr int MIXED_SLICES = 3;  // digit slices of A held for the mixed modes (BF16x3 uses the first two)

struct Workspace {
  bool ready = false;
  bool complex_ = true;
  int64_t n_max = 0;
  int ne_max = 0;
  // FP64-class products
  void* a_res = nullptr;      // residue planes of A: a_mods moduli at a time
  int a_mods = 0;             // crt::NMOD: all of them stay resident; fewer: converted per product in passes
  void* l_res = nullptr;      // residue planes of a general left operand
  void* residue = nullptr;    // residues of a product (residue_bytes)
  int64_t residue_bytes = 0;
  int* a_ex = nullptr;        // per-row exponents of A
  int* l_ex = nullptr;        // of the general left operand
  int* b_ex = nullptr;        // per-column exponents of the right operand
  // mixed modes
  void* a_planes = nullptr;   // bf16 digit planes of A (MIXED_SLICES slices)
  double* a_scale = nullptr;  // per-row power-of-two scale of A
  double* b_scale = nullptr;  // per-column scale of the right operand
  double* partial = nullptr;  // FP64 partial sums of products split along K
  int64_t partial_elems = 0;
  void* b_planes = nullptr;   // planes of the right operand (residues or digits, b_bytes)
  int64_t b_bytes = 0;
  int* flags = nullptr;       // device error flags of the bounded waits
  int group_m = 8;            // row blocks per tile group of the mixed launch order (untuned launches)
  bool autotune = true;       // choose LaunchCfg per size class by timing the candidates
  std::map<uint64_t, TuneEntry> tune;  // size class -> measurements and choice
  // optional CUDA-event timing of the product kernels (filter roofline)
  bool timing = false;
  std::vector<cudaEvent_t> ev;
  int ev_used = 0;
  bool span_open = false;  // a span of small products has its start recorded in ev[ev_used]
  int timed = 0;           // products timed
  // A whose exponents and residues (a_src) or digit planes (d_src) are held
  const void* a_src = nullptr;
  int64_t a_n = 0;
  const void* d_src = nullptr;
  int64_t d_n = 0;
};

// One product C = L R of a grouped mixed-precision launch: digit planes and scales of both operands, sizes,
// epilogue and the tile-order group size.
struct ProductOp {
  const void* lpl;
  const double* lsc;
  int l_slices_total;
  const void* rpl;
  const double* rsc;
  int64_t M, N, K;
  Epi e;
  int group_m;
  int ksplit = 1;           // K slices (> 1: partial sums to `part`, then a reduction launch)
  int klen = 0;             // slice length along K (multiple of 96)
  double* part = nullptr;   // ksplit x M x N (x 2 complex) doubles
};

bool available();
// Bytes of a workspace that holds the residue planes of A for a_mods moduli (0: the fewest it works with).
int64_t workspace_bytes(int64_t n_max, int ne_max, bool complex_, int a_mods);
// Moduli of A that `budget` bytes hold, between the fewest and all.
int a_mods_within(int64_t n_max, bool complex_, int64_t budget);
// Planes of A for a_mods moduli, or of fewer (the fewest at least) when the allocation fails.
void create(Workspace& w, int64_t n_max, int ne_max, bool complex_, int a_mods);
// Gives back A's planes beyond the fewest (no call may be using them); the bytes given back.
int64_t shrink(Workspace& w);
void destroy(Workspace& w);
// the tuner's choices so far: (size-class key, candidate index) pairs, for reports
std::vector<std::pair<uint64_t, int>> tuned(const Workspace& w);
void invalidate(Workspace& w);
// start recording event pairs around the product kernels (ProductTimer); collect returns (ms, products)
void timing_begin(Workspace& w);
double timing_collect(cudaStream_t st, Workspace& w, int* launches);

// Event pair around one product's kernels (filter roofline), or, for products of less than SPAN_FLOPS of bf16 work (100
// us), one pair around a whole run of them and what lies between.  Nothing overlaps across an event, and a pair takes
// about 10 us of a small product's 32: a pair each cost a solve with n = 512 1.6 of 10.6 ms, with n = 3001 1.5 of 52.
struct ProductTimer {
  static constexpr double SPAN_FLOPS = 2e11;
  cudaStream_t st;
  Workspace& w;
  bool on = false;
  ProductTimer(cudaStream_t s, Workspace& ws, double flops) : st(s), w(ws) {
    if (!w.timing) return;
    if (flops >= SPAN_FLOPS) close(st, w);
    if (w.span_open) {
      ++w.timed;
    } else if (w.ev_used + 2 <= (int)w.ev.size()) {
      CHASE_CUDA(cudaEventRecord(w.ev[w.ev_used], st));
      ++w.timed;
      if (flops >= SPAN_FLOPS) on = true;
      else w.span_open = true;
    }
  }
  void stop() {
    if (on) end(st, w);
  }
  static void close(cudaStream_t st, Workspace& w) {
    if (w.span_open) end(st, w);
    w.span_open = false;
  }
  static void end(cudaStream_t st, Workspace& w) {
    CHASE_CUDA(cudaEventRecord(w.ev[w.ev_used + 1], st));
    w.ev_used += 2;
  }
};
int read_flags(cudaStream_t st, Workspace& w);
// planes of A for the given mode (cached until invalidate)
template <typename T>
void prepare_A(cudaStream_t st, Workspace& w, const T* A, int64_t n, int64_t lda, int mode);
// C = A B with epilogue (prepare_A first)
template <typename T>
void hemm(cudaStream_t st, Workspace& w, const T* A, int64_t n, int64_t lda, const T* B, int64_t ldb, int k,
          const Epi& e, int mode);
// C = op(A) op(B) (M x N, inner K), FP64 class; op(A) = A (M x K) or A^H (A: K x M), op(B) = B (K x N) or B^H
// (B: N x K).  C may be A's storage.
template <typename T>
void gemm(cudaStream_t st, Workspace& w, Op opA, const T* A, int64_t lda, Op opB, const T* B, int64_t ldb, int64_t M,
          int64_t N, int64_t K, const Epi& e);

// The same with a left operand that is converted once for several products: its planes (crt::plane_bytes(M, K, ...)
// bytes, 16-byte aligned) and M exponents.
template <typename T>
void left_planes(cudaStream_t st, Op opA, const T* A, int64_t lda, int64_t M, int64_t K, void* planes, int* ex);
template <typename T>
void gemm_planes(cudaStream_t st, Workspace& w, const void* planes, const int* ex, const T* B, int64_t ldb, int64_t M,
                 int64_t N, int64_t K, const Epi& e);

// Grouped launches over several problems' workspaces.  Mixed modes: digit planes of the right operand B
// (n x k, ld ldb) into w's right-operand buffer, then one launch (per 64 products) over the tiles of all products.
template <typename T>
void split_right(cudaStream_t st, Workspace& w, int mode, const T* B, int64_t ldb, int k, int64_t n);
template <bool CPLX> void launch_group(cudaStream_t st, Workspace& w, int mode, const ProductOp* ops, int nops);
// FP64: whether w's next product C = A B of k columns can join a group; its operands; and the group's launches.
bool groupable(const Workspace& w, int64_t n, int k);
template <typename T>
crt::Product group_product(Workspace& w, const T* B, int64_t ldb, int k, int64_t n, const Epi& e);
template <typename T> void multiply_group(cudaStream_t st, Workspace& w, const crt::Product* ops, int nops);

}  // namespace oz
}  // namespace chase
