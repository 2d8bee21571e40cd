// FP64-class products from residues (tcgen05), host interface.  See crt.cu.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.h"

namespace chase {
namespace crt {

constexpr int NMOD = 16;  // moduli
// residue planes per modulus: real operands one; complex ones re, im and re + im
constexpr int planes(bool cplx) { return cplx ? 3 : 1; }
inline int64_t kpad(int64_t K) { return (K + 7) / 8 * 8; }   // plane row pitch (16-byte rows for TMA)
inline int64_t rpad(int64_t M) { return (M + 15) / 16 * 16; }   // pitch of the product's residue columns

// Bytes of the residue planes of nvec vectors of length K for nmod moduli
inline int64_t plane_bytes(int64_t nvec, int64_t K, bool cplx, int nmod) {
  return (int64_t)nmod * planes(cplx) * nvec * kpad(K) * 2;
}
// Bytes of the residues of an M x N product (all moduli)
inline int64_t residue_bytes(int64_t M, int64_t N, bool cplx) { return (int64_t)NMOD * planes(cplx) * N * rpad(M); }

// Exponents ex[v] with the 2-norm of vector v below 2^ex[v] (NONFINITE when the vector holds a NaN or an
// infinity): vector = column of the column-major X (K rows), or row when by_rows.
constexpr int NONFINITE = 0x7fffffff;
template <typename T>
void scales(cudaStream_t st, bool by_rows, int64_t nvec, int64_t K, const T* X, int64_t ldx, int* ex);

// Residue planes of the moduli [mod0, mod0 + nmod): plane ((i - mod0) * planes + p), each nvec rows of kpad(K)
// bf16 values.  conj negates the imaginary part.
template <typename T>
void residues(cudaStream_t st, bool by_rows, bool conj, int64_t nvec, int64_t K, const T* X, int64_t ldx, const int* ex,
              int mod0, int nmod, void* planes);

// One product C = L R (M x N, inner length K) from residue planes.  The left planes cover the moduli
// [mod0, mod0 + nmod) only; the right planes and the residues R cover all of them.
struct Product {
  const void* lpl;
  const int* lex;
  void* rpl;
  int* rex;
  void* res;
  int64_t M, N, K;
  Epi e;
  const void* X;  // the right operand (K x N, column-major), for right_planes
  int64_t ldx;
};

// exponents and planes (all moduli) of the products' right operands, one launch per 64 products
template <typename T> void right_planes(cudaStream_t st, const Product* ops, int nops);

// residues of the products for the moduli [mod0, mod0 + nmod), one launch per 64 products
template <bool CPLX>
void multiply(cudaStream_t st, const Product* ops, int nops, int mod0, int nmod, int* err);
// C = alpha * product + gamma ycol Y + beta Z from the residues of all moduli, one launch per 64 products
template <bool CPLX> void combine(cudaStream_t st, const Product* ops, int nops);

}  // namespace crt
}  // namespace chase
