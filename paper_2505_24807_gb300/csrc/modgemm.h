// Float64 matrix products on the BF16 tensor cores by residues (modgemm.cu).
//
// C = A B^T with float64 A (M x K) and B (N x K).  Every row of A and B is
// scaled by a power of two of its 2-norm and rounded to 57-bit integers a', b'
// (the rounding is 2^-58 of the row's norm per element), the integer product
// C' = sum a' b' is formed exactly modulo 13 pairwise coprime moduli m_l <= 512,
// and C' (|C'| <= 2^114 by Cauchy-Schwarz, a quarter of the moduli's product)
// is recovered by the Chinese remainder theorem: the second scheme of Ozaki,
// Uchino and Imamura (arXiv:2504.08009), here with bfloat16 residues instead of
// 8-bit integers, whose tensor rate on this part is far below bfloat16's.
// Residues |r| <= 256 are exact in bfloat16 (8 significant bits), 256 products
// of two of them sum exactly in a float32 accumulator (2^8 2^16 = 2^24).  13
// bfloat16 products replace one on the float64 pipe (1.2 TFLOP/s measured).
//
// The error is relative to the rows' norms: every entry of a row is rounded to
// 2^-58 of a power of two at most 2.01 times its norm, so an output is off by at most
// 2^-57 (|a| sum|b_k| + |b| sum|a_k|) before its one rounding to float64, about 2^-57.8 |a| |b|
// with entries of random signs, against about 2^-54 |a| |b| of a K-term float64
// accumulation.  An entry 2^-k of its row's norm keeps 57 - k bits, and an output in
// which only small entries meet (graded rows, distant fragments) is not accurate to
// its own size, as a float64 GEMM's would be.  Products A X and (A + B) X of 4 response
// vectors against a float64 evaluation elsewhere, root mean square of the difference
// over that of the part that the transforms form: 2200 AOs 2.3e-15 and 2.6e-15 (float64
// pipe 2.9e-15 and 3.2e-15), 579 AOs 1.3e-15 and 1.6e-15 (1.6e-15, 1.8e-15), 222 AOs
// 8.3e-16 and 9.7e-16 (9.9e-16, 1.1e-15).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace xs {

constexpr int kModuli = 13;
// largest K: mg_split_rows stages a row of K float64 in shared memory, 64 KB of the
// 227 KB a CTA may have, so that three CTAs share an SM.  (The sums of a product's
// chunks, 32 of them below 2^8 at this K, would stay exact in float32 to K = 2^23.)
constexpr int kMgMaxK = 8192;
using mg_t = uint16_t;             // bfloat16 bit pattern of one residue

// K-major operand of a product: `batch` matrices (1: shared by the batch) of
// rows x K float64 at src + b bs + r rs + k ks (rs or ks is 1), its residue
// planes [modulus][batch][rows][Kp] and row exponents [batch][rows].
struct MgOperand {
  const double* src = nullptr;
  long long rs = 0, ks = 1, bs = 0;
  int rows = 0, K = 0, batch = 1;
  const mg_t* planes = nullptr;
  const int* exps = nullptr;
};

// Residue planes of one operand, kept where the operand is.
struct MgPlanes {
  DevBuf<mg_t> planes;
  DevBuf<int> exps;
};

// Scratch of one context: operands that change with every product, and the
// residues of the result.
struct MgWork {
  MgPlanes a, b;
  DevBuf<uint16_t> res;
};

inline int mg_kp(int K) { return (K + 63) / 64 * 64; }
inline int mg_ldn(int N) { return (N + 15) / 16 * 16; }
inline size_t mg_plane_count(int rows, int K, int batch) {
  return static_cast<size_t>(kModuli) * batch * rows * mg_kp(K);
}

// Split op.src into residue planes (p, grown as needed) and point op at them.
// side 0: left operand (A), side 1: right operand (B, residues premultiplied
// by the remainder theorem's weights).
void mg_split(cudaStream_t s, int side, MgOperand& op, MgPlanes& p);

// C[b] (M x N, row stride ldc, batch stride sC) = alpha A[b] B[b]^T + beta C[b]
// for b < batch, plus, when X is set, (eps[o + col] - eps[row]) X[b] (X with
// C's layout).  d_err: device word raised when a bounded wait gave up.
struct MgOut {
  double* C = nullptr;
  int ldc = 0;
  long long sC = 0;
  double alpha = 1.0, beta = 0.0;
  const double* X = nullptr;
  const double* eps = nullptr;
  int o = 0;
};
void mg_product(cudaStream_t s, const MgOperand& A, const MgOperand& B, int batch, const MgOut& out, MgWork& w,
                int* d_err);

}  // namespace xs
