// Split-precision (TF32 or float16 hi + lo) tensor-core GEMM of libxs (tc_gemm.cu).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace xs {

// One K-major operand: rows x Kpad pairs (hi, lo), row stride ld (16-byte rows
// and base), batch entries bstride apart when batched.  Kpad is a multiple of 32
// and the padding columns are zero.  T = float: TF32 pairs.  T = __half: float16
// pairs of x 2^-e, with one exponent e per batch entry (one for the operand when
// it is not batched) that puts the entry's largest |x|, or a bound of it, just below
// 2^15.  Down to 2^-17 of that a value has the two 11-bit significands of a TF32 pair;
// below, the low half meets float16's smallest step, 2^-25 absolute, 2^-40 of the
// largest: smaller values keep fewer bits than a TF32 pair's 22 and end there.
template <typename T>
struct TcPair {
  const T* hi;
  const T* lo;
  int ld;
  long long bstride;
  bool batched;
  const int* e = nullptr;   // T = __half: device exponents
};
using TcOperand = TcPair<float>;
using TcOperand16 = TcPair<__half>;

// Epilogue: mode 0 stores float D and, when rowmax is set, raises rowmax[b] to the
// bits of the largest |D| of batch entry b (the caller zeroes it first); mode 1
// stores the TF32 pair (D, Dlo) of the result; mode 2 (float16 pairs in and out)
// stores the pair (Dh, Dhl) of D 2^-eout[b] with eout[b] = eA + eB + 15 +
// ceil(log2 Kpad), which bounds |D| whatever the operands hold, and eout[b].
struct TcEpilogue {
  int mode = 0;
  float* D = nullptr;
  float* Dlo = nullptr;
  int ld = 0;
  long long bstride = 0;
  unsigned int* rowmax = nullptr;
  __half* Dh = nullptr;
  __half* Dhl = nullptr;
  int* eout = nullptr;
};

// D[b] (M x N) = A[b] B[b]^T from TF32 pairs: hi*hi + hi*lo + lo*hi, float32
// accumulation.  d_err: device int set to a nonzero code when a bounded
// device-side wait timed out.  The first call of a new problem class runs the
// product several times (tile-width timing), so the output must not alias an
// input.
void tc_gemm(cudaStream_t s, const TcOperand& A, const TcOperand& B, int M, int N, int Kpad, int batch,
             const TcEpilogue& e, int* d_err);
// The same product from float16 pairs (modes 0 and 2), at twice the TF32 rate.
void tc_gemm(cudaStream_t s, const TcOperand16& A, const TcOperand16& B, int M, int N, int Kpad, int batch,
             const TcEpilogue& e, int* d_err);

// Zero-padded TF32 pair of a row-major matrix (rows x cols, source row stride
// ld_src), optionally transposed (dst[r][c] = src[c][r]); batched over
// grid.z with the given strides.
template <typename S>
void split_pad(cudaStream_t s, int rows, int cols, int ld_dst, const S* src, int ld_src, long long sstride,
               long long dstride, int batch, bool transpose, float* hi, float* lo);

// Transposed split of float64 matrices through shared-memory tiles:
// dst[r][c] (rows x ld_dst) = TF32 pair of src[c][r] for c < cols, zero up to
// ld_dst; src holds cols rows of row stride ld_src; batched over grid.z.
void split_pad_t(cudaStream_t s, int rows, int cols, int ld_dst, const double* src, int ld_src, long long sstride,
                 long long dstride, int batch, float* hi, float* lo);

int pad32(int k);

// Y = D + (eps_a - eps_i) X of nvec o x v vectors; rowmax (optional, zeroed by
// the caller): per vector raised to abs_hi of the largest |Y|
void add_gaps(cudaStream_t s, int nvec, int o, int v, const double* eps, const float* D, const double* X, double* Y,
              unsigned int* rowmax);

// Float16 pairs (TcPair<__half>).  amax: per batch entry, the bits of the largest
// |x| (abs_hi of a double for float64 sources, a float's bits for float32 ones);
// the split writes the entry's exponent to e.
// raise amax to the largest |x| (abs_hi) of float64 batch entries of `count` elements, sstride apart
void absmax_f64(cudaStream_t s, long long count, const double* src, long long sstride, int batch, unsigned int* amax);
// float64 source, plain or transposed: dst[r][c] = src[r][c] or src[c][r], zero up to ld_dst
void split16(cudaStream_t s, int rows, int cols, int ld_dst, const double* src, int ld_src, long long sstride,
             long long dstride, int batch, bool transpose, const unsigned int* amax, int* e, __half* hi, __half* lo);
// float32 source of row stride cols (sstride between batch entries)
void split16(cudaStream_t s, int rows, int cols, int ld_dst, const float* src, long long sstride, long long dstride,
             int batch, const unsigned int* amax, int* e, __half* hi, __half* lo);

}  // namespace xs
