// Lowest eigenpairs of the small symmetric Davidson matrices, float64, one CTA
// (paper, Section "GPU Implementation", batched step 3: diagonalise the
// projected matrix and keep the lowest K states).
//
// This part's float64 pipe issues one warp instruction per 64 cycles per
// sub-partition whatever the number of active lanes, and a float64 divide
// costs ~640 cycles, so the kernel keeps float64 work in as few warps as hold
// data and moves what can be approximate to float32:
//   1. Householder tridiagonalisation Q^T A Q = T in float64 on the packed
//      lower triangle (shared memory up to S = kSmemMax = 224, else global
//      scratch); the reflectors stay in the triangle's columns, reductions run
//      in integers in the warps that hold data, scalars come from float32
//      estimates;
//   2. the k lowest eigenvalues of T by Sturm-count multisection in float32,
//      one warp per eigenvalue and 32 counts per round, to ~2e-7 |T|;
//   3. inverse iteration on T (pivoted tridiagonal LU, one thread per
//      eigenvector): two float32 solves with the float32 shift, then two
//      float64 solves shifted by the Rayleigh quotient; the Rayleigh quotient
//      of the result is the float64 eigenvalue (its error is quadratic in the
//      vector's).  Eigenvalues closer than 2e-6 |T| form clusters, which take in
//      what lies within 1e-4 |T| of them: start vectors of their own, two float64
//      solves with the float32 shift, two shifted by the Rayleigh quotient and one
//      more with the float32 shift, each followed by Gram-Schmidt against the members
//      already found and, up to eight members, a Rayleigh-Ritz rotation inside the
//      cluster;
//   4. back-transformation z = H_0 H_1 ... H_{S-3} y in blocks of eight
//      reflectors (compact WY form).
// Figures are at syevk_body.
//
// Also: Cholesky factorisation a = L L^T of the TDHF matrix a- (positive
// definite unless the reference is unstable); 70 x 70 104 -> 70 us, 100 x 100
// 177 -> 127 us since the pivot's root and reciprocal come from a float32
// estimate in the warps that scale the column and the trailing update has no
// idle lanes.
#include <cfloat>

#include "kernels.h"
#include "prof.h"
#include "syev.h"
#include "syev_body.cuh"

namespace xs {

namespace {

// (S <= kSmemMax runs with 512 threads: the float64 pipe is full at four warps a
// sub-partition, and barriers cost half of what 1024 threads pay)
template <bool SMEM>
__global__ void __launch_bounds__(SMEM ? 512 : 1024) syevk_kernel(int S, int k, const double* __restrict__ Ain, int lda,
                                                     double* __restrict__ wout, double* __restrict__ Z, int ldz,
                                                     double* __restrict__ gscratch, int* info, bool zsm) {
  syevk_body<SMEM>(S, k, Ain, lda, wout, Z, ldz, gscratch, info, zsm);
}

template <bool SMEM>
__global__ void __launch_bounds__(SMEM ? 512 : 1024) cholesky_kernel(int S, double* A, int lda, int* flag) {
  cholesky_body<SMEM>(S, A, lda, flag);
}

}  // namespace


void syevk(cudaStream_t s, int S, int k, const double* A, int lda, double* w, double* Z, int ldz,
           DevBuf<double>& scratch, int* info) {
  if (S <= 0 || k <= 0) return;
  if (k > S) k = S;
  if (S > 1024) throw Error(XS_EINVAL, "syevk: matrix larger than 1024");
  // working set (matrix, tridiagonal, reflector, products, eigenvalues,
  // float32 copy, cluster indices) in doubles
  const size_t wd = syevk_work_doubles(S);
  scratch.ensure(syevk_scratch_doubles(S, k));
  ProfScope ps(s, "syevk_f64", 0.0, (4.0 / 3.0) * S * (double)S * S);
  if (S <= kSmemMax) {
    const bool zsm = syevk_z_fits(S, k);
    const size_t smem = sizeof(double) * (wd + (zsm ? syevk_z_doubles(S, k) : 0));
    static std::atomic<unsigned long long> allowed{0};
    allow_smem(allowed, syevk_kernel<true>, sizeof(double) * kEigSmemDoubles);
    syevk_kernel<true><<<1, 512, smem, s>>>(S, k, A, lda, w, Z, ldz, scratch.get(), info, zsm);
  } else {
    syevk_kernel<false><<<1, 1024, 0, s>>>(S, k, A, lda, w, Z, ldz, scratch.get(), info, false);
  }
  XS_CHECK_LAUNCH();
}

void cholesky(cudaStream_t s, int S, double* A, int lda, int* flag) {
  if (S <= 0) return;
  ProfScope ps(s, "cholesky_f64", 0.0, S * (double)S * S / 3.0);
  if (S <= kCholSmemMax) {
    const size_t smem = sizeof(double) * (size_t)S * (S + 1) / 2;
    static std::atomic<unsigned long long> allowed{0};
    allow_smem(allowed, cholesky_kernel<true>, sizeof(double) * kCholSmemMax * (kCholSmemMax + 1) / 2);
    cholesky_kernel<true><<<1, 512, smem, s>>>(S, A, lda, flag);
  } else {
    cholesky_kernel<false><<<1, 1024, 0, s>>>(S, A, lda, flag);
  }
  XS_CHECK_LAUNCH();
}

}  // namespace xs
