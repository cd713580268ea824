// Device bodies of libxs's small float64 eigensolver and Cholesky factor:
// one CTA (up to 1024 threads) per matrix.  Included by syev.cu (one matrix
// per launch) and batch.cu (one matrix per CTA, one CTA per molecule).  The
// algorithm is described at the top of syev.cu.
#pragma once

#include <cfloat>

#include "common.cuh"
#include "f64_estimates.cuh"

namespace xs {
namespace {


constexpr int kSmemMax = 224;   // largest S whose working set fits in shared memory
constexpr int kSeg = 8;         // row segments of the tridiagonalisation's matrix-vector product
constexpr int kMaxRR = 8;       // clusters up to this size get a Rayleigh-Ritz rotation
constexpr int kScaleFree = 12;  // matrices with entries up to 2^+-12 are not scaled

// packed lower triangle: element (i, j), j <= i
__host__ __device__ __forceinline__ int tri(int i, int j) { return i * (i + 1) / 2 + j; }   // i <= 1024

__device__ __forceinline__ double warp_sum(double x) {
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// block-wide sum (red: 33 doubles); every thread gets the result
__device__ double block_sum(double x, double* red) {
  x = warp_sum(x);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();
  if (l == 0) red[w] = x;
  __syncthreads();
  if (w == 0) {
    double y = l < nw ? red[l] : 0.0;
    y = warp_sum(y);
    if (l == 0) red[32] = y;
  }
  __syncthreads();
  return red[32];
}

// Sum of a warp's 32 values off the float64 pipe (a shuffle tree of adds takes
// 540 cycles, this 300): the values as integers of 2^(emax - 57), emax the
// largest exponent, added by the warp's integer reduction in 26-bit limbs.
// Each is truncated at 2^-57 of the largest, below the rounding of the tree.
__device__ __forceinline__ double warp_sum_int(double x) {
  const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
  const int ex = static_cast<int>((bits >> 52) & 0x7FF);
  const int emax = __reduce_max_sync(0xffffffffu, ex);
  if (emax > 1900 || emax < 100) return warp_sum(x);   // non-finite, or near the ends of the range
  const int sh = emax - ex;
  const unsigned long long mant = ex ? (((bits & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << 5) : 0ull;
  const unsigned long long m = sh > 63 ? 0ull : mant >> sh;
  const long long q = (bits >> 63) ? -static_cast<long long>(m) : static_cast<long long>(m);
  const unsigned l0 = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(q) & 0x3FFFFFFu);
  const unsigned l1 = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(q >> 26) & 0x3FFFFFFu);
  const int l2 = __reduce_add_sync(0xffffffffu, static_cast<int>(q >> 52));
  const long long t =
      static_cast<long long>(l0) + (static_cast<long long>(l1) << 26) + static_cast<long long>(static_cast<unsigned long long>(l2) << 52);
  if (t == 0) return 0.0;
  const double d = static_cast<double>(t);              // exponent field 1023 .. 1086
  return __hiloint2double(__double2hiint(d) + (emax - 1080) * (1 << 20), __double2loint(d));
}

// number of eigenvalues of the float32 tridiagonal (d, e^2) below x
__device__ int sturm_count_f(int n, const float* d, const float* e2, float x, float pivmin) {
  int c = 0;
  float q = d[0] - x;
  if (q < 0.0f) ++c;
  for (int i = 1; i < n; ++i) {
    if (fabsf(q) < pivmin) q = -pivmin;
    q = d[i] - x - __fdividef(e2[i - 1], q);
    if (q < 0.0f) ++c;
  }
  return c;
}

// y^T T y for the float64 tridiagonal (d, e), y with stride ldy
__device__ double rayleigh(int n, const double* d, const double* e, const double* y, int ldy) {
  double s = 0.0, yp = 0.0;
  for (int i = 0; i < n; ++i) {
    const double yi = y[(long long)i * ldy];
    s = fma(d[i] * yi, yi, s);
    if (i > 0) s = fma(2.0 * e[i - 1] * yp, yi, s);
    yp = yi;
  }
  return s;
}

// Solve (T - shift I) x = y in place (y: stride ldy), factoring the pivoted
// LU into lu (5 n doubles: 1/pivot, the two super-diagonals of U, the
// multiplier, the row-swap flag; field f of row i at lu[(f n + i) ldy]) when
// factor is set, else reusing it; then normalise y unless raw.  Pivots below
// tiny are raised to tiny, and a row is not exchanged for a coupling below it: where
// the couplings fall off by many decades, exchanges for smaller and smaller ones would
// grow the vector past every range.
__device__ void inverse_step(int n, const double* d, const double* e, double shift, double tiny, bool factor,
                             double* lu, double* y, int ldy, bool raw = false) {
  const int fs = n * ldy;
  double* rc = lu;
  double* u1 = lu + fs;
  double* u2 = lu + 2 * fs;
  double* fm = lu + 3 * fs;
  double* sw = lu + 4 * fs;
  double cur = y[0];
  if (factor) {
    // the next row's entries are loaded a step ahead of the elimination chain
    double c0 = d[0] - shift, c1 = n > 1 ? e[0] : 0.0, c2 = 0.0;
    double pe = c1, pd = n > 1 ? d[1] : 0.0, py = n > 1 ? y[ldy] : 0.0;
    for (int i = 0; i + 1 < n; ++i) {
      double n0 = pe, n1 = pd - shift, nr = py;
      const bool more = i + 2 < n;
      pe = more ? e[i + 1] : 0.0;
      pd = more ? d[i + 2] : 0.0;
      py = more ? y[(i + 2) * ldy] : 0.0;
      double n2 = pe;
      const bool swp = mag_bits(n0) > mag_bits(c0) && mag_bits(n0) > mag_bits(tiny);
      const double t0 = c0, t1 = c1, t2 = c2, tr = cur;
      c0 = swp ? n0 : t0; c1 = swp ? n1 : t1; c2 = swp ? n2 : t2; cur = swp ? nr : tr;
      n0 = swp ? t0 : n0; n1 = swp ? t1 : n1; n2 = swp ? t2 : n2; nr = swp ? tr : nr;
      if (mag_bits(c0) < mag_bits(tiny)) c0 = copysign(tiny, c0);
      const double r = rcp_fast(c0);
      const double f = n0 * r;
      const int at = i * ldy;
      rc[at] = r; u1[at] = c1; u2[at] = c2; fm[at] = f; sw[at] = swp ? 1.0 : 0.0;
      y[at] = cur;
      c0 = fma(-f, c1, n1);
      c1 = fma(-f, c2, n2);
      c2 = 0.0;
      cur = fma(-f, cur, nr);
    }
    if (mag_bits(c0) < mag_bits(tiny)) c0 = copysign(tiny, c0);
    const int at = (n - 1) * ldy;
    rc[at] = rcp_fast(c0); u1[at] = 0.0; u2[at] = 0.0;
    y[at] = cur;
  } else {
    double py = n > 1 ? y[ldy] : 0.0, ps = sw[0], pf = fm[0];
    for (int i = 0; i + 1 < n; ++i) {
      double nr = py;
      const double swi = ps, f = pf;
      const bool more = i + 2 < n;
      py = more ? y[(i + 2) * ldy] : 0.0;
      ps = more ? sw[(i + 1) * ldy] : 0.0;
      pf = more ? fm[(i + 1) * ldy] : 0.0;
      const bool swp = __double2hiint(swi) != 0;
      const double t = cur;
      cur = swp ? nr : t;
      nr = swp ? t : nr;
      y[i * ldy] = cur;
      cur = fma(-f, cur, nr);
    }
    y[(n - 1) * ldy] = cur;
  }
  // back substitution, then normalisation
  double y1 = 0.0, y2 = 0.0, nrm = 0.0;
  int at = (n - 1) * ldy;
  double qy = y[at], q1 = u1[at], q2 = u2[at], qr = rc[at];
  for (int i = n - 1; i >= 0; --i) {
    const double yy = qy, a1 = q1, a2 = q2, ar = qr;
    const int here = at;
    at -= ldy;
    if (i > 0) { qy = y[at]; q1 = u1[at]; q2 = u2[at]; qr = rc[at]; }
    const double yi = fma(-a1, y1, fma(-a2, y2, yy)) * ar;
    y[here] = yi;
    if (!raw) nrm = fma(yi, yi, nrm);
    y2 = y1;
    y1 = yi;
  }
  if (raw) return;
  const double inv = 1.0 / sqrt(nrm);
  for (int i = 0; i < n; ++i) y[(long long)i * ldy] *= inv;
}

// Two float32 inverse-iteration solves of (T - shift I) from the start vector in
// y, one factorisation (fields as in inverse_step); pivots below tiny are raised
// to it.  A solve grows the vector by 1 / |lambda - shift|, which has no lower
// bound in a graded T (a root coupled to the others by 1e-13 of |T| and a shift that
// rounds to its diagonal entry: 1e20 and more), so a grown vector is scaled back
// between the solves; what overflows all the same the caller finds in its norm.
__device__ void inverse_step_f(int n, const float* d, const float* e, float shift, float tiny, float* lu, float* y,
                               int ldy) {
  const int fs = n * ldy;
  float* rc = lu;
  float* u1 = lu + fs;
  float* u2 = lu + 2 * fs;
  float* fm = lu + 3 * fs;
  float* sw = lu + 4 * fs;
  for (int pass = 0; pass < 2; ++pass) {
    float cur = y[0];
    if (pass == 0) {
      float c0 = d[0] - shift, c1 = n > 1 ? e[0] : 0.0f, c2 = 0.0f;
      for (int i = 0; i + 1 < n; ++i) {
        float n0 = e[i], n1 = d[i + 1] - shift, n2 = i + 2 < n ? e[i + 1] : 0.0f, nr = y[(i + 1) * ldy];
        const bool swp = fabsf(n0) > fabsf(c0) && fabsf(n0) > tiny;
        const float t0 = c0, t1 = c1, t2 = c2, tr = cur;
        c0 = swp ? n0 : t0; c1 = swp ? n1 : t1; c2 = swp ? n2 : t2; cur = swp ? nr : tr;
        n0 = swp ? t0 : n0; n1 = swp ? t1 : n1; n2 = swp ? t2 : n2; nr = swp ? tr : nr;
        if (fabsf(c0) < tiny) c0 = copysignf(tiny, c0);
        const float r = __fdividef(1.0f, c0), f = n0 * r;
        const int at = i * ldy;
        rc[at] = r; u1[at] = c1; u2[at] = c2; fm[at] = f; sw[at] = swp ? 1.0f : 0.0f;
        y[at] = cur;
        c0 = fmaf(-f, c1, n1);
        c1 = fmaf(-f, c2, n2);
        c2 = 0.0f;
        cur = fmaf(-f, cur, nr);
      }
      if (fabsf(c0) < tiny) c0 = copysignf(tiny, c0);
      const int at = (n - 1) * ldy;
      rc[at] = __fdividef(1.0f, c0); u1[at] = 0.0f; u2[at] = 0.0f;
      y[at] = cur;
    } else {
      for (int i = 0; i + 1 < n; ++i) {
        float nr = y[(i + 1) * ldy];
        const int at = i * ldy;
        const bool swp = sw[at] != 0.0f;
        const float t = cur;
        cur = swp ? nr : t;
        nr = swp ? t : nr;
        y[at] = cur;
        cur = fmaf(-fm[at], cur, nr);
      }
      y[(n - 1) * ldy] = cur;
    }
    float y1 = 0.0f, y2 = 0.0f, top = 0.0f;
    for (int i = n - 1; i >= 0; --i) {
      const int at = i * ldy;
      const float yi = fmaf(-u1[at], y1, fmaf(-u2[at], y2, y[at])) * rc[at];
      y[at] = yi;
      top = fmaxf(top, fabsf(yi));
      y2 = y1;
      y1 = yi;
    }
    if (pass == 0 && top > 1e12f) {
      const float down = 1.0f / top;
      for (int i = 0; i < n; ++i) y[i * ldy] *= down;
    }
  }
}

// Jacobi eigen-decomposition of a c x c symmetric matrix (c <= kMaxRR), one
// thread: H is overwritten by its eigenvalues on the diagonal, R holds the
// eigenvectors in columns; then sorted ascending.
__device__ void jacobi_small(int c, double (*H)[kMaxRR], double (*R)[kMaxRR]) {
  for (int i = 0; i < c; ++i)
    for (int j = 0; j < c; ++j) R[i][j] = i == j ? 1.0 : 0.0;
  for (int sweep = 0; sweep < 12; ++sweep) {
    double off = 0.0, dia = 0.0;
    for (int i = 0; i < c; ++i)
      for (int j = 0; j < c; ++j) (i == j ? dia : off) += H[i][j] * H[i][j];
    if (off <= 1e-32 * dia || off == 0.0) break;
    for (int p = 0; p < c; ++p)
      for (int q = p + 1; q < c; ++q) {
        if (H[p][q] == 0.0) continue;
        const double th = (H[q][q] - H[p][p]) / (2.0 * H[p][q]);
        const double t = (th >= 0.0 ? 1.0 : -1.0) / (fabs(th) + sqrt(th * th + 1.0));
        const double cs = 1.0 / sqrt(t * t + 1.0), sn = t * cs;
        for (int k = 0; k < c; ++k) {
          const double hp = H[k][p], hq = H[k][q];
          H[k][p] = cs * hp - sn * hq;
          H[k][q] = sn * hp + cs * hq;
        }
        for (int k = 0; k < c; ++k) {
          const double hp = H[p][k], hq = H[q][k];
          H[p][k] = cs * hp - sn * hq;
          H[q][k] = sn * hp + cs * hq;
        }
        for (int k = 0; k < c; ++k) {
          const double rp = R[k][p], rq = R[k][q];
          R[k][p] = cs * rp - sn * rq;
          R[k][q] = sn * rp + cs * rq;
        }
      }
  }
  for (int i = 0; i < c; ++i)
    for (int j = i + 1; j < c; ++j)
      if (H[j][j] < H[i][i]) {
        const double t = H[i][i]; H[i][i] = H[j][j]; H[j][j] = t;
        for (int k = 0; k < c; ++k) { const double r = R[k][i]; R[k][i] = R[k][j]; R[k][j] = r; }
      }
}

// working set of syevk_body in doubles (matrix, tridiagonal, reflectors,
// products, eigenvalues, float32 copy, cluster indices); shared memory when
// S <= kSmemMax
__host__ __device__ constexpr size_t syevk_work_doubles(int n) {
  return (size_t)n * (n + 1) / 2 + (size_t)(8 + kSeg) * n + (n + 1) / 2 + 64;
}
// eigenvectors, inverse-iteration factors and back-transformation scratch: after
// the working set in shared memory when both fit (syevk_z_fits), else in
// global scratch
__host__ __device__ constexpr size_t syevk_z_doubles(int S, int k) { return (size_t)6 * S * k + (size_t)16 * k; }
constexpr size_t kEigSmemDoubles = 28968;   // 226.3 KB: the working set at S = 224
__host__ __device__ constexpr bool syevk_z_fits(int S, int k) {
  return S <= kSmemMax && syevk_work_doubles(S) + syevk_z_doubles(S, k) <= kEigSmemDoubles;
}
__host__ __device__ constexpr size_t syevk_scratch_doubles(int S, int k) {
  return (S <= kSmemMax ? 0 : syevk_work_doubles(S)) + syevk_z_doubles(S, k) + 64;
}

constexpr int kWy = 8;          // reflectors per block of the back-transformation

// zsm: the dynamic shared memory holds syevk_z_doubles(S, k) more doubles after
// the working set, else they are in gscratch.
//
// Every float64 instruction of a warp holds its sub-partition's pipe for 64
// cycles whatever the number of active lanes (latency 64 too), so the body is
// bound by the number of float64 instructions on its critical path.  Solve times
// before -> after the present form (one CTA): 48 x 48, 10 vectors 438 -> 203 us
// (tridiagonalisation 221 -> 106, inverse iteration 141 -> 56,
// back-transformation 72 -> 29); 100 x 100 1117 -> 567 us; 200 x 200 3316 ->
// 2474 us.
template <bool SMEM>
__device__ void syevk_body(int S, int k, const double* __restrict__ Ain, int lda, double* __restrict__ wout,
                           double* __restrict__ Z, int ldz, double* __restrict__ gscratch, int* info, bool zsm) {
  extern __shared__ double sh[];
  __shared__ double red[33];
  __shared__ double scal[8];
  double* base = SMEM ? sh : gscratch;
  double* a = base;                          // packed lower triangle; column j keeps reflector j below the diagonal
  double* d = a + tri(S, 0);
  double* e = d + S;
  double* beta = e + S;                      // reflector j: H_j = I - beta_j u_j u_j^T
  double* vb = beta + S;                     // two buffers of the current reflector u
  double* p = vb + 2 * S;                    // B u, then w
  double* ps = p + S;                        // kSeg x S matrix-vector partials
  double* lam = ps + (size_t)kSeg * S + 64;  // eigenvalues
  float* df = reinterpret_cast<float*>(lam + S);
  float* e2f = df + S;
  int* cl = reinterpret_cast<int*>(e2f + S); // first index of each eigenvalue's cluster
  double* gfree = gscratch + (SMEM ? 0 : syevk_work_doubles(S));
  double* Zw = SMEM && zsm ? sh + syevk_work_doubles(S) : gfree;   // S x k, row stride k
  double* lu = Zw + (size_t)S * k;                                 // 5 S x k, then 16 k
  const int tid = threadIdx.x, nt = blockDim.x;
  const int warp = tid >> 5, lane = tid & 31, nwarp = nt >> 5;

  // Entries whose largest lies outside 2^+-kScaleFree (products in eV and eV^2 do not)
  // are scaled by a power of two, undone on the eigenvalues: the float32 stages below
  // square and invert numbers of |T|'s size, and two unnormalised float32 solves grow
  // a vector to 1e16 / |T|^2, past float32 from |T| of 1e-11 down.
  __shared__ unsigned int tops[32];
  unsigned int top = 0;
  for (int i = warp; i < S; i += nwarp)
    for (int j = lane; j <= i; j += 32) {
      const double x = Ain[(long long)i * lda + j];
      a[tri(i, j)] = x;
      top = max(top, abs_hi(x));
    }
  top = __reduce_max_sync(0xffffffffu, top);
  if (lane == 0) tops[warp] = top;
  __syncthreads();
  for (int w = 0; w < nwarp; ++w) top = max(top, tops[w]);
  const bool zero = top == 0;              // zero, or below 2^-1042
  int scale = 0;
  {
    const int ex = static_cast<int>(top >> 20) - 1023;
    if (!zero && ex < 1024 && (ex < -kScaleFree || ex > kScaleFree)) scale = max(ex, -1000);
  }
  if (scale != 0) {
    for (int i = warp; i < S; i += nwarp)
      for (int j = lane; j <= i; j += 32) a[tri(i, j)] = scalbn(a[tri(i, j)], -scale);
    __syncthreads();
  }

  // 1. Tridiagonalisation by Householder reflectors H = I - beta u u^T on the
  // packed lower triangle.  The products of a step of m remaining rows take m^2
  // cycles (matrix-vector product and rank-2 update at two multiply-adds per
  // clock); the chain of reductions and scalars between them is kept short:
  // integer reductions, scalars from float32 estimates, u left unnormalised so
  // that beta is formed beside the matrix-vector product, and the next column's
  // norm formed beside the rank-2 update.

  // row segments of the matrix-vector product by remaining rows (segment count
  // and length): the split with the fewest float64 instructions on the critical
  // path, the segments' sum included
  short* segs = reinterpret_cast<short*>(lam);   // the eigenvalues come later
  for (int m = tid + 1; m < S; m += nt) {
    int best = 1 | (m << 4), cost = 1 << 30;
    for (int g = 1; g <= kSeg; ++g) {
      if (g > 1 && g * m > nt - 32) break;
      const int len = (m + g - 1) / g;
      const int c = ((g * m + 127) >> 7) * len + g;
      if (c < cost) { cost = c; best = g | (len << 4); }
    }
    segs[m] = static_cast<short>(best);
  }

  // reflector of column j from its m entries below the diagonal: x is entry idx,
  // held by the threads of the first nw warps (0 outside 0 <= idx < m)
  auto reflector = [&](int j, int m, int idx, int nw, double x, double* u) {
    double sig = warp_sum_int(x * x);
    if (idx == 0) scal[0] = x;
    if (nw > 1) {
      if (lane == 0) red[warp] = sig;
      asm volatile("bar.sync 1, %0;" ::"r"(32 * nw) : "memory");
      sig = red[0];
      for (int w = 1; w < nw; ++w) sig += red[w];
    } else {
      __syncwarp();
    }
    const double x0 = scal[0];
    // a column that is zero to rounding keeps its first entry (H = I)
    const bool skip = mag_bits(sig) < mag_bits(1e-300);
    const double nx = skip ? 0.0 : sqrt_fast(sig);
    const double al = skip ? x0 : -copysign(nx, x0);
    if (idx >= 0 && idx < m) {
      const double ui = skip ? 0.0 : (idx == 0 ? x0 - al : x);
      u[idx] = ui;
      a[tri(j + 1 + idx, j)] = ui;
    }
    if (idx == 0) {
      e[j] = al;
      scal[1] = skip ? 0.0 : fma(fabs(x0), nx, sig);   // 1 / beta
    }
  };
  if (S > 2 && warp < (S + 30) / 32)
    reflector(0, S - 1, tid, (S + 30) / 32, tid < S - 1 ? a[tri(1 + tid, 0)] : 0.0, vb);
  __syncthreads();
  for (int j = 0; j + 2 < S; ++j) {
    const int r0 = j + 1, m = S - r0, nw = (m + 31) >> 5;
    const double* v = vb + (j & 1) * S;
    // B u, B symmetric and held as its lower triangle (B[i][l] read from row
    // max(i, l)), split over nseg row segments; the last warp forms beta
    const int nseg = segs[m] & 15, len = segs[m] >> 4;
    const float rm = __fdividef(1.0f, static_cast<float>(m));
    if (warp == nwarp - 1 && lane == 0) {
      const double q = scal[1];
      const double b = mag_bits(q) ? rcp_full(q) : 0.0;
      scal[2] = b;
      scal[3] = 0.5 * b;
      beta[j] = b;
    }
    for (int q = tid; q < nseg * m; q += nt) {
      const int g = static_cast<int>((static_cast<float>(q) + 0.5f) * rm), i = q - g * m;
      const int l0 = g * len, l1 = min(m, l0 + len);
      double acc = 0.0;
      int at = l0 <= i ? tri(r0 + i, r0 + l0) : tri(r0 + l0, r0 + i);
      for (int l = l0; l < l1; ++l) {
        acc = fma(a[at], v[l], acc);
        at += l < i ? 1 : r0 + l + 1;
      }
      ps[g * m + i] = acc;
    }
    __syncthreads();
    double ui = 0.0, wi = 0.0;
    if (warp < nw) {
      if (tid < m) {
        for (int g = 0; g < nseg; ++g) wi += ps[g * m + tid];
        wi *= scal[2];
        ui = v[tid];
      }
      double K = warp_sum_int(ui * wi);
      if (nw > 1) {
        if (lane == 0) red[warp] = K;
        asm volatile("bar.sync 1, %0;" ::"r"(32 * nw) : "memory");
        K = red[0];
        for (int w = 1; w < nw; ++w) K += red[w];
      }
      wi = fma(-(K * scal[3]), ui, wi);      // w = beta B u - (beta / 2) (u . beta B u) u
      if (tid < m) p[tid] = wi;
    }
    __syncthreads();
    // rank-2 update B -= u w^T + w u^T of the lower triangle: column 0 and the
    // next reflector by the vector warps, the other columns by the rest
    if (warp < nw) {
      double x = 0.0;
      if (tid < m) {
        x = fma(-ui, p[0], fma(-wi, v[0], a[tri(r0 + tid, r0)]));
        if (tid == 0) d[r0] = x;
        a[tri(r0 + tid, r0)] = x;
        if (tid == 0) x = 0.0;               // the diagonal is not part of the column below it
      }
      if (j + 3 < S) reflector(r0, m - 1, tid - 1, nw, x, vb + ((j + 1) & 1) * S);
    }
    {
      // rows 1..m-1, columns 1..row, all lanes busy: rows i and m - i have m entries together
      const bool apart = nwarp > nw;
      const int nup = apart ? nt - 32 * nw : nt, t0 = apart ? tid - 32 * nw : tid;
      const int work = (m >> 1) * m;
      if (t0 >= 0)
        for (int q = t0; q < work; q += nup) {
          int pr = static_cast<int>((static_cast<float>(q) + 0.5f) * rm);
          int off = q - pr * m;
          if (off < 0) { --pr; off += m; }
          if (off >= m) { ++pr; off -= m; }
          const int ia = pr + 1, ib = m - ia;
          if (off >= ia && ia == ib) continue;       // the middle row of an even m
          const int i = off < ia ? ia : ib, l = off < ia ? off + 1 : off - ia + 1;
          double* at = a + tri(r0 + i, r0 + l);
          *at = fma(-v[i], p[l], fma(-p[i], v[l], *at));
        }
    }
    __syncthreads();
  }
  if (tid == 0) d[0] = a[0];
  if (tid == 0) {
    if (S >= 2) {
      d[S - 2] = a[tri(S - 2, S - 2)];
      e[S - 2] = a[tri(S - 1, S - 2)];
    }
    d[S - 1] = a[tri(S - 1, S - 1)];
  }
  __syncthreads();
  for (int i = tid; i < S; i += nt) {
    df[i] = static_cast<float>(d[i]);
    e2f[i] = (i + 1 < S) ? static_cast<float>(e[i] * e[i]) : 0.0f;
  }
  __syncthreads();

  // 2. float32 multisection: one warp per eigenvalue, 32 Sturm counts per
  //    round, to about 2e-7 of |T| (inverse iteration refines it)
  // Gershgorin bracket and scale, warp 0
  if (warp == 0) {
    double lo = 1e300, hi = -1e300, emax2 = 0.0;
    for (int i = lane; i < S; i += 32) {
      const double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i + 1 < S ? fabs(e[i]) : 0.0);
      lo = fmin(lo, d[i] - r);
      hi = fmax(hi, d[i] + r);
      if (i + 1 < S) emax2 = fmax(emax2, e[i] * e[i]);
    }
    for (int o = 16; o > 0; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      emax2 = fmax(emax2, __shfl_xor_sync(0xffffffffu, emax2, o));
    }
    if (lane == 0) {
      scal[3] = lo;
      scal[4] = hi;
      scal[5] = zero ? 1.0 : fmax(fmax(fabs(lo), fabs(hi)), 1e-300);   // any scale serves a zero matrix
      scal[6] = fmax(1e-30 * fmax(emax2, 1.0), 1e-30 * scal[5]);
    }
  }
  __syncthreads();
  const double lo = scal[3], hi = scal[4], tnorm = scal[5];
  const float pivmin = static_cast<float>(scal[6]);
  for (int t = warp; t < k; t += nwarp) {
    const float span = static_cast<float>(hi - lo);
    float a0 = static_cast<float>(lo) - 1e-6f * span - 1e-30f, b0 = static_cast<float>(hi) + 1e-6f * span + 1e-30f;
    const float tolf = 2e-7f * static_cast<float>(tnorm);
    for (int round = 0; round < 16 && (b0 - a0) > tolf; ++round) {
      const float x = a0 + (b0 - a0) * (static_cast<float>(lane + 1) / 33.0f);
      const bool above = sturm_count_f(S, df, e2f, x, pivmin) > t;
      const unsigned mask = __ballot_sync(0xffffffffu, above);
      const int f = mask ? __ffs(mask) - 1 : 32;
      const float xf = __shfl_sync(0xffffffffu, x, f < 32 ? f : 31);
      const float xl = __shfl_sync(0xffffffffu, x, f > 0 ? f - 1 : 0);
      const float na = f > 0 ? xl : a0;
      const float nb = f < 32 ? xf : b0;
      if (!(nb > na) || (na == a0 && nb == b0)) break;
      a0 = na;
      b0 = nb;
    }
    if (lane == 0) lam[t] = 0.5 * (static_cast<double>(a0) + static_cast<double>(b0));
  }
  __syncthreads();
  // clusters: eigenvalues closer than the float32 values can tell; a cluster of several
  // takes in what lies within 1e-4 |T| of it, whose float32 solves would let in too much
  // of the cluster (at 1e-5 |T|: residuals of 4e-13 |T|)
  if (tid == 0) {
    cl[0] = 0;
    for (int t = 1; t < k; ++t) cl[t] = lam[t] - lam[t - 1] < 2e-6 * tnorm ? cl[t - 1] : t;
    for (int t = 1; t < k; ++t) {
      if (cl[t] != t || !(lam[t] - lam[t - 1] < 1e-4 * tnorm)) continue;
      if (cl[t - 1] == t - 1 && (t + 1 == k || cl[t + 1] != t)) continue;   // one beside one
      for (int u = t; u < k && (u == t || cl[u] == t); ++u) cl[u] = cl[t - 1];
    }
  }
  __syncthreads();

  // 3. float64 inverse iteration, one thread per cluster (an isolated
  //    eigenvalue is a cluster of one) -> columns of Zw.  Inside a cluster the
  //    members are found in order, each solve followed by Gram-Schmidt against
  //    the members already found: independent iterations of a nearly
  //    degenerate pair converge to nearly the same vector, and orthogonalising
  //    them afterwards would magnify their error outside the cluster by the
  //    inverse of the angle between them.
  const double tiny = 0x1p-56 * tnorm;   // below the rounding of T
  auto orth_against = [&](double* y, int c0, int u) {   // y -= sum_{c0 <= v < u} (z_v . y) z_v, then normalise
    for (int v = c0; v < u; ++v) {
      const double* z = Zw + v;
      double dot = 0.0;
      for (int i = 0; i < S; ++i) dot = fma(z[(long long)i * k], y[(long long)i * k], dot);
      for (int i = 0; i < S; ++i) y[(long long)i * k] = fma(-dot, z[(long long)i * k], y[(long long)i * k]);
    }
    double nrm = 0.0;
    for (int i = 0; i < S; ++i) nrm = fma(y[(long long)i * k], y[(long long)i * k], nrm);
    const double inv = nrm > 0.0 ? 1.0 / sqrt(nrm) : 0.0;
    for (int i = 0; i < S; ++i) y[(long long)i * k] *= inv;
  };
  auto isolated = [&](int t) { return cl[t] == t && (t + 1 == k || cl[t + 1] != t); };
  // isolated eigenvalues, a thread each in step: two float32 solves with the
  // float32 shift leave an error of about 1e-7 |T| / gap in the vector and its
  // square in the Rayleigh quotient; two float64 solves with that shift (one
  // factorisation) raise it to the fifth power.  Norms and quotients by a warp
  // per vector in between.
  auto normalise = [&]() {
    for (int t = warp; t < k; t += nwarp) {
      if (!isolated(t)) continue;
      double* y = Zw + t;
      double nn = 0.0, rq = 0.0;
      for (int i = lane; i < S; i += 32) {
        const double yi = y[(long long)i * k];
        double ty = d[i] * yi;
        if (i > 0) ty = fma(e[i - 1], y[(long long)(i - 1) * k], ty);
        if (i + 1 < S) ty = fma(e[i], y[(long long)(i + 1) * k], ty);
        nn = fma(yi, yi, nn);
        rq = fma(yi, ty, rq);
      }
      nn = warp_sum_int(nn);
      rq = warp_sum_int(rq);
      // a vector that overflowed or vanished: its eigenvalue keeps its shift and is
      // solved again below, in float64 and normalised after every solve
      if (!(mag_bits(nn) > 0 && mag_bits(nn) < mag_bits(1e300) && mag_bits(rq) < mag_bits(1e300))) {
        if (lane == 0) cl[t] = -1 - t;
        continue;
      }
      const double inv = rsqrt_full(nn);
      for (int i = lane; i < S; i += 32) y[(long long)i * k] *= inv;
      if (lane == 0) lam[t] = rq * rcp_full(nn);
    }
    __syncthreads();
  };
  {
    // float32 solves: the tridiagonal in vb, factors and vectors in lu
    float* ef = reinterpret_cast<float*>(vb);
    float* luf = reinterpret_cast<float*>(lu);
    float* yf = luf + (size_t)5 * S * k;
    for (int i = tid; i + 1 < S; i += nt) ef[i] = static_cast<float>(e[i]);
    for (int q = tid; q < S * k; q += nt) {
      const int i = q / k, t = q - i * k;
      yf[q] = 1.0f + 0.01f * ((i * 7 + t * 3) % 11);
    }
    __syncthreads();
    const float tinyf = 1e-8f * static_cast<float>(tnorm);
    for (int t = tid; t < k; t += nt)
      if (isolated(t)) inverse_step_f(S, df, ef, static_cast<float>(lam[t]), tinyf, luf + t, yf + t, k);
    __syncthreads();
    for (int q = tid; q < S * k; q += nt) Zw[q] = static_cast<double>(yf[q]);
    __syncthreads();
  }
  normalise();
  for (int t = tid; t < k; t += nt) {
    if (!isolated(t)) continue;
    inverse_step(S, d, e, lam[t], tiny, true, lu + t, Zw + t, k, true);
    inverse_step(S, d, e, lam[t], tiny, false, lu + t, Zw + t, k, true);
  }
  __syncthreads();
  normalise();
  // clusters, a thread each, and the vectors given up above
  for (int c0 = tid; c0 < k; c0 += nt) {
    if (cl[c0] != -1 - c0 && (cl[c0] != c0 || isolated(c0))) continue;
    int c1 = c0 + 1;
    while (c1 < k && cl[c1] == c0) ++c1;
    for (int t = c0; t < c1; ++t) {
      double* y = Zw + t;
      double* lut = lu + t;
      // start vectors of their own (a scrambled index): members started alike differ by
      // little once the earlier ones are taken out, and what is left of other
      // eigenvectors weighs the more
      for (int i = 0; i < S; ++i) {
        unsigned r = static_cast<unsigned>(i) * 2654435761u + static_cast<unsigned>(t + 1) * 2246822519u;
        r = (r ^ (r >> 15)) * 3266489917u;
        r ^= r >> 13;
        y[(long long)i * k] = static_cast<double>(static_cast<int>(r)) * 0x1p-31;
      }
      inverse_step(S, d, e, lam[t], tiny, true, lut, y, k);
      orth_against(y, c0, t);
      inverse_step(S, d, e, lam[t], tiny, false, lut, y, k);
      orth_against(y, c0, t);
      // the shift is off by 2e-7 |T|, which leaves neighbouring eigenvectors in y at
      // its square over the gap's; two solves shifted by the Rayleigh quotient take
      // that to the third power each
      for (int pass = 0; pass < 2; ++pass) {
        const double rq = rayleigh(S, d, e, y, k);
        inverse_step(S, d, e, rq, tiny, true, lut, y, k);
        orth_against(y, c0, t);
      }
      // that close to a degenerate eigenvalue the members found before grow at rates of
      // their own, and taking them out magnifies the rounding outside the cluster: the
      // float32 shift treats them alike
      inverse_step(S, d, e, lam[t], tiny, true, lut, y, k);
      orth_against(y, c0, t);
    }
    for (int t = c0; t < c1; ++t) lam[t] = rayleigh(S, d, e, Zw + t, k);
  }
  __syncthreads();
  // clusters: Gram-Schmidt inside each, then (up to kMaxRR members) a
  // Rayleigh-Ritz rotation; warp 0, lanes over rows
  if (warp == 0) {
    int c0 = 0;
    while (c0 < k) {
      int c1 = c0 + 1;
      while (c1 < k && cl[c1] == c0) ++c1;
      if (c1 - c0 > 1) {
        for (int t = c0; t < c1; ++t) {
          for (int u = c0; u < t; ++u) {
            double dot = 0.0;
            for (int i = lane; i < S; i += 32) dot = fma(Zw[i * k + t], Zw[i * k + u], dot);
            dot = warp_sum(dot);
            for (int i = lane; i < S; i += 32) Zw[i * k + t] -= dot * Zw[i * k + u];
          }
          double nn = 0.0;
          for (int i = lane; i < S; i += 32) nn = fma(Zw[i * k + t], Zw[i * k + t], nn);
          nn = warp_sum(nn);
          const double inv = 1.0 / sqrt(nn);
          for (int i = lane; i < S; i += 32) Zw[i * k + t] *= inv;
          __syncwarp();
        }
        const int c = c1 - c0;
        if (c <= kMaxRR) {
          // H = Yc^T T Yc, (T y)_i = e_{i-1} y_{i-1} + d_i y_i + e_i y_{i+1}
          double H[kMaxRR][kMaxRR], Rr[kMaxRR][kMaxRR];
          for (int aa = 0; aa < c; ++aa)
            for (int bb = aa; bb < c; ++bb) {
              double h = 0.0;
              for (int i = lane; i < S; i += 32) {
                const double* yb = Zw + c0 + bb;
                double ty = d[i] * yb[i * k];
                if (i > 0) ty = fma(e[i - 1], yb[(i - 1) * k], ty);
                if (i + 1 < S) ty = fma(e[i], yb[(i + 1) * k], ty);
                h = fma(Zw[i * k + c0 + aa], ty, h);
              }
              h = warp_sum(h);
              H[aa][bb] = h;
              H[bb][aa] = h;
            }
          jacobi_small(c, H, Rr);   // every lane, same result
          __syncwarp();
          for (int i = lane; i < S; i += 32) {
            double yrow[kMaxRR];
            for (int aa = 0; aa < c; ++aa) yrow[aa] = Zw[i * k + c0 + aa];
            for (int bb = 0; bb < c; ++bb) {
              double z = 0.0;
              for (int aa = 0; aa < c; ++aa) z = fma(yrow[aa], Rr[aa][bb], z);
              Zw[i * k + c0 + bb] = z;
            }
          }
          if (lane == 0)
            for (int aa = 0; aa < c; ++aa) lam[c0 + aa] = H[aa][aa];
        } else {
          __syncwarp();
          for (int t = c0; t < c1; ++t) {
            const double r = rayleigh(S, d, e, Zw + t, k);   // identical in every lane
            if (lane == 0) lam[t] = r;
          }
        }
        __syncwarp();
      }
      c0 = c1;
    }
  }
  __syncthreads();
  // 4. Back-transformation z = H_0 ... H_{S-3} y in blocks of kWy reflectors,
  // H_jb ... H_jb+7 = I - U T U^T (T upper triangular): the dot products of a
  // block are independent, so the cross-thread sums come once per block instead
  // of once per reflector.
  const int nref = S > 2 ? S - 2 : 0, nblk = (nref + kWy - 1) / kWy;
  double* T = vb;                            // nblk x 64 (vb, p and ps are free now)
  auto refl = [&](int i, int jb, int r) { return i > jb + r && jb + r < nref ? a[tri(i, jb + r)] : 0.0; };
  for (int b = warp; b < nblk; b += nwarp) {
    const int jb = b * kWy;
    double* Tb = T + b * 64;
    // strictly upper part: u_q . u_r for q < r, one lane each
    int r = 1;
    while (r * (r + 1) / 2 <= lane) ++r;     // lane = r (r - 1) / 2 + q
    const int q = lane - r * (r - 1) / 2;
    double g = 0.0;
    if (r < kWy)
      for (int i = jb + r + 1; i < S; ++i) g = fma(refl(i, jb, q), refl(i, jb, r), g);
    if (r < kWy) Tb[q * kWy + r] = g;
    __syncwarp();
    for (int c = 0; c < kWy; ++c) {
      const double bc = jb + c < nref ? beta[jb + c] : 0.0;
      double t = 0.0;
      if (lane < c) {
        for (int w = lane; w < c; ++w) t = fma(Tb[lane * kWy + w], Tb[w * kWy + c], t);
        t *= -bc;
      }
      __syncwarp();
      if (lane < c) Tb[lane * kWy + c] = t;
      if (lane == c) Tb[c * kWy + c] = bc;
      __syncwarp();
    }
  }
  const int tg = (k + 3) / 4;                // groups of four vectors
  const int nsg = max(1, min(nwarp / tg, 5 * S / kWy));
  double* P = lu;                            // nsg x kWy x k partial dot products
  double* sv = lu + (size_t)5 * S * k;       // kWy x k: U^T z, then T U^T z after it
  double* yv = sv + kWy * k;
  const float rk = 1.0f / static_cast<float>(k);
  auto div_k = [&](int q) {                  // q / k (q < 2^20)
    int g = static_cast<int>((static_cast<float>(q) + 0.5f) * rk);
    if (g * k > q) --g;
    return g;
  };
  __syncthreads();
  for (int b = nblk - 1; b >= 0; --b) {
    const int jb = b * kWy, i0 = jb + 1, rows = S - i0;
    const int len = (rows + nsg - 1) / nsg;
    for (int w = warp; w < tg * nsg; w += nwarp) {
      const int sg = w / tg, r = lane & 7, t = (w - sg * tg) * 4 + (lane >> 3);
      const int i1 = min(S, i0 + (sg + 1) * len);
      double acc = 0.0;
      if (t < k && jb + r < nref) {
        const int ib = max(i0 + sg * len, jb + r + 1);
        int at = tri(ib, jb + r);
        for (int i = ib; i < i1; ++i) {
          acc = fma(a[at], Zw[i * k + t], acc);
          at += i + 1;
        }
      }
      if (t < k) P[(sg * kWy + r) * k + t] = acc;
    }
    __syncthreads();
    for (int q = tid; q < kWy * k; q += nt) {
      double t = P[q];
      for (int sg = 1; sg < nsg; ++sg) t += P[sg * kWy * k + q];
      sv[q] = t;
    }
    __syncthreads();
    for (int q = tid; q < kWy * k; q += nt) {
      const int r = div_k(q), t = q - r * k;
      double y = 0.0;
      for (int w = r; w < kWy; ++w) y = fma(T[b * 64 + r * kWy + w], sv[w * k + t], y);
      yv[q] = y;
    }
    __syncthreads();
    for (int q = tid; q < rows * k; q += nt) {
      const int g = div_k(q), i = i0 + g, t = q - g * k;
      const int nr = min(min(kWy, nref - jb), g + 1);     // reflectors that reach row i
      const double* u = a + tri(i, jb);
      double z = Zw[i0 * k + q];
      for (int r = 0; r < nr; ++r) z = fma(-u[r], yv[r * k + t], z);
      Zw[i0 * k + q] = z;
    }
    __syncthreads();
  }
  for (int q = tid; q < S * k; q += nt) Z[(long long)(q / k) * ldz + q % k] = Zw[q];
  for (int t = tid; t < k; t += nt) wout[t] = scale ? scalbn(lam[t], scale) : lam[t];
  if (tid == 0 && info) *info = 0;
}

// a = L L^T (lower L, in place, lda), flag[0] = 1 when a pivot is not positive
// Right-looking Cholesky on the lower triangle, one CTA: the triangle staged
// packed in shared memory when it fits, the column scaled by one reciprocal
// per step, the trailing update one warp per row.
constexpr int kCholSmemMax = 224;

template <bool SMEM>
__device__ void cholesky_body(int S, double* A, int lda, int* flag) {
  extern __shared__ double sh[];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int warp = tid >> 5, lane = tid & 31, nwarp = nt >> 5;
  // element (i, l), l <= i: packed in shared memory, else in place in A
  auto at = [&](int i, int l) -> double& { return SMEM ? sh[tri(i, l)] : A[(long long)i * lda + l]; };
  if (SMEM) {
    for (int i = warp; i < S; i += nwarp)
      for (int l = lane; l <= i; l += 32) sh[tri(i, l)] = A[(long long)i * lda + l];
  }
  __syncthreads();
  for (int j = 0; j < S; ++j) {
    const int m = S - 1 - j;                 // rows below the pivot
    // the warps that scale the column each form 1 / sqrt(pivot) from a float32
    // estimate (sqrt and divide took 1100 cycles on one thread)
    double x = at(j, j);
    const long long xb = __double_as_longlong(x);
    const bool bad = xb <= 0 || xb > 0x7FF0000000000000ll;   // not positive, or NaN
    if (bad) x = 1e-300;
    const double r = 32 * warp < max(m, 1) ? rsqrt_full(x) : 0.0;
    for (int i = tid; i < m; i += nt) at(j + 1 + i, j) *= r;
    __syncthreads();
    if (tid == 0) {
      if (bad) *flag = 1;
      at(j, j) = x * r;
    }
    // trailing update, all lanes busy: rows i and m - 1 - i of the triangle have m + 1 entries together
    const float rm = 1.0f / static_cast<float>(m + 1);
    const int work = ((m + 1) >> 1) * (m + 1);
    for (int q = tid; q < work; q += nt) {
      int pr = static_cast<int>((static_cast<float>(q) + 0.5f) * rm);
      int off = q - pr * (m + 1);
      if (off < 0) { --pr; off += m + 1; }
      if (off > m) { ++pr; off -= m + 1; }
      const int ib = m - 1 - pr;
      if (off > pr && pr == ib) continue;    // the middle row of an odd m
      const int i = off <= pr ? pr : ib, l = off <= pr ? off : off - pr - 1;
      double& c = at(j + 1 + i, j + 1 + l);
      c = fma(-at(j + 1 + i, j), at(j + 1 + l, j), c);
    }
    __syncthreads();
  }
  for (int idx = tid; idx < S * S; idx += nt) {
    const int i = idx / S, l = idx % S;
    if (l > i) A[(long long)i * lda + l] = 0.0;
    else if (SMEM) A[(long long)i * lda + l] = sh[tri(i, l)];
  }
}


}  // namespace
}  // namespace xs
