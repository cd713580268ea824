// G(R) build of libxs: the NDDO two-electron contraction of the A*X product.
//
// Paper, Section "GPU Implementation", Eq. ftilde:
//   Ft_{mu nu} = sum_{lam sig} [(mu nu|lam sig) - (mu lam|nu sig)] R_{lam sig},
// with NDDO leaving Coulomb on the diagonal atom blocks (symmetrised R) and
// exchange everywhere, contracted with the symmetric and antisymmetric parts
// of R.  With J(R) = sum (mu nu|lam sig) R and K(R) = sum (mu lam|nu sig) R the
// singlet products need (spin adaptation, see xs.h):
//   CIS (and the Fock build at P = D/2):  G  = 2 J(R) - K(R)
//   TDHF:                                 G+ = 4 J(Rs) - 2 K(Rs) = 4 J(R) - K(R) - K(R^T)
//                                         G- = -2 K(Ra)          = -K(R) + K(R^T)
//
// Float32 builds run over super-atom pairs (gpair.cu).  Float64 builds, here, are
// bound by the float64 pipe (two multiply-adds per clock and SM), so both steps
// form no product twice:
//   1. two-centre Coulomb J2 = W r of the dense product supermatrix W with the
//      product vectors r_B[q] of the diagonal atom blocks (R_ls + R_sl for l < s,
//      R_ll on the diagonal), with exactly nvec columns;
//   2. atom-aligned tiles of G (one row group x one column tile per CTA, the
//      tile's pair-integral block staged once in shared memory, the nvec
//      matrices streamed through it): diagonal atom blocks combine J2 with the
//      closed-form one-centre Coulomb/exchange; off-diagonal blocks hold the
//      two-centre exchange sum_{nu in A, sig in B} (mu nu|lam sig) R_{nu sig}.
//      The TDHF outputs contract R + R^T (G+, symmetric) and R - R^T (G-,
//      antisymmetric), so only the blocks A < B are contracted and the others
//      are written as their (negated) transposes: 8 multiply-adds per element of
//      heavy atoms and output, a quarter of the 32 that K(R) and K(R^T) in every
//      block took.
#include <vector>

#include "kernels.h"
#include "model.h"
#include "prof.h"
#include "gbuild_dev.cuh"

namespace xs {

namespace {

// outputs of the TDHF modes to form (template parameter OUT)
constexpr int kPlusOnly = 1, kMinusOnly = 2, kBoth = 3;

// Atom-aligned tiles of G: a CTA owns one row group (a heavy atom's 4 AOs, or
// up to 4 consecutive hydrogens) and one column tile (whole atoms, at most 64
// AOs).  It stages the pair-integral block W[products of the rows' atoms]
// [products of the columns' atoms] in shared memory once and then streams the
// nvec matrices: per matrix, R's tile (and for TDHF its transpose tile) goes
// through shared memory, the next one loading meanwhile, and every thread forms
// one element.  G+ of 4 matrices at 2200 AOs 854 -> 314 us
// (float64 pipe alone: 215); CIS builds (nonsymmetric R, 16 multiply-adds an
// element) take 150 us for 4 matrices at 1233 AOs, the pipe's 112.
template <GMode MODE, int OUT>
__global__ void __launch_bounds__(256, 4) gtile_kernel(int n, int np, int nvec, const int4* __restrict__ rows,
                                                       const int4* __restrict__ cols, const int* __restrict__ ao_atom,
                                                       const int* __restrict__ ao_local,
                                                       const int* __restrict__ atom_ao_off,
                                                       const int* __restrict__ atom_nao,
                                                       const int* __restrict__ atom_prod_off,
                                                       const int* __restrict__ atom_elem,
                                                       const double* __restrict__ par, const double* __restrict__ W,
                                                       const double* __restrict__ J2, int njc,
                                                       const double* __restrict__ R, double* __restrict__ G,
                                                       double* __restrict__ Gm) {
  constexpr bool kRpa = MODE == G_RPA || MODE == G_RPA_T;        // G+ and G- outputs, R^T tiles
  constexpr bool kTriplet = MODE == G_CIS_T || MODE == G_RPA_T;  // no Coulomb terms
  constexpr bool kPlus = !kRpa || (OUT & kPlusOnly), kMinus = kRpa && (OUT & kMinusOnly);
  // tiles padded by 4 rows / columns of zeros: a hydrogen's block is handled as
  // a 4 x 4 block with zero weights past its single AO
  __shared__ double Ws[kGP][kGQ + 1];
  __shared__ double Rt[2][kGR + 4][kGC + 4];       // R (TDHF uses the first; CIS alternates)
  __shared__ double Rtt[kRpa ? kGC : 1][kGR + 1];  // R^T
  __shared__ double Rs[kPlus && kRpa ? kGR + 4 : 1][kGC + 4], Ra[kMinus ? kGR + 4 : 1][kGC + 4];   // R +- R^T
  __shared__ double Gs[kPlus && kRpa ? kGC : 1][kGR + 1], Ms[kMinus ? kGC : 1][kGR + 1];           // mirrored blocks
  const int4 rg = rows[blockIdx.y], ct = cols[blockIdx.x];
  if (kRpa && ct.w <= rg.z) return;                // every block of the tile is a mirror image
  const int ra = rg.x, nr = rg.y, cb = ct.x, nc = ct.y;
  const int PA0 = atom_prod_off[rg.z], PB0 = atom_prod_off[ct.z];
  const int nPA = atom_prod_off[rg.w - 1] + (atom_nao[rg.w - 1] == 4 ? 10 : 1) - PA0;
  const int nPB = atom_prod_off[ct.w - 1] + (atom_nao[ct.w - 1] == 4 ? 10 : 1) - PB0;
  const int tid = threadIdx.x;
  // one warp per pair-integral row, lanes along the row (no integer division)
  for (int pr = tid >> 5; pr < nPA; pr += blockDim.x >> 5)
    for (int pc = tid & 31; pc < nPB; pc += 32) Ws[pr][pc] = W[(long long)(PA0 + pr) * np + PB0 + pc];
  for (int idx = tid; idx < 2 * (kGR + 4) * (kGC + 4); idx += blockDim.x) (&Rt[0][0][0])[idx] = 0.0;
  if constexpr (kPlus && kRpa)
    for (int idx = tid; idx < (kGR + 4) * (kGC + 4); idx += blockDim.x) (&Rs[0][0])[idx] = 0.0;
  if constexpr (kMinus)
    for (int idx = tid; idx < (kGR + 4) * (kGC + 4); idx += blockDim.x) (&Ra[0][0])[idx] = 0.0;
  const int ri = tid / kGC, ci = tid % kGC;
  const bool active = ri < nr && ci < nc;
  const int mu = ra + ri, lam = cb + ci;
  int A = 0, B = 0, a = 0, b = 0, nA = 1, nB = 1, rA = 0, cA = 0, rB = 0, pA = 0, pB = 0, PA = 0;
  const double* pd = par;   // the diagonal block's element parameters (read where used)
  if (active) {
    A = ao_atom[mu]; B = ao_atom[lam];
    a = ao_local[mu]; b = ao_local[lam];
    nA = atom_nao[A]; nB = atom_nao[B];
    rA = atom_ao_off[A] - ra;          // A's first row in the tile
    cA = atom_ao_off[A] - cb;          // A's first column (diagonal block)
    rB = atom_ao_off[B] - cb;          // B's first column in the tile
    PA = atom_prod_off[A];
    pA = PA - PA0;
    pB = atom_prod_off[B] - PB0;
    if (A == B) pd = par + atom_elem[A] * XS_NPARAM;
  }
  const bool form = active && (!kRpa || B >= A);
  __syncthreads();
  // this output's 16 exchange weights (mu nu|lam sig) for nu in A, sig in B,
  // zero past a hydrogen's single AO; independent of the matrix index
  double wv[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) wv[q] = 0.0;
  if (form && A != B) {
#pragma unroll
    for (int nu = 0; nu < 4; ++nu)
#pragma unroll
      for (int sg = 0; sg < 4; ++sg)
        if (nu < nA && sg < nB)
          wv[nu * 4 + sg] = Ws[pA + ((nA == 4) ? pidx(a, nu) : 0)][pB + ((nB == 4) ? pidx(b, sg) : 0)];
  }
  const int tr = tid % kGR, tc = tid / kGR;   // transposed tile: 4 consecutive threads per row
  const bool tact = kRpa && tr < nr && tc < nc;
  const bool mirror = tact && ao_atom[cb + tc] > ao_atom[ra + tr];
  const long long nn = (long long)n * n;
  const long long at_r = (long long)mu * n + lam, at_t = (long long)(cb + tc) * n + ra + tr;
  // K of one atom block: sum over the block's nonzero weights (a hydrogen has
  // one AO; warps are nearly always uniform in the atom kinds, heavy atoms
  // preceding hydrogens in the AO order of the generated molecules)
  auto exchange = [&](const double (*X)[kGC + 4]) {
    double kr = 0.0;
    if (nA == 4 && nB == 4) {
#pragma unroll
      for (int nu = 0; nu < 4; ++nu)
#pragma unroll
        for (int sg = 0; sg < 4; ++sg) kr = fma(wv[nu * 4 + sg], X[rA + nu][rB + sg], kr);
    } else if (nA == 4) {
#pragma unroll
      for (int nu = 0; nu < 4; ++nu) kr = fma(wv[nu * 4], X[rA + nu][rB], kr);
    } else if (nB == 4) {
#pragma unroll
      for (int sg = 0; sg < 4; ++sg) kr = fma(wv[sg], X[rA][rB + sg], kr);
    } else {
      kr = wv[0] * X[rA][rB];
    }
    return kr;
  };
  double nxt = active ? R[at_r] : 0.0, nxtt = tact ? R[at_t] : 0.0;
  int buf = 0;
  for (int v = 0; v < nvec; ++v) {
    if (active) Rt[buf][ri][ci] = nxt;
    if (tact) Rtt[tc][tr] = nxtt;
    if (v + 1 < nvec) {
      if (active) nxt = R[(v + 1) * nn + at_r];
      if (tact) nxtt = R[(v + 1) * nn + at_t];
    }
    __syncthreads();
    if constexpr (kRpa) {
      if (active) {
        const double x = Rt[0][ri][ci], y = Rtt[ci][ri];
        if constexpr (kPlus) Rs[ri][ci] = x + y;
        if constexpr (kMinus) Ra[ri][ci] = x - y;
      }
      __syncthreads();
    }
    if (form) {
      double g = 0.0, gm = 0.0;
      if (A == B) {
        double J1, K1ab, K1ba;
        if (nA == 1) {
          J1 = K1ab = K1ba = pd[4] * Rt[buf][rA][cA];
        } else {
          double Rd[16];
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) Rd[i * 4 + j] = Rt[buf][rA + i][cA + j];
          double p[XS_NPARAM];
#pragma unroll
          for (int i = 0; i < XS_NPARAM; ++i) p[i] = (i >= 4 && i <= 8) ? pd[i] : 0.0;
          one_centre<double>(p, a, b, Rd, J1, K1ab, K1ba);
        }
        if constexpr (kTriplet) {
          g = kRpa ? -(K1ab + K1ba) : -K1ab;
        } else if constexpr (kPlus) {
          const int pab = (nA == 4) ? pidx(a, b) : 0;
          double J = J1;
          for (int c = 0; c < njc; ++c) J += J2[((long long)c * np + PA + pab) * nvec + v];
          g = kRpa ? 4.0 * J - (K1ab + K1ba) : 2.0 * J - K1ab;
        }
        if constexpr (kMinus) gm = -(K1ab - K1ba);
      } else {
        if constexpr (!kRpa) g = -exchange(Rt[buf]);
        if constexpr (kRpa && kPlus) g = -exchange(Rs);
        if constexpr (kMinus) gm = -exchange(Ra);
      }
      if constexpr (kPlus) G[v * nn + at_r] = g;
      if constexpr (kMinus) Gm[v * nn + at_r] = gm;
      if constexpr (kRpa && kPlus) Gs[ci][ri] = g;
      if constexpr (kMinus) Ms[ci][ri] = -gm;
    }
    if constexpr (kRpa) {
      __syncthreads();
      if (mirror) {
        if constexpr (kPlus) G[v * nn + at_t] = Gs[tc][tr];
        if constexpr (kMinus) Gm[v * nn + at_t] = Ms[tc][tr];
      }
    } else {
      buf ^= 1;   // the other buffer was last read before this iteration's barrier
    }
  }
}

template <GMode MODE, int OUT>
void launch_mode(cudaStream_t s, const DevMol& m, const double* d_par, int nvec, const double* J2, int njc,
                 const double* R, double* G, double* Gm) {
  dim3 grid(m.gb_ncols, m.gb_nrows);
  const int4* rows = reinterpret_cast<const int4*>(m.gb_rows.get());
  const int4* cols = reinterpret_cast<const int4*>(m.gb_cols.get());
  gtile_kernel<MODE, OUT><<<grid, 256, 0, s>>>(m.n, m.np, nvec, rows, cols, m.ao_atom.get(), m.ao_local.get(),
                                               m.atom_ao_off.get(), m.atom_nao.get(), m.atom_prod_off.get(),
                                               m.atom_elem.get(), d_par, m.W.get(), J2, njc, R, G, Gm);
}

// J2: njc partial sums (np x nvec each) of the two-centre Coulomb
void launch_tiles(cudaStream_t s, const DevMol& m, const double* d_par, GMode mode, int nvec, const double* J2,
                  int njc, const double* R, double* G, double* Gm) {
#define XS_TILES(MODE, OUT) launch_mode<MODE, OUT>(s, m, d_par, nvec, J2, njc, R, G, Gm)
  if (mode == G_CIS) XS_TILES(G_CIS, kPlusOnly);
  else if (mode == G_CIS_T) XS_TILES(G_CIS_T, kPlusOnly);
  else if (!G) XS_TILES(G_RPA_T, kMinusOnly);   // G- = -K(R) + K(R^T) has no Coulomb part
  else if (mode == G_RPA && Gm) XS_TILES(G_RPA, kBoth);
  else if (mode == G_RPA) XS_TILES(G_RPA, kPlusOnly);
  else if (Gm) XS_TILES(G_RPA_T, kBoth);
  else XS_TILES(G_RPA_T, kPlusOnly);
#undef XS_TILES
  XS_CHECK_LAUNCH();
}

// Partial sums of J2 = W r over a chunk of rows of the symmetric W: threads along
// q (row segments of W), the chunk's r formed from R's diagonal blocks (prod: the
// two AOs of every on-atom product), NV vectors starting at v0 + NV blockIdx.z.
// Float64-pipe bound: np^2 NV multiply-adds, with no padded vectors.
template <int NV>
__global__ void __launch_bounds__(128) j2_f64_kernel(int n, int np, int nvec, int v0, int chunk,
                                                     const int2* __restrict__ prod, const double* __restrict__ W,
                                                     const double* __restrict__ R, double* __restrict__ part) {
  __shared__ double rs[128][NV];
  const int q = blockIdx.x * 128 + threadIdx.x;
  const int p0 = blockIdx.y * chunk, rows = min(chunk, np - p0);
  const int vb = v0 + NV * blockIdx.z;
  const long long nn = (long long)n * n;
  for (int idx = threadIdx.x; idx < rows * NV; idx += 128) {
    const int pr = idx / NV, v = idx - pr * NV;
    const int2 ao = prod[p0 + pr];
    const double* Rv = R + (vb + v) * nn;
    double x = Rv[(long long)ao.x * n + ao.y];
    if (ao.x != ao.y) x += Rv[(long long)ao.y * n + ao.x];
    rs[pr][v] = x;
  }
  __syncthreads();
  if (q >= np) return;
  double acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = 0.0;
  const double* w = W + (long long)p0 * np + q;
#pragma unroll 4
  for (int p = 0; p < rows; ++p) {
    const double x = __ldg(w + (long long)p * np);
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = fma(x, rs[p][v], acc[v]);
  }
  double* out = part + ((long long)blockIdx.y * np + q) * nvec + vb;
#pragma unroll
  for (int v = 0; v < NV; ++v) out[v] = acc[v];
}

__global__ void j2_f64_reduce_kernel(long long count, int nchunk, const double* __restrict__ part,
                                     double* __restrict__ J2) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  double s = 0.0;
  for (int c = 0; c < nchunk; ++c) s += part[c * count + i];
  J2[i] = s;
}

template <int NV>
void launch_j2(cudaStream_t s, const DevMol& m, int nvec, int v0, int groups, int chunk, int nchunk, const double* R,
               double* part) {
  j2_f64_kernel<NV><<<dim3((m.np + 127) / 128, nchunk, groups), 128, 0, s>>>(
      m.n, m.np, nvec, v0, chunk, reinterpret_cast<const int2*>(m.gb_prod.get()), m.W.get(), R, part);
  XS_CHECK_LAUNCH();
}

// rows of W per partial sum: 128 fill the device from 2048 products up; fewer for
// smaller molecules, whose W rows would otherwise be too few CTAs (the chain of a
// chunk is 64 cycles a row)
int j2_chunk(int np) { return np >= 2048 ? 128 : (np >= 512 ? 64 : 32); }
// partial sums that the tile kernel adds itself (above: a kernel of their own)
constexpr int kFusedPartials = 8;

// J2 of nvec matrices into ws; returns the number of partial sums at *J2.  4
// vectors at 4600 products 438 -> 159 us (a skinny GEMM padded to 8 vectors
// before; the pipe alone: 146), 1 vector at 691 products 41 -> 11 us.
int coulomb_j2_f64(cudaStream_t s, const DevMol& m, int nvec, const double* R, DevBuf<double>& ws, const double** J2) {
  const int np = m.np, chunk = j2_chunk(np), nchunk = (np + chunk - 1) / chunk;
  const size_t count = (size_t)np * nvec;
  ws.ensure((nchunk + 1) * count);
  double* part = ws.get() + count;
  ProfScope ps(s, "coulomb_j2_f64", 8.0 * ((double)np * np + 2.0 * count), 2.0 * (double)np * np * nvec);
  if (nvec >= 8) launch_j2<8>(s, m, nvec, 0, nvec / 8, chunk, nchunk, R, part);
  const int v0 = nvec / 8 * 8;
  switch (nvec - v0) {
    case 1: launch_j2<1>(s, m, nvec, v0, 1, chunk, nchunk, R, part); break;
    case 2: launch_j2<2>(s, m, nvec, v0, 1, chunk, nchunk, R, part); break;
    case 3: launch_j2<3>(s, m, nvec, v0, 1, chunk, nchunk, R, part); break;
    case 4: launch_j2<4>(s, m, nvec, v0, 1, chunk, nchunk, R, part); break;
    case 5: launch_j2<5>(s, m, nvec, v0, 1, chunk, nchunk, R, part); break;
    case 6: launch_j2<6>(s, m, nvec, v0, 1, chunk, nchunk, R, part); break;
    case 7: launch_j2<7>(s, m, nvec, v0, 1, chunk, nchunk, R, part); break;
    default: break;
  }
  if (nchunk <= kFusedPartials) {
    *J2 = part;
    return nchunk;
  }
  j2_f64_reduce_kernel<<<grid1((long long)count, 256), 256, 0, s>>>((long long)count, nchunk, part, ws.get());
  XS_CHECK_LAUNCH();
  *J2 = ws.get();
  return 1;
}

inline bool has_coulomb(GMode mode) { return mode == G_CIS || mode == G_RPA; }

// zero columns [n, ldo) of rows x ldo matrices (batch stride rows * ldo)
__global__ void zero_pad_cols_kernel(int rows, int n, int ldo, int nvec, float* a, float* b) {
  const int w = ldo - n;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)nvec * rows * w) return;
  const long long r = idx / w;
  const long long at = r * ldo + n + idx % w;
  a[at] = 0.0f;
  if (b) b[at] = 0.0f;
}

}  // namespace

template <>
void gbuild<float>(cudaStream_t s, const DevMol& m, const double* d_par, GMode mode, int nvec, const float* R, float* G,
                   float* Gm, DevBuf<float>& ws) {
  if (nvec <= 0) return;
  const int n = m.n, np = m.np;
  ws.ensure((size_t)2 * np * nvec);
  float* rT = ws.get();
  float* J2 = ws.get() + (size_t)np * nvec;
  const float* W = m.Wf.get();
  if (has_coulomb(mode) && G) {   // G- has no Coulomb part (J2 is then not formed, G not stored)
    dim3 block(8, 32);
    dim3 grid((m.L.natoms + 31) / 32);
    pack_diag_kernel<float><<<grid, block, 0, s>>>(m.L.natoms, n, np, nvec, m.atom_ao_off.get(), m.atom_nao.get(),
                                                   m.atom_prod_off.get(), R, rT);
    XS_CHECK_LAUNCH();
    static thread_local ThreadScratch<float> j2_ws;
    coulomb_j2(s, np, nvec, W, rT, J2, j2_ws.here());
  }
  // algorithmic traffic: read R, write G (and G-), read the pair integrals once
  const double outs = (G ? 1.0 : 0.0) + (Gm ? 1.0 : 0.0);
  ProfScope ps(s, "gbuild_assemble_f32", 4.0 * ((double)nvec * n * n * (1.0 + outs) + (double)np * np), 0.0);
  gpair_build(s, m, d_par, mode, nvec, W, J2, nvec, R, G, Gm);
}

template <>
void gbuild<double>(cudaStream_t s, const DevMol& m, const double* d_par, GMode mode, int nvec, const double* R,
                    double* G, double* Gm, DevBuf<double>& ws) {
  if (nvec <= 0) return;
  const double* J2 = nullptr;
  int njc = 0;
  if (has_coulomb(mode) && G) njc = coulomb_j2_f64(s, m, nvec, R, ws, &J2);   // G- has no Coulomb part
  const double outs = (G ? 1.0 : 0.0) + (Gm ? 1.0 : 0.0);
  ProfScope ps(s, "gbuild_assemble_f64", 8.0 * ((double)nvec * m.n * m.n * (1.0 + outs) + (double)m.np * m.np), 0.0);
  launch_tiles(s, m, d_par, mode, nvec, J2, njc, R, G, Gm);
}

void gbuild_split(cudaStream_t s, const DevMol& m, const double* d_par, GMode mode, int nvec, const float* R,
                  float* Gh, float* Gl, float* Gmh, float* Gml, int ldo, DevBuf<float>& ws) {
  if (nvec <= 0) return;
  const int n = m.n, np = m.np;
  if (ldo < n) throw Error(XS_EINVAL, "gbuild_split: row stride below n");
  ws.ensure((size_t)2 * np * nvec);
  float* rT = ws.get();
  float* J2 = ws.get() + (size_t)np * nvec;
  const float* W = m.Wf.get();
  const bool coulomb = has_coulomb(mode) && Gh;
  if (coulomb) {
    dim3 block(8, 32);
    dim3 grid((m.L.natoms + 31) / 32);
    pack_diag_kernel<float><<<grid, block, 0, s>>>(m.L.natoms, n, np, nvec, m.atom_ao_off.get(),
                                                          m.atom_nao.get(), m.atom_prod_off.get(), R, rT);
    XS_CHECK_LAUNCH();
    static thread_local ThreadScratch<float> j2_ws;
    coulomb_j2(s, np, nvec, W, rT, J2, j2_ws.here());
  }
  if (ldo > n) {
    const long long cnt = (long long)nvec * n * (ldo - n);
    if (Gh) zero_pad_cols_kernel<<<grid1(cnt, 256), 256, 0, s>>>(n, n, ldo, nvec, Gh, Gl);
    if (Gmh) zero_pad_cols_kernel<<<grid1(cnt, 256), 256, 0, s>>>(n, n, ldo, nvec, Gmh, Gml);
    XS_CHECK_LAUNCH();
  }
  // algorithmic traffic: read R, write the G (and G-) TF32 pairs, read the pair integrals once
  const double outs = (Gh ? 1.0 : 0.0) + (Gmh ? 1.0 : 0.0);
  ProfScope ps(s, "gbuild_assemble_f32", 4.0 * ((double)nvec * n * n * (1.0 + 2.0 * outs) + (double)np * np), 0.0);
  gpair_build_split(s, m, d_par, mode, nvec, W, J2, nvec, R, Gh, Gl, Gmh, Gml, ldo);
}

void gbuild_raw(cudaStream_t s, const DevMol& m, const double* d_par, GMode mode, int nvec, const double* R, double* G,
                double* Gm, double* r, double* J2) {
  if (nvec <= 0) return;
  const int n = m.n, np = m.np;
  {
    dim3 block(8, 32);
    dim3 grid((m.L.natoms + 31) / 32);
    pack_diag_kernel<double><<<grid, block, 0, s>>>(m.L.natoms, n, np, nvec, m.atom_ao_off.get(), m.atom_nao.get(),
                                                    m.atom_prod_off.get(), R, r);
    XS_CHECK_LAUNCH();
  }
  gemm<double>(s, false, false, np, nvec, np, 1.0, m.W.get(), np, 0, r, nvec, 0, 0.0, J2, nvec, 0, 1);
  launch_tiles(s, m, d_par, mode, nvec, J2, 1, R, G, Gm);
}

void build_gtiles(cudaStream_t s, DevMol& m) {
  const MolLayout& L = m.L;
  std::vector<int> rows, cols;   // per tile: first AO, AO count, first atom, end atom
  for (int A = 0; A < L.natoms;) {
    int A1 = A, cnt = 0;
    if (L.nao_atom[A] == 4) {
      A1 = A + 1;
      cnt = 4;
    } else {
      while (A1 < L.natoms && L.nao_atom[A1] == 1 && cnt < kGR) { ++A1; ++cnt; }
    }
    rows.insert(rows.end(), {L.ao_off[A], cnt, A, A1});
    A = A1;
  }
  for (int A = 0; A < L.natoms;) {
    int A1 = A, cnt = 0;
    while (A1 < L.natoms && cnt + L.nao_atom[A1] <= kGC) { cnt += L.nao_atom[A1]; ++A1; }
    cols.insert(cols.end(), {L.ao_off[A], cnt, A, A1});
    A = A1;
  }
  std::vector<int> prod;         // the two AOs of every on-atom product, in product order
  for (int A = 0; A < L.natoms; ++A)
    for (int a = 0; a < L.nao_atom[A]; ++a)
      for (int b = a; b < L.nao_atom[A]; ++b) prod.insert(prod.end(), {L.ao_off[A] + a, L.ao_off[A] + b});
  m.gb_prod.alloc(prod.size());
  XS_CUDA(cudaMemcpyAsync(m.gb_prod.get(), prod.data(), sizeof(int) * prod.size(), cudaMemcpyHostToDevice, s));
  m.gb_nrows = static_cast<int>(rows.size() / 4);
  m.gb_ncols = static_cast<int>(cols.size() / 4);
  m.gb_rows.alloc(rows.size());
  m.gb_cols.alloc(cols.size());
  XS_CUDA(cudaMemcpyAsync(m.gb_rows.get(), rows.data(), sizeof(int) * rows.size(), cudaMemcpyHostToDevice, s));
  XS_CUDA(cudaMemcpyAsync(m.gb_cols.get(), cols.data(), sizeof(int) * cols.size(), cudaMemcpyHostToDevice, s));
  XS_CUDA(cudaStreamSynchronize(s));
}

}  // namespace xs
