// The Davidson matrix-vector product of libxs (paper, Section "GPU
// Implementation", Eqs. cis_matrix_vector and ftilde):
//   (1) R_k = C_occ X_k C_vir^T                    (transition densities)
//   (2) G_k = G(R_k) over the atom-pair blocks      (gbuild.cu)
//   (3) Y_k = C_occ^T G_k C_vir + (eps_a - eps_i) X_k
// For TDHF one G build gives G+ and G- and two back-transforms give (A+B)X and
// (A-B)X.  The two transforms contract the smaller of nocc and nvir against
// n^2 last.  Batches of vectors share each GEMM (the vectors are stacked into
// one tall operand where the shared factor is on the right).  In float64 the
// transforms of all but small molecules are residue products on the tensor
// cores (modgemm.h; rule and figures at mg_applies), the others run on the
// float64 pipe.
#include <algorithm>

#include "kernels.h"
#include "modgemm.h"
#include "products.h"
#include "tc.h"

namespace xs {

namespace {

// R (nvec x n x n) from X (nvec x o x v); CT is the MO-major coefficient matrix.
template <typename T>
void pbuild(cudaStream_t s, int n, int o, int v, int nvec, const T* CT, const T* X, T* R, T* tmp) {
  const T* CTocc = CT;
  const T* CTvir = CT + (size_t)o * n;
  if (v <= o) {
    // T_k = C_occ X_k (n x v), then R = [T_1; ..; T_k] C_vir^T
    gemm<T>(s, true, false, n, v, o, T(1), CTocc, n, 0, X, v, (long long)o * v, T(0), tmp, v, (long long)n * v, nvec);
    gemm<T>(s, false, false, nvec * n, n, v, T(1), tmp, v, 0, CTvir, n, 0, T(0), R, n, 0, 1);
  } else {
    // U = [X_1; ..; X_k] C_vir^T (o x n each), then R_k = C_occ U_k
    gemm<T>(s, false, false, nvec * o, n, v, T(1), X, v, 0, CTvir, n, 0, T(0), tmp, n, 0, 1);
    gemm<T>(s, true, false, n, n, o, T(1), CTocc, n, 0, tmp, n, (long long)o * n, T(0), R, n, (long long)n * n, nvec);
  }
}

// Y (nvec x o x v) = C_occ^T G_k C_vir
template <typename T>
void backtransform(cudaStream_t s, int n, int o, int v, int nvec, const T* CT, const T* G, T* Y, T* tmp) {
  const T* CTocc = CT;
  const T* CTvir = CT + (size_t)o * n;
  if (v <= o) {
    // S = [G_1; ..; G_k] C_vir (n x v each), Y_k = C_occ^T S_k
    gemm<T>(s, false, true, nvec * n, v, n, T(1), G, n, 0, CTvir, n, 0, T(0), tmp, v, 0, 1);
    gemm<T>(s, false, false, o, v, n, T(1), CTocc, n, 0, tmp, v, (long long)n * v, T(0), Y, v, (long long)o * v, nvec);
  } else {
    // Q_k = C_occ^T G_k (o x n), Y = [Q_1; ..; Q_k] C_vir
    gemm<T>(s, false, false, o, n, n, T(1), CTocc, n, 0, G, n, (long long)n * n, T(0), tmp, n, (long long)o * n, nvec);
    gemm<T>(s, false, true, nvec * o, v, n, T(1), tmp, n, 0, CTvir, n, 0, T(0), Y, v, 0, 1);
  }
}

// Residue operands of the orbitals (modgemm.h), made on first use and kept with
// the molecule until its orbitals change, like the mixed path's TF32 pairs:
// C_occ (n x o) and C_vir (n x v) of the P build, C_vir^T (v x n) and C_occ^T
// (o x n) of the back-transform.
struct MgOrbitals {
  MgPlanes s_occ, s_vir, s_virT, s_occT;
  MgOperand occ, vir, virT, occT;
};

// bytes of residue planes (operands and result) that one context holds at most
// beyond a single vector's; larger batches run in chunks
constexpr double kMgBytes = 1.5e9;

// Where the residue products run: from 160 AOs up, and from 96 AOs up when the
// batch gives them work.  Four products cost the residue path 105-115 us in
// kernels whatever their size (16 launches) and the float64 pipe 55 us at 62
// AOs, so the line is where they meet; kernel time of the four products of A X,
// pipe -> residues: 62 AOs, 20 vectors 61 -> 125 us; 134 AOs, 8 vectors (54 MFLOP)
// 116 -> 128, 16 vectors (108 MFLOP) 170 -> 158; 178 AOs, 1 vector 118 -> 122,
// 4 vectors 131 -> 127; 222 AOs, 1 vector 133 -> 123; 579 AOs, 20 vectors
// 9932 -> 807 us.
// Above kMgMaxK AOs a row does not fit the split kernel's share of shared memory and the
// float64 pipe serves the products, as it did all before.
bool mg_applies(const DevMol& m, int nvec) {
  const double n = m.n, o = m.o, v = m.v;
  if (m.v > m.o || m.n < 96 || m.n > kMgMaxK) return false;
  return m.n >= 160 || 4.0 * nvec * (n * o * v + n * n * v) >= 8e7;
}

// vectors per pass of the residue products: kMgBytes of planes
int mg_chunk(const DevMol& m, int nvec) {
  const double per = 2.0 * kModuli * m.n * (2.0 * mg_kp(m.n) + mg_kp(m.v));
  return std::max(1, std::min(std::min(nvec, product_batch(m)), static_cast<int>(kMgBytes / per)));
}

// scratch of a pass (mg_prepare) and operands of the orbitals
size_t mg_scratch_bytes(const DevMol& m, int chunk) {
  return sizeof(mg_t) * (mg_plane_count(m.n, m.v, chunk) +
                         std::max(mg_plane_count(m.n, m.n, chunk), mg_plane_count(m.v, m.o, chunk)) +
                         (size_t)kModuli * chunk * m.n * mg_ldn(m.n)) + sizeof(int) * 2 * (size_t)chunk * m.n;
}
size_t mg_orbital_bytes(const DevMol& m) {
  return sizeof(mg_t) * (mg_plane_count(m.n, m.o, 1) + mg_plane_count(m.n, m.v, 1) + mg_plane_count(m.v, m.n, 1) +
                         mg_plane_count(m.o, m.n, 1)) + sizeof(int) * 3 * (size_t)m.n;
}

// operands and scratch for the residue products of `chunk` vectors, or null
// where they do not fit the device beside those of the other molecules, which are
// dropped first (the float64-pipe path serves those)
MgOrbitals* mg_prepare(Ctx& c, DevMol& m, int chunk) {
  const int n = m.n, o = m.o, v = m.v;
  cudaStream_t s = c.stream;
  for (;;) try {
    if (!c.mg_work) c.mg_work = std::make_shared<MgWork>();
    MgWork& w = *static_cast<MgWork*>(c.mg_work.get());
    w.a.planes.ensure(mg_plane_count(n, v, chunk));
    w.a.exps.ensure((size_t)chunk * n);
    w.b.planes.ensure(std::max(mg_plane_count(n, n, chunk), mg_plane_count(v, o, chunk)));
    w.b.exps.ensure((size_t)chunk * n);
    w.res.ensure((size_t)kModuli * chunk * n * mg_ldn(n));
    if (!c.tc_err.get()) {
      c.tc_err.alloc(1);
      XS_CUDA(cudaMemsetAsync(c.tc_err.get(), 0, sizeof(int), s));
    }
    if (!m.mg_orb) {
      auto q = std::make_shared<MgOrbitals>();
      const double* occ = m.CT.get();
      const double* vir = occ + (size_t)o * n;
      // C[mu][p] = CT[p][mu]: rows along mu are contiguous, K strided
      q->occ = MgOperand{occ, 1, n, 0, n, o, 1};
      q->vir = MgOperand{vir, 1, n, 0, n, v, 1};
      q->virT = MgOperand{vir, n, 1, 0, v, n, 1};
      q->occT = MgOperand{occ, n, 1, 0, o, n, 1};
      mg_split(s, 0, q->occ, q->s_occ);
      mg_split(s, 1, q->vir, q->s_vir);
      mg_split(s, 0, q->virT, q->s_virT);
      mg_split(s, 0, q->occT, q->s_occT);
      m.mg_orb = q;
    }
    return static_cast<MgOrbitals*>(m.mg_orb.get());
  } catch (const Error& e) {
    if (e.status != XS_ENOMEM) throw;
    cudaGetLastError();
    c.mg_work.reset();
    if (!c.drop_operands(&m)) return nullptr;
  }
}

// R (nvec x n x n) = C_occ X C_vir^T by residue products: W = C_occ X (n x v,
// right operand X^T), then R = W C_vir^T
void mg_pbuild(Ctx& c, const DevMol& m, const MgOrbitals& q, int nvec, const double* X, double* R, double* tmp) {
  cudaStream_t s = c.stream;
  MgWork& w = *static_cast<MgWork*>(c.mg_work.get());
  const int n = m.n, o = m.o, v = m.v;
  MgOperand x{X, 1, v, (long long)o * v, v, o, nvec};
  mg_split(s, 1, x, w.b);
  MgOut out;
  out.C = tmp; out.ldc = v; out.sC = (long long)n * v;
  mg_product(s, q.occ, x, nvec, out, w, c.tc_err.get());
  MgOperand t{tmp, v, 1, (long long)n * v, n, v, nvec};
  mg_split(s, 0, t, w.a);
  out.C = R; out.ldc = n; out.sC = (long long)n * n;
  mg_product(s, t, q.vir, nvec, out, w, c.tc_err.get());
}

// Y (nvec x o x v) = C_occ^T G C_vir + (eps_a - eps_i) X by residue products:
// S^T = C_vir^T G^T (v x n), Y = C_occ^T S
void mg_backtransform(Ctx& c, const DevMol& m, const MgOrbitals& q, int nvec, const double* G, const double* X,
                      double* Y, double* tmp) {
  cudaStream_t s = c.stream;
  MgWork& w = *static_cast<MgWork*>(c.mg_work.get());
  const int n = m.n, o = m.o, v = m.v;
  MgOperand g{G, n, 1, (long long)n * n, n, n, nvec};
  mg_split(s, 1, g, w.b);
  MgOut out;
  out.C = tmp; out.ldc = n; out.sC = (long long)v * n;
  mg_product(s, q.virT, g, nvec, out, w, c.tc_err.get());
  MgOperand t{tmp, n, 1, (long long)v * n, v, n, nvec};
  mg_split(s, 1, t, w.b);
  out.C = Y; out.ldc = v; out.sC = (long long)o * v;
  out.X = X; out.eps = m.eps.get(); out.o = o;
  mg_product(s, q.occT, t, nvec, out, w, c.tc_err.get());
}

}  // namespace

int product_batch(const DevMol& m) {
  // vectors per pass: bound the AO work arrays (R, G+, G-, tmp) to ~4 GB
  const double per = 8.0 * ((double)m.n * m.n * 3 + (double)m.n * (m.o > m.v ? m.o : m.v));
  int nb = static_cast<int>(4.0e9 / per);
  if (nb < 1) nb = 1;
  if (nb > 64) nb = 64;
  return nb;
}

size_t residue_bytes(const Ctx& c, const DevMol& m, int nvec) {
  if (!c.residues || !mg_applies(m, nvec)) return 0;
  size_t held = 0;
  if (c.mg_work) {
    const MgWork& w = *static_cast<const MgWork*>(c.mg_work.get());
    held = sizeof(mg_t) * (w.a.planes.n + w.b.planes.n + w.res.n) + sizeof(int) * (w.a.exps.n + w.b.exps.n);
  }
  const size_t need = mg_scratch_bytes(m, mg_chunk(m, nvec));
  return (need > held ? need - held : 0) + (m.mg_orb ? 0 : mg_orbital_bytes(m));
}

void products_fp64(Ctx& c, DevMol& m, int method, int nvec, const double* X, double* Y1, double* Y2, bool triplet) {
  cudaStream_t s = c.stream;
  const int n = m.n, o = m.o, v = m.v;
  const long long ov = (long long)o * v, nn = (long long)n * n;
  const int nb = product_batch(m);
  int chunk = nvec < nb ? nvec : nb;
  MgOrbitals* q = nullptr;
  if (c.residues && mg_applies(m, nvec)) {
    const int mc = mg_chunk(m, nvec);
    q = mg_prepare(c, m, mc);
    if (q) chunk = mc;
  }
  c.ws1.ensure((size_t)chunk * nn);                         // R
  double *G = nullptr, *Gm = nullptr;                       // G or G+, G-
  if (Y1) {
    c.ws2.ensure((size_t)chunk * nn);
    G = c.ws2.get();
  }
  if (method != XS_CIS && Y2) {
    c.ws3.ensure((size_t)chunk * nn);
    Gm = c.ws3.get();
  }
  c.ws4.ensure((size_t)chunk * n * (o > v ? o : v));        // transform scratch
  for (int k0 = 0; k0 < nvec; k0 += chunk) {
    const int k = (nvec - k0) < chunk ? (nvec - k0) : chunk;
    const double* Xk = X + k0 * ov;
    if (q) {
      const bool rpa = method != XS_CIS;
      mg_pbuild(c, m, *q, k, Xk, c.ws1.get(), c.ws4.get());
      gbuild<double>(s, m, c.d_par.get(), gmode(rpa, triplet), k, c.ws1.get(), G, Gm, c.ws0);
      if (Y1) mg_backtransform(c, m, *q, k, G, Xk, Y1 + k0 * ov, c.ws4.get());
      if (Gm) mg_backtransform(c, m, *q, k, Gm, Xk, Y2 + k0 * ov, c.ws4.get());
      continue;
    }
    pbuild<double>(s, n, o, v, k, m.CT.get(), Xk, c.ws1.get(), c.ws4.get());
    gbuild<double>(s, m, c.d_par.get(), gmode(method != XS_CIS, triplet), k, c.ws1.get(), G, Gm, c.ws0);
    if (Y1) {
      backtransform<double>(s, n, o, v, k, m.CT.get(), G, Y1 + k0 * ov, c.ws4.get());
      add_diag_term<double>(s, k, o, v, m.eps.get(), Xk, Y1 + k0 * ov);
    }
    if (Gm) {
      backtransform<double>(s, n, o, v, k, m.CT.get(), Gm, Y2 + k0 * ov, c.ws4.get());
      add_diag_term<double>(s, k, o, v, m.eps.get(), Xk, Y2 + k0 * ov);
    }
  }
}

// float32 SIMT products: float32 coefficients, R, G and integrals, float32
// accumulation with round-to-nearest (no tensor cores); the accurate
// reference for the final Rayleigh-Ritz step of a mixed-precision solve.
void products_f32(Ctx& c, DevMol& m, int method, int nvec, const double* X, double* Y1, double* Y2, bool triplet) {
  cudaStream_t s = c.stream;
  const int n = m.n, o = m.o, v = m.v;
  const long long ov = (long long)o * v, nn = (long long)n * n;
  if (!m.Wf.get()) {
    m.Wf.alloc((size_t)m.np * m.np);
    convert_d2f(s, (long long)m.np * m.np, m.W.get(), m.Wf.get());
  }
  if (!m.CTf.get()) {
    m.CTf.alloc(nn);
    convert_d2f(s, nn, m.CT.get(), m.CTf.get());
  }
  const int nb = product_batch(m);
  const int chunk = nvec < nb ? nvec : nb;
  const size_t tmpn = (size_t)chunk * n * (o > v ? o : v);
  c.fs2.ensure((size_t)chunk * nn * 3 + tmpn + (size_t)chunk * ov * 2);
  float* R = c.fs2.get();
  float* G = R + (size_t)chunk * nn;
  float* Gm = G + (size_t)chunk * nn;
  float* tmp = Gm + (size_t)chunk * nn;
  float* Xf = tmp + tmpn;
  float* Yf = Xf + (size_t)chunk * ov;
  for (int k0 = 0; k0 < nvec; k0 += chunk) {
    const int k = (nvec - k0) < chunk ? (nvec - k0) : chunk;
    const double* Xk = X + k0 * ov;
    convert_d2f(s, k * ov, Xk, Xf);
    pbuild<float>(s, n, o, v, k, m.CTf.get(), Xf, R, tmp);
    const bool rpa = method != XS_CIS;
    gbuild<float>(s, m, c.d_par.get(), gmode(rpa, triplet), k, R, Y1 ? G : nullptr, rpa && Y2 ? Gm : nullptr, c.fs1);
    for (int pass = 0; pass < (rpa ? 2 : 1); ++pass) {
      if (!(pass == 0 ? Y1 : Y2)) continue;
      double* Y = (pass == 0 ? Y1 : Y2) + k0 * ov;
      backtransform<float>(s, n, o, v, k, m.CTf.get(), pass == 0 ? G : Gm, Yf, tmp);
      convert_f2d(s, k * ov, Yf, Y);
      add_diag_term<double>(s, k, o, v, m.eps.get(), Xk, Y);
    }
  }
}

void products(Ctx& c, DevMol& m, int method, int precision, int nvec, const double* X, double* Y1, double* Y2,
              bool triplet, unsigned int* mx1, unsigned int* mx2) {
  if (nvec <= 0) return;
  if (precision == XS_MIXED) {
    products_mixed(c, m, method, nvec, X, Y1, Y2, triplet, mx1, mx2);
    return;
  }
  if (precision == kPrecF32) {
    products_f32(c, m, method, nvec, X, Y1, Y2, triplet);
    return;
  }
  products_fp64(c, m, method, nvec, X, Y1, Y2, triplet);
}

void gmatrix(Ctx& c, const DevMol& m, int precision, int nvec, const double* R, double* G) {
  (void)precision;
  gbuild<double>(c.stream, m, c.d_par.get(), G_CIS, nvec, R, G, nullptr, c.ws0);
}

}  // namespace xs
