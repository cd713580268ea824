// Mixed-precision A*X path of libxs (see tc.h).
//
// Per batch of k trial vectors (all tensor-core operands K-major TF32 pairs; float16 pairs in products_half):
//   1. X_k (o x v)                    -> TF32 pair, v padded to 32
//   2. U_k^T (n x o) = C_vir X_k^T    (tc_gemm, epilogue writes a TF32 pair)
//   3. R_k (n x n)   = C_occ U_k      (tc_gemm, float32 out)
//   4. G_k = G(R_k)                   (float32 G build, epilogue writes the TF32 pair, n padded)
//   5. S_k^T (v x n) = C_vir^T G_k^T  (tc_gemm, TF32 pair out)
//   6. D_k (o x v)   = C_occ^T S_k                (tc_gemm, float32 out)
//   7. Y_k = D_k + (eps_a - eps_i) X_k            (add_gaps, float64)
// For TDHF steps 5-7 run for G+ and G-.  When v < o, steps 1-3 contract the
// n x n product over v instead (2 n^2 v rather than 2 n^2 o flops):
//   1'. X_k^T (v x o) -> TF32 pair; 2'. W_k (n x v) = C_occ X_k;
//   3'. R_k = W_k C_vir^T.
// Steps 5-6 contract the n x n product over v (S^T is v x n).
#include "kernels.h"
#include "products.h"
#include "tc.h"
#include "tc_gemm.h"

namespace xs {

namespace {

// Products of at least this many AOs take float16 pairs; below, their four more
// launches cost more than the faster MMAs give.  (A+B)X, TF32 -> float16 pairs, 1 and
// 20 vectors: 331 AOs 132 -> 138 and 296 -> 337 us, 600 AOs 154 -> 151 and 397 -> 387,
// 840 AOs 177 -> 159 and 580 -> 524, 1234 AOs 232 -> 190 and 985 -> 813.
constexpr int kHalfMinAOs = 512;

// carve a sub-buffer of `count` elements, 256-byte aligned
struct Carver {
  char* base = nullptr;
  size_t at = 0;
  template <typename T>
  T* take(size_t count) {
    T* p = reinterpret_cast<T*>(base + at);
    at += (count * sizeof(T) + 255) / 256 * 256;
    return p;
  }
};

// The same pipeline with float16 pairs (tc_gemm.h): their MMA rate is twice that
// of TF32 and their two 11-bit significands the same, so the products are as
// accurate; float16's exponent range asks for a power of two per vector and stage:
//   X      from its largest entry (one pass over X);
//   U / W  from a bound inside the GEMM's epilogue (mode 2);
//   G, G-  from a bound on G by the largest |R| and |J2| (gbuild_half);
//   S      stored in float32 with its largest entry, split in a pass of its own
//          (a bound would lie 2^21 above typical entries, beyond the pairs' reach).
void products_half(Ctx& c, DevMol& m, int method, int nvec, const double* X, double* Y1, double* Y2, bool triplet,
                   unsigned int* mx1, unsigned int* mx2) {
  cudaStream_t s = c.stream;
  const int n = m.n, o = m.o, v = m.v;
  const int np_ = pad32(n), op = pad32(o), vp = pad32(v);
  const long long ov = (long long)o * v, nn = (long long)n * n;
  const size_t s_vir = (size_t)n * vp, s_occ = (size_t)n * op, s_virT = (size_t)v * np_, s_occT = (size_t)o * np_;
  if (!m.w_max.get()) {
    m.w_max.alloc(1);
    XS_CUDA(cudaMemsetAsync(m.w_max.get(), 0, sizeof(unsigned int), s));
    absmax_f64(s, (long long)m.np * m.np, m.W.get(), 0, 1, m.w_max.get());
  }
  if (!m.CTh_hi.get()) {
    // orbital operands, cached until the orbitals change (as in products_mixed), one exponent;
    // the molecule gets them when they are complete
    const size_t orb = s_vir + s_occ + s_virT + s_occT;
    DevBuf<unsigned int> amax(1);
    DevBuf<int> ce(1);
    DevBuf<__half> ch(orb), cl(orb);
    XS_CUDA(cudaMemsetAsync(amax.get(), 0, sizeof(unsigned int), s));
    const double* CT = m.CT.get();
    absmax_f64(s, nn, CT, 0, 1, amax.get());
    __half* h = ch.get();
    __half* l = cl.get();
    int* e = ce.get();
    split16(s, n, v, vp, CT + (size_t)o * n, n, 0, 0, 1, true, amax.get(), e, h, l);
    split16(s, n, o, op, CT, n, 0, 0, 1, true, amax.get(), e, h + s_vir, l + s_vir);
    split16(s, v, n, np_, CT + (size_t)o * n, n, 0, 0, 1, false, amax.get(), e, h + s_vir + s_occ, l + s_vir + s_occ);
    split16(s, o, n, np_, CT, n, 0, 0, 1, false, amax.get(), e, h + s_vir + s_occ + s_virT, l + s_vir + s_occ + s_virT);
    m.CTh_e = std::move(ce);
    m.CTh_lo = std::move(cl);
    m.CTh_hi = std::move(ch);
  }
  const __half* ch = m.CTh_hi.get();
  const __half* cl = m.CTh_lo.get();
  const int* ce = m.CTh_e.get();
  const TcOperand16 vir{ch, cl, vp, 0, false, ce}, occ{ch + s_vir, cl + s_vir, op, 0, false, ce},
      virT{ch + s_vir + s_occ, cl + s_vir + s_occ, np_, 0, false, ce},
      occT{ch + s_vir + s_occ + s_virT, cl + s_vir + s_occ + s_virT, np_, 0, false, ce};

  const int nb = product_batch(m);
  const int chunk = nvec < nb ? nvec : nb;
  const bool vfirst = v < o, rpa = method != XS_CIS;
  const bool plus = Y1 != nullptr, minus = rpa && Y2;   // products asked for
  const size_t nX = (size_t)chunk * (vfirst ? (size_t)v * op : (size_t)o * vp), nU = (size_t)chunk * n * (vfirst ? vp : op);
  const size_t nG = (size_t)chunk * n * np_, nS = (size_t)chunk * v * np_;
  __half *Xh, *Xl, *Uh, *Ul, *Sh, *Sl;
  GHalf g;
  float *R, *S, *D;
  unsigned int *xmax, *rmax, *smax;
  int *eX, *eU, *eS;
  Carver cv;
  for (int pass = 0; pass < 2; ++pass) {   // sizes, then pointers
    if (pass == 1) {
      c.fs0.ensure((cv.at + 3) / 4);
      cv = Carver{reinterpret_cast<char*>(c.fs0.get()), 0};
    }
    Xh = cv.take<__half>(nX); Xl = cv.take<__half>(nX);
    Uh = cv.take<__half>(nU); Ul = cv.take<__half>(nU);
    R = cv.take<float>((size_t)chunk * nn);
    if (plus) { g.h = cv.take<__half>(nG); g.l = cv.take<__half>(nG); }
    if (minus) { g.mh = cv.take<__half>(nG); g.ml = cv.take<__half>(nG); }
    S = cv.take<float>((size_t)chunk * v * n);
    D = cv.take<float>((size_t)chunk * ov);
    Sh = cv.take<__half>(nS); Sl = cv.take<__half>(nS);
    xmax = cv.take<unsigned int>(chunk); rmax = cv.take<unsigned int>(chunk); smax = cv.take<unsigned int>(2 * chunk);
    eX = cv.take<int>(chunk); eU = cv.take<int>(chunk); eS = cv.take<int>(chunk);
    g.e = cv.take<int>(chunk); g.em = cv.take<int>(chunk);
  }
  int* err = c.tc_err.get();
  for (int k0 = 0; k0 < nvec; k0 += chunk) {
    const int k = (nvec - k0) < chunk ? (nvec - k0) : chunk;
    const double* Xk = X + k0 * ov;
    XS_CUDA(cudaMemsetAsync(xmax, 0, reinterpret_cast<char*>(smax + 2 * chunk) - reinterpret_cast<char*>(xmax), s));   // and rmax
    absmax_f64(s, ov, Xk, ov, k, xmax);
    TcEpilogue ew, er;
    ew.mode = 2; ew.Dh = Uh; ew.Dhl = Ul; ew.eout = eU;
    er.mode = 0; er.D = R; er.ld = n; er.bstride = nn; er.rowmax = rmax;
    if (vfirst) {
      // W = C_occ X (n x v), R = W C_vir^T
      split16(s, v, o, op, Xk, v, ov, (long long)v * op, k, true, xmax, eX, Xh, Xl);
      ew.ld = vp; ew.bstride = (long long)n * vp;
      tc_gemm(s, occ, TcOperand16{Xh, Xl, op, (long long)v * op, true, eX}, n, v, op, k, ew, err);
      tc_gemm(s, TcOperand16{Uh, Ul, vp, (long long)n * vp, true, eU}, vir, n, n, vp, k, er, err);
    } else {
      // U^T = C_vir X^T (n x o), R = C_occ U
      split16(s, o, v, vp, Xk, v, ov, (long long)o * vp, k, false, xmax, eX, Xh, Xl);
      ew.ld = op; ew.bstride = (long long)n * op;
      tc_gemm(s, vir, TcOperand16{Xh, Xl, vp, (long long)o * vp, true, eX}, n, o, vp, k, ew, err);
      tc_gemm(s, occ, TcOperand16{Uh, Ul, op, (long long)n * op, true, eU}, n, n, op, k, er, err);
    }
    gbuild_half(s, m, c.d_par.get(), gmode(rpa, triplet), k, R, rmax, m.w_max.get(), g, np_, c.fs1);
    for (int pass = 0; pass < (rpa ? 2 : 1); ++pass) {
      const __half* Gh = pass == 0 ? g.h : g.mh;
      if (!Gh) continue;
      // S^T = C_vir^T G^T (v x n), Y = C_occ^T S + d eps X
      TcEpilogue es, ey;
      es.mode = 0; es.D = S; es.ld = n; es.bstride = (long long)v * n; es.rowmax = smax + pass * chunk;
      tc_gemm(s, virT, TcOperand16{Gh, pass == 0 ? g.l : g.ml, np_, (long long)n * np_, true, pass == 0 ? g.e : g.em}, v,
              n, np_, k, es, err);
      split16(s, v, n, np_, S, (long long)v * n, (long long)v * np_, k, es.rowmax, eS, Sh, Sl);
      unsigned int* mxo = pass == 0 ? mx1 : mx2;
      ey.mode = 0; ey.D = D; ey.ld = v; ey.bstride = ov;
      tc_gemm(s, occT, TcOperand16{Sh, Sl, np_, (long long)v * np_, true, eS}, o, v, np_, k, ey, err);
      add_gaps(s, k, o, v, m.eps.get(), D, Xk, (pass == 0 ? Y1 : Y2) + k0 * ov, mxo ? mxo + k0 : nullptr);
    }
  }
}

}  // namespace

void products_mixed(Ctx& c, DevMol& m, int method, int nvec, const double* X, double* Y1, double* Y2, bool triplet,
                    unsigned int* mx1, unsigned int* mx2) {
  cudaStream_t s = c.stream;
  const int n = m.n, o = m.o, v = m.v;
  const int np_ = pad32(n), op = pad32(o), vp = pad32(v);
  const long long ov = (long long)o * v, nn = (long long)n * n;
  if (!m.Wf.get()) {
    m.Wf.alloc((size_t)m.np * m.np);
    convert_d2f(s, (long long)m.np * m.np, m.W.get(), m.Wf.get());
  }
  DevBuf<int>& err = c.tc_err;
  if (!err.get()) {
    err.alloc(1);
    XS_CUDA(cudaMemsetAsync(err.get(), 0, sizeof(int), s));
  }
  if (mx1) XS_CUDA(cudaMemsetAsync(mx1, 0, sizeof(unsigned int) * nvec, s));
  if (mx2 && method != XS_CIS && Y2) XS_CUDA(cudaMemsetAsync(mx2, 0, sizeof(unsigned int) * nvec, s));
  if (n >= kHalfMinAOs) {
    products_half(c, m, method, nvec, X, Y1, Y2, triplet, mx1, mx2);
    return;
  }
  // orbital operands, cached until the orbitals change:
  //   Cvir (n x vp) = C[mu][o + a], Cocc (n x op) = C[mu][i],
  //   CTvir (v x np) = CT[o + a][mu], CTocc (o x np) = CT[i][mu]
  const size_t orb = (size_t)n * vp + (size_t)n * op + (size_t)v * np_ + (size_t)o * np_;
  if (!m.CTf_hi.get()) {
    DevBuf<float> hi(orb), lo(orb);   // the molecule gets them when they are complete
    float* h = hi.get();
    float* l = lo.get();
    const double* CT = m.CT.get();
    split_pad<double>(s, n, v, vp, CT + (size_t)o * n, n, 0, 0, 1, true, h, l);
    h += (size_t)n * vp; l += (size_t)n * vp;
    split_pad<double>(s, n, o, op, CT, n, 0, 0, 1, true, h, l);
    h += (size_t)n * op; l += (size_t)n * op;
    split_pad<double>(s, v, n, np_, CT + (size_t)o * n, n, 0, 0, 1, false, h, l);
    h += (size_t)v * np_; l += (size_t)v * np_;
    split_pad<double>(s, o, n, np_, CT, n, 0, 0, 1, false, h, l);
    m.CTf_lo = std::move(lo);
    m.CTf_hi = std::move(hi);
  }
  const float* Cvir_h = m.CTf_hi.get();
  const float* Cvir_l = m.CTf_lo.get();
  const float* Cocc_h = Cvir_h + (size_t)n * vp;
  const float* Cocc_l = Cvir_l + (size_t)n * vp;
  const float* CTvir_h = Cocc_h + (size_t)n * op;
  const float* CTvir_l = Cocc_l + (size_t)n * op;
  const float* CTocc_h = CTvir_h + (size_t)v * np_;
  const float* CTocc_l = CTvir_l + (size_t)v * np_;

  const int nb = product_batch(m);
  const int chunk = nvec < nb ? nvec : nb;
  // P build order: the n^2 contraction runs over the smaller of o and v
  //   o <= v: U^T = C_vir X^T (n x o), R = C_occ U
  //   v <  o: W = C_occ X (n x v), R = W C_vir^T
  const bool vfirst = v < o;
  // per vector: X pair (X, or X^T when vfirst), U^T or W pair, R, G+, G-, G pair, S^T pair
  // sub-buffers start on 256-byte boundaries (tensor maps need 16-byte aligned bases)
  auto up = [](size_t x) { return (x + 63) / 64 * 64; };
  const size_t sX = up((size_t)chunk * (vfirst ? (size_t)v * op : (size_t)o * vp));
  const size_t sU = up((size_t)chunk * n * (vfirst ? vp : op)), sR = up((size_t)chunk * nn);
  const size_t sG = up((size_t)chunk * n * np_), sS = up((size_t)chunk * v * np_);
  const bool rpa = method != XS_CIS;
  const bool plus = Y1 != nullptr, minus = rpa && Y2;   // products asked for
  c.fs0.ensure(2 * sX + 2 * sU + sR + ((plus ? 2 : 0) + (minus ? 2 : 0)) * sG + 2 * sS +
              up((size_t)chunk * ov));
  float* p = c.fs0.get();
  float* Xh = p; p += sX;
  float* Xl = p; p += sX;
  float* Uh = p; p += sU;
  float* Ul = p; p += sU;
  float* R = p; p += sR;
  float* Gh = nullptr;        // TF32 pair of G (CIS) or G+ (TDHF)
  float* Gl = nullptr;
  float* Gmh = nullptr;       // TF32 pair of G- (TDHF)
  float* Gml = nullptr;
  if (plus) {
    Gh = p; p += sG;
    Gl = p; p += sG;
  }
  if (minus) {
    Gmh = p; p += sG;
    Gml = p; p += sG;
  }
  float* Sh = p; p += sS;
  float* Sl = p; p += sS;
  float* D = p;               // C_occ^T G C_vir

  for (int k0 = 0; k0 < nvec; k0 += chunk) {
    const int k = (nvec - k0) < chunk ? (nvec - k0) : chunk;
    const double* Xk = X + k0 * ov;
    if (vfirst) {
      split_pad_t(s, v, o, op, Xk, v, ov, (long long)v * op, k, Xh, Xl);   // X^T pair: v x op
      {  // W = C_occ X : M = n, N = v, K = o
        TcOperand A{Cocc_h, Cocc_l, op, 0, false};
        TcOperand B{Xh, Xl, op, (long long)v * op, true};
        TcEpilogue e;
        e.mode = 1; e.D = Uh; e.Dlo = Ul; e.ld = vp; e.bstride = (long long)n * vp;
        tc_gemm(s, A, B, n, v, op, k, e, err.get());
      }
      {  // R = W C_vir^T : M = n, N = n, K = v
        TcOperand A{Uh, Ul, vp, (long long)n * vp, true};
        TcOperand B{Cvir_h, Cvir_l, vp, 0, false};
        TcEpilogue e;
        e.mode = 0; e.D = R; e.ld = n; e.bstride = nn;
        tc_gemm(s, A, B, n, n, vp, k, e, err.get());
      }
    } else {
      split_pad<double>(s, o, v, vp, Xk, v, ov, (long long)o * vp, k, false, Xh, Xl);
      {  // U^T = C_vir X^T : M = n, N = o, K = v
        TcOperand A{Cvir_h, Cvir_l, vp, 0, false};
        TcOperand B{Xh, Xl, vp, (long long)o * vp, true};
        TcEpilogue e;
        e.mode = 1; e.D = Uh; e.Dlo = Ul; e.ld = op; e.bstride = (long long)n * op;
        tc_gemm(s, A, B, n, o, vp, k, e, err.get());
      }
      {  // R = C_occ U : M = n, N = n, K = o
        TcOperand A{Cocc_h, Cocc_l, op, 0, false};
        TcOperand B{Uh, Ul, op, (long long)n * op, true};
        TcEpilogue e;
        e.mode = 0; e.D = R; e.ld = n; e.bstride = nn;
        tc_gemm(s, A, B, n, n, op, k, e, err.get());
      }
    }
    // G (and G-) written directly as the back-transform's TF32 pairs
    gbuild_split(s, m, c.d_par.get(), gmode(rpa, triplet), k, R, Gh, Gl, Gmh, Gml, np_, c.fs1);
    for (int pass = 0; pass < (rpa ? 2 : 1); ++pass) {
      const float* Gph = pass == 0 ? Gh : Gmh;
      const float* Gpl = pass == 0 ? Gl : Gml;
      if (!Gph) continue;
      double* Yout = (pass == 0 ? Y1 : Y2) + k0 * ov;
      unsigned int* mxo = pass == 0 ? mx1 : mx2;
      {  // S^T = C_vir^T G^T : M = v, N = n, K = n
        TcOperand A{CTvir_h, CTvir_l, np_, 0, false};
        TcOperand B{Gph, Gpl, np_, (long long)n * np_, true};
        TcEpilogue e;
        e.mode = 1; e.D = Sh; e.Dlo = Sl; e.ld = np_; e.bstride = (long long)v * np_;
        tc_gemm(s, A, B, v, n, np_, k, e, err.get());
      }
      {  // D = C_occ^T S : M = o, N = v, K = n; Y = D + d eps X
        TcOperand A{CTocc_h, CTocc_l, np_, 0, false};
        TcOperand B{Sh, Sl, np_, (long long)v * np_, true};
        TcEpilogue e;
        e.mode = 0; e.D = D; e.ld = v; e.bstride = ov;
        tc_gemm(s, A, B, o, v, np_, k, e, err.get());
        add_gaps(s, k, o, v, m.eps.get(), D, Xk, Yout, mxo ? mxo + k0 : nullptr);
      }
    }
  }
  // the error word (bounded waits) is read by the caller at its next
  // synchronisation (check_device_error), not here: no per-product host sync
}

}  // namespace xs
