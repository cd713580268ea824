// Float32 G(R) build over unordered pairs of super-atoms (the G build of the
// mixed-precision products; paper, Section "GPU Implementation", Eq. ftilde).
//
// A super-atom is a heavy atom (4 AOs) or a run of up to 4 consecutive
// hydrogens.  One thread owns one unordered pair (I, J) of super-atoms: it
// loads the pair's two-centre integrals (mu nu|lam sig) once into shared
// memory (at most 10 x 10 products) and then, for every matrix of the batch, reads
// the two 4 x 4 blocks R_IJ and R_JI once, forms both exchange blocks
//   K_IJ[mu][lam] = sum_{nu in at(mu), sig in at(lam)} (mu nu|lam sig) R[nu][sig]
//   K_JI[lam][mu] = sum (mu nu|lam sig) R[sig][nu]
// and writes both G blocks.  Because K(R^T)_IJ = K_JI^T, the TDHF outputs
// need no second pass over R:
//   CIS:  G_IJ = -K_IJ,                G_JI = -K_JI
//   TDHF: G+_IJ = -(K_IJ + K_JI^T),    G+_JI = G+_IJ^T
//         G-_IJ = -(K_IJ - K_JI^T),    G-_JI = -G-_IJ^T
// Pairs with I = J hold the diagonal atom blocks: the closed-form one-centre
// Coulomb and exchange terms, the two-centre Coulomb J2 = W r of the diagonal
// blocks, and inside a hydrogen run the exchange between its hydrogens.
// Every R element is read once and every G element written once per matrix.
// A warp holds 2 consecutive super-atoms I x 16 consecutive super-atoms J, so
// the row segments it reads and writes are contiguous (16-byte loads and
// stores where the blocks start on multiples of 4 AOs), and each thread keeps
// the next matrix's blocks in flight while it contracts the current one.
#include <algorithm>
#include <vector>

#include "gpair_dev.cuh"
#include "kernels.h"
#include "prof.h"

namespace xs {

namespace {

// A thread's walk over the vectors is a chain of uncoalesced loads, contraction and
// stores, so the vectors are dealt out to enough CTAs to keep the SMs' 16 resident warps
// replaced four times over; the integrals are read again by each (from L2, 100 floats
// against 64 of R and G per vector).  One walk per pair -> this split, 256 -> 64 threads:
// 2200 AOs x 20 vectors 467 -> 406 us, 1233 x 20 300 -> 182, 600 x 10 116 -> 38,
// 222 x 8 82 -> 15.5; one vector 17 -> 15.  Twice or half as many CTAs are within 3%
// or up to 10% slower.
constexpr int kPairThreads = 64;
constexpr int kPairTargetCTAs = 4 * 8 * 152;

template <GMode MODE, int SPLIT, int OUT>
__global__ void __launch_bounds__(kPairThreads, 8) gpair_kernel(int n, int np, int nvec, int npairs,
                                                                const int2* __restrict__ pairs,
                                                                const int4* __restrict__ sa,
                                                                const double* __restrict__ par,
                                                                const float* __restrict__ W,
                                                                const float* __restrict__ J2, int ldj,
                                                                const float* __restrict__ R, int per, PairOut o) {
  extern __shared__ float wsm[];   // 100 integrals per thread
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= npairs) return;
  const int v0 = blockIdx.y * per, nv = min(per, nvec - v0);
  const size_t at = (size_t)v0 * n * (SPLIT ? o.ldo : n);
  if (SPLIT == kPlain) {
    o.G += at;
    o.Gm += at;
  } else if (SPLIT == kTf32Pair) {
    o.Gh += at; o.Gl += at;
    o.Gmh += at; o.Gml += at;
  } else {
    o.Hh += at; o.Hl += at; o.e += v0;
    o.Hmh += at; o.Hml += at; o.em += v0;
  }
  gpair_one<MODE, SPLIT, OUT>(n, np, nv, pairs[t], sa, par, W, J2 + v0, ldj, R + (size_t)v0 * n * n, o,
                              wsm + threadIdx.x * 100);
}

template <GMode MODE, int SPLIT, int OUT>
void launch_mode(cudaStream_t s, const DevMol& m, const double* d_par, int nvec, const float* W, const float* J2,
                 int ldj, const float* R, const PairOut& o) {
  const size_t smem = sizeof(float) * 100 * kPairThreads;
  static std::atomic<unsigned long long> allowed{0};
  allow_smem(allowed, gpair_kernel<MODE, SPLIT, OUT>, smem);
  const int npairs = m.gp_npairs;
  const int ctas = (npairs + kPairThreads - 1) / kPairThreads;
  const int chunks = std::min(nvec, std::max(1, (kPairTargetCTAs + ctas - 1) / ctas));
  const int per = (nvec + chunks - 1) / chunks;
  gpair_kernel<MODE, SPLIT, OUT><<<dim3(ctas, (nvec + per - 1) / per), kPairThreads, smem, s>>>(
      m.n, m.np, nvec, npairs, reinterpret_cast<const int2*>(m.gp_pairs.get()),
      reinterpret_cast<const int4*>(m.gp_sa.get()), d_par, W, J2, ldj, R, per, o);
  XS_CHECK_LAUNCH();
}

template <int SPLIT>
void launch_pairs(cudaStream_t s, const DevMol& m, const double* d_par, GMode mode, int nvec, const float* W,
                  const float* J2, int ldj, const float* R, const PairOut& o) {
  const bool plus = SPLIT == kHalfPair ? o.Hh != nullptr : (SPLIT == kTf32Pair ? o.Gh != nullptr : o.G != nullptr);
  const bool minus = SPLIT == kHalfPair ? o.Hmh != nullptr : (SPLIT == kTf32Pair ? o.Gmh != nullptr : o.Gm != nullptr);
#define XS_PAIRS(MODE, OUT) launch_mode<MODE, SPLIT, OUT>(s, m, d_par, nvec, W, J2, ldj, R, o)
  if (mode == G_CIS) XS_PAIRS(G_CIS, kOutPlus);
  else if (mode == G_CIS_T) XS_PAIRS(G_CIS_T, kOutPlus);
  else if (mode == G_RPA && plus && minus) XS_PAIRS(G_RPA, kOutBoth);
  else if (mode == G_RPA && plus) XS_PAIRS(G_RPA, kOutPlus);
  else if (mode == G_RPA_T && plus && minus) XS_PAIRS(G_RPA_T, kOutBoth);
  else if (mode == G_RPA_T && plus) XS_PAIRS(G_RPA_T, kOutPlus);
  else XS_PAIRS(G_RPA_T, kOutMinus);   // G- = -K(R) + K(R^T) has no Coulomb part
#undef XS_PAIRS
}

// Two-centre Coulomb of the diagonal blocks, J2 = W r (np x nvec, row
// stride nvec), W symmetric np x np, r np x nvec (row stride nvec).
// W is streamed once: J2[q][v] = sum_p W[p][q] r[p][v], threads along q (row
// segments of W), CTAs along q blocks and p chunks; the chunk partials are
// summed in chunk order (deterministic).
constexpr int kJ2Rows = 128;   // p rows per chunk
constexpr int kJ2Vec = 16;     // vectors per pass

__global__ void __launch_bounds__(256) j2_partial_kernel(int np, int nvec, const float* __restrict__ W,
                                                         const float* __restrict__ r, float* __restrict__ part) {
  __shared__ float rs[kJ2Rows][kJ2Vec];
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  const int p0 = blockIdx.y * kJ2Rows, p1 = min(np, p0 + kJ2Rows);
  for (int v0 = 0; v0 < nvec; v0 += kJ2Vec) {
    const int nv = min(kJ2Vec, nvec - v0);
    __syncthreads();
    for (int idx = threadIdx.x; idx < kJ2Rows * kJ2Vec; idx += blockDim.x) {
      const int pp = idx / kJ2Vec, v = idx - pp * kJ2Vec;
      rs[pp][v] = (p0 + pp < p1 && v < nv) ? r[(long long)(p0 + pp) * nvec + v0 + v] : 0.0f;
    }
    __syncthreads();
    if (q < np) {
      float acc[kJ2Vec];
#pragma unroll
      for (int v = 0; v < kJ2Vec; ++v) acc[v] = 0.0f;
      for (int p = p0; p < p1; ++p) {
        const float w = __ldg(W + (long long)p * np + q);
#pragma unroll
        for (int v = 0; v < kJ2Vec; ++v) acc[v] = fmaf(w, rs[p - p0][v], acc[v]);
      }
      float* out = part + ((long long)blockIdx.y * np + q) * nvec + v0;
      for (int v = 0; v < nv; ++v) out[v] = acc[v];
    }
  }
}

__global__ void j2_reduce_kernel(int np, int nvec, int nchunk, const float* __restrict__ part, float* __restrict__ J2) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)np * nvec) return;
  float s = 0.0f;
  for (int c = 0; c < nchunk; ++c) s += part[(long long)c * np * nvec + idx];
  J2[idx] = s;
}

// Exponents of the float16 pairs of G and G-, one CTA per matrix: a bound of
// |G| from the largest |R| (bits in rmax), the largest |J2| of the matrix and the
// largest integral w (two-centre products, abs_hi in wmax, and one-centre
// parameters): the exchange of a block sums at most 16 products w R, the
// one-centre Coulomb and exchange 4, G+ twice and four times those.
__global__ void __launch_bounds__(256) g_exponents_kernel(int np, int nvec, const float* __restrict__ J2, int ldj,
                                                          const unsigned int* __restrict__ rmax,
                                                          const unsigned int* __restrict__ wmax,
                                                          const double* __restrict__ par, int* __restrict__ e,
                                                          int* __restrict__ em) {
  __shared__ unsigned int top;
  const int v = blockIdx.x;
  if (threadIdx.x == 0) top = 0;
  __syncthreads();
  unsigned int j = 0;
  if (J2)
    for (int q = threadIdx.x; q < np; q += blockDim.x) j = max(j, __float_as_uint(J2[(long long)q * ldj + v]) & 0x7FFFFFFFu);
  j = __reduce_max_sync(0xffffffffu, j);
  if ((threadIdx.x & 31) == 0) atomicMax(&top, j);
  __syncthreads();
  if (threadIdx.x > 0) return;
  float w = static_cast<float>(__hiloint2double(static_cast<int>(*wmax + 1), 0));
  for (int z = 0; z < XS_NELEM; ++z)
    for (int q = 4; q <= 8; ++q) w = fmaxf(w, fabsf(static_cast<float>(par[z * XS_NPARAM + q])));
  const float r = __uint_as_float(rmax[v]), jm = __uint_as_float(top);
  auto exponent = [](float bound) {          // bound < 2^(e + 15)
    const int ex = static_cast<int>(__float_as_uint(bound) >> 23);
    return ex == 0 || ex == 0xFF ? 0 : ex - 127 - 14;
  };
  // rounding of the sums stays far below the factor 48 / 32 over the exchange alone
  if (e) e[v] = exponent(48.0f * w * r + 4.0f * jm);
  if (em) em[v] = exponent(33.0f * w * r);
}

__global__ void zero_pad_half_kernel(int rows, int n, int ldo, int nvec, __half* a, __half* b) {
  const int w = ldo - n;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)nvec * rows * w) return;
  const long long at = (idx / w) * ldo + n + idx % w;
  a[at] = __float2half_rn(0.0f);
  b[at] = __float2half_rn(0.0f);
}

}  // namespace

void build_gpairs(cudaStream_t s, DevMol& m) {
  const MolLayout& L = m.L;
  std::vector<int> sa;   // x, y, z, w per super-atom
  for (int A = 0; A < L.natoms;) {
    if (L.nao_atom[A] == 4) {
      sa.insert(sa.end(), {L.ao_off[A], 4 | 16, L.prod_off[A], L.elem[A]});
      ++A;
      continue;
    }
    int A1 = A, cnt = 0;
    while (A1 < L.natoms && L.nao_atom[A1] == 1 && cnt < 4) { ++A1; ++cnt; }
    sa.insert(sa.end(), {L.ao_off[A], cnt, L.prod_off[A], L.elem[A]});
    A = A1;
  }
  const int ns = static_cast<int>(sa.size() / 4);
  // warp blocks: 2 consecutive super-atoms I x 16 consecutive super-atoms J >= I
  std::vector<int> pairs;
  for (int I0 = 0; I0 < ns; I0 += 2)
    for (int J0 = (I0 / 16) * 16; J0 < ns; J0 += 16) {
      for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 16; ++b) {
          const int I = I0 + a, J = J0 + b;
          const bool ok = I < ns && J < ns && J >= I;
          pairs.push_back(ok ? I : -1);
          pairs.push_back(ok ? J : -1);
        }
    }
  m.gp_nsa = ns;
  m.gp_npairs = static_cast<int>(pairs.size() / 2);
  m.gp_sa.alloc(sa.size());
  m.gp_pairs.alloc(pairs.size());
  XS_CUDA(cudaMemcpyAsync(m.gp_sa.get(), sa.data(), sizeof(int) * sa.size(), cudaMemcpyHostToDevice, s));
  XS_CUDA(cudaMemcpyAsync(m.gp_pairs.get(), pairs.data(), sizeof(int) * pairs.size(), cudaMemcpyHostToDevice, s));
  XS_CUDA(cudaStreamSynchronize(s));
}

void coulomb_j2(cudaStream_t s, int np, int nvec, const float* W, const float* r, float* J2, DevBuf<float>& ws) {
  if (nvec <= 0) return;
  const int nchunk = (np + kJ2Rows - 1) / kJ2Rows;
  ws.ensure((size_t)nchunk * np * nvec);
  ProfScope ps(s, "coulomb_j2_f32", 4.0 * ((double)np * np + 2.0 * np * nvec), 2.0 * (double)np * np * nvec);
  j2_partial_kernel<<<dim3((np + 255) / 256, nchunk), 256, 0, s>>>(np, nvec, W, r, ws.get());
  XS_CHECK_LAUNCH();
  j2_reduce_kernel<<<grid1((long long)np * nvec, 256), 256, 0, s>>>(np, nvec, nchunk, ws.get(), J2);
  XS_CHECK_LAUNCH();
}

void gpair_build(cudaStream_t s, const DevMol& m, const double* d_par, GMode mode, int nvec, const float* W,
                 const float* J2, int ldj, const float* R, float* G, float* Gm) {
  PairOut o{G, Gm, nullptr, nullptr, nullptr, nullptr, 0};
  launch_pairs<kPlain>(s, m, d_par, mode, nvec, W, J2, ldj, R, o);
}

void gpair_build_split(cudaStream_t s, const DevMol& m, const double* d_par, GMode mode, int nvec, const float* W,
                       const float* J2, int ldj, const float* R, float* Gh, float* Gl, float* Gmh, float* Gml,
                       int ldo) {
  PairOut o{nullptr, nullptr, Gh, Gl, Gmh, Gml, ldo};
  launch_pairs<kTf32Pair>(s, m, d_par, mode, nvec, W, J2, ldj, R, o);
}

void gbuild_half(cudaStream_t s, const DevMol& m, const double* d_par, GMode mode, int nvec, const float* R,
                 const unsigned int* rmax, const unsigned int* wmax, const GHalf& o, int ldo, DevBuf<float>& ws) {
  if (nvec <= 0) return;
  const int n = m.n, np = m.np;
  ws.ensure((size_t)2 * np * nvec);
  float* r = ws.get();
  float* J2 = r + (size_t)np * nvec;
  const bool coulomb = (mode == G_CIS || mode == G_RPA) && o.h;   // G- has no Coulomb part
  if (coulomb) {
    pack_diag_kernel<float><<<(m.L.natoms + 31) / 32, dim3(8, 32), 0, s>>>(
        m.L.natoms, n, np, nvec, m.atom_ao_off.get(), m.atom_nao.get(), m.atom_prod_off.get(), R, r);
    XS_CHECK_LAUNCH();
    static thread_local ThreadScratch<float> j2_ws;
    coulomb_j2(s, np, nvec, m.Wf.get(), r, J2, j2_ws.here());
  }
  g_exponents_kernel<<<nvec, 256, 0, s>>>(np, nvec, coulomb ? J2 : nullptr, nvec, rmax, wmax, d_par, o.e, o.em);
  XS_CHECK_LAUNCH();
  if (ldo > n) {
    const long long cnt = (long long)nvec * n * (ldo - n);
    if (o.h) zero_pad_half_kernel<<<grid1(cnt, 256), 256, 0, s>>>(n, n, ldo, nvec, o.h, o.l);
    if (o.mh) zero_pad_half_kernel<<<grid1(cnt, 256), 256, 0, s>>>(n, n, ldo, nvec, o.mh, o.ml);
    XS_CHECK_LAUNCH();
  }
  PairOut p{nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, ldo, o.h, o.l, o.mh, o.ml, o.e, o.em};
  // algorithmic traffic: read R, write the float16 pairs, read the pair integrals once
  const double outs = (o.h ? 1.0 : 0.0) + (o.mh ? 1.0 : 0.0);
  ProfScope ps(s, "gbuild_assemble_f32", 4.0 * ((double)nvec * n * n * (1.0 + outs) + (double)np * np), 0.0);
  launch_pairs<kHalfPair>(s, m, d_par, mode, nvec, m.Wf.get(), J2, nvec, R, p);
}

}  // namespace xs
