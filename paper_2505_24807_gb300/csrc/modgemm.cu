// Float64 matrix products on the BF16 tensor cores by residues (modgemm.h).
//
//   mg_norm / mg_split_rows / mg_split_cols   row exponents and residue planes
//   mg_kernel    one bfloat16 GEMM per modulus, accumulated exactly, reduced
//   mg_crt       the remainder theorem, one rounding to float64
//
// Nothing here uses the float64 pipe (two lanes per clock and SM): integers
// come from the IEEE fields, the remainder theorem runs in 128-bit integers,
// and the result's bits are assembled.  Rows with a non-finite entry are
// flagged, and every output that meets one is computed as a plain float64 dot
// product of the sources in the last step, so infinities and NaN come out as a
// float64 GEMM gives them.
#include <algorithm>

#include "modgemm.h"
#include "prof.h"
#include "tcgen05.cuh"

namespace xs {

namespace {

using namespace tc5;

constexpr int kBits = 57;            // bits of a row's 2-norm
constexpr int kBad = -(1 << 20);     // exponent of a row that takes the plain dot product

// 13 pairwise coprime moduli; their product M is 2^116.36, so 4 2^(2 57) <= M
__host__ __device__ constexpr int mod_at(int l) {
  constexpr int m[kModuli] = {512, 511, 509, 507, 505, 503, 499, 493, 491, 487, 479, 473, 467};
  return m[l];
}

using u128 = unsigned __int128;

__host__ __device__ constexpr u128 mod_product() {
  u128 p = 1;
  for (int l = 0; l < kModuli; ++l) p *= static_cast<u128>(mod_at(l));
  return p;
}

__host__ __device__ constexpr int mod_inverse(int a, int m) {   // a^-1 mod m by search (compile time)
  for (int x = 1; x < m; ++x)
    if ((static_cast<long long>(a) * x) % m == 1) return x;
  return 0;
}

// weight of modulus l: (M / m_l)^-1 mod m_l
__host__ __device__ constexpr int crt_weight(int l) {
  return mod_inverse(static_cast<int>((mod_product() / mod_at(l)) % mod_at(l)), mod_at(l));
}

__host__ __device__ constexpr int sym_mod(long long x, int m) {
  const int h = m / 2;
  return static_cast<int>(((x + h) % m + m) % m) - h;
}

// an integer a' = a0 + 2^20 a1 + 2^40 a2 (0 <= a0, a1 < 2^20, |a2| <= 2^17) has
// the residue a0 c0 + a1 c1 + a2 c2 (|.| < 2^29.1) with c_j = 2^(20 j) q mod m,
// q = 1 for left and the remainder weight for right operands
__host__ __device__ constexpr int piece(int side, int l, int j) {
  const long long q = side ? crt_weight(l) : 1;
  const long long p = j == 0 ? 1 : (j == 1 ? (1ll << 20) : (1ll << 40));
  return sym_mod((p % mod_at(l)) * q, mod_at(l));
}

__host__ __device__ constexpr uint32_t mod_offset(int l) {   // a multiple of m near 2^30
  return static_cast<uint32_t>((1u << 30) / mod_at(l)) * mod_at(l);
}
// floor(y / m) = (y magic) >> 40 for y < 2^31: magic m - 2^40 <= 2^9
__host__ __device__ constexpr uint32_t mod_magic(int l) {
  return static_cast<uint32_t>((1ull << 40) / mod_at(l) + 1);
}

struct PieceTable {
  int c[2][kModuli][3];
  int m[kModuli];
  uint32_t shift[kModuli], magic[kModuli];   // mod_offset + m / 2, mod_magic
};
constexpr PieceTable make_pieces() {
  PieceTable t{};
  for (int s = 0; s < 2; ++s)
    for (int l = 0; l < kModuli; ++l)
      for (int j = 0; j < 3; ++j) t.c[s][l][j] = piece(s, l, j);
  for (int l = 0; l < kModuli; ++l) {
    t.m[l] = mod_at(l);
    t.shift[l] = mod_offset(l) + mod_at(l) / 2;
    t.magic[l] = mod_magic(l);
  }
  return t;
}
__device__ constexpr PieceTable kPieces = make_pieces();

// Moduli 0..11 in four groups of three, modulus 12 alone: with m a group's
// product, w_0 / m_0 + w_1 / m_1 + w_2 / m_2 = u / m, u < 3 2^27, so that 3 + 3
// multiplications per group replace 12 in sum_l w_l (M / m_l).
constexpr int kGroups = 4;
struct ModTable {
  uint32_t pair[kGroups][3];       // m / m_i inside the group
  uint32_t word[kGroups][3];       // M / m (below 2^92) in 32-bit words
  uint32_t last[4];                // M / m_12
  float inv[kGroups + 1];          // 1 / m, 1 / m_12
  float m[kModuli], rec[kModuli];  // m_l, 1 / m_l
};
constexpr ModTable make_mods() {
  ModTable t{};
  for (int l = 0; l < kModuli; ++l) {
    t.m[l] = static_cast<float>(mod_at(l));
    t.rec[l] = 1.0f / mod_at(l);
  }
  for (int g = 0; g < kGroups; ++g) {
    const long long p = static_cast<long long>(mod_at(3 * g)) * mod_at(3 * g + 1) * mod_at(3 * g + 2);
    for (int i = 0; i < 3; ++i) t.pair[g][i] = static_cast<uint32_t>(p / mod_at(3 * g + i));
    const u128 w = mod_product() / static_cast<u128>(p);
    for (int j = 0; j < 3; ++j) t.word[g][j] = static_cast<uint32_t>(w >> (32 * j));
    t.inv[g] = 1.0f / static_cast<float>(p);
  }
  const u128 w = mod_product() / mod_at(kModuli - 1);
  for (int j = 0; j < 4; ++j) t.last[j] = static_cast<uint32_t>(w >> (32 * j));
  t.inv[kGroups] = 1.0f / mod_at(kModuli - 1);
  return t;
}
__constant__ ModTable kMods = make_mods();

// ---- row norms and residues -------------------------------------------------

// sum of squares s 2^(2 e) of the entries seen, as an upper estimate: the
// float32 mantissas are truncated to 20 bits, covered by the final factor
struct NormAcc {
  int e = -5000;
  float s = 0.0f;
  int bad = 0;
  __device__ __forceinline__ void add(double x) {
    const unsigned int hi = abs_hi(x);
    const int exf = static_cast<int>(hi >> 20);
    if (exf == 0x7FF) bad = 1;
    if (exf == 0 && (hi | static_cast<unsigned int>(__double_as_longlong(x))) == 0u) return;
    // a subnormal counts as 2^-1022
    const float f = exf ? __uint_as_float(0x3F800000u | ((hi & 0xFFFFFu) << 3)) : 1.0f;
    merge(exf ? exf - 1023 : -1022, f * f);
  }
  __device__ __forceinline__ void merge(int e2, float s2) {
    const int d = e2 - e;
    if (d > 0) {
      s = d > 60 ? s2 : fmaf(s, __int_as_float((127 - 2 * d) << 23), s2);
      e = e2;
    } else if (d > -60) {
      s = fmaf(s2, __int_as_float((127 + 2 * d) << 23), s);
    }
  }
  // e_n with |row| <= 2^(e_n), or kBad
  __device__ __forceinline__ int exponent() const {
    if (bad) return kBad;
    if (s == 0.0f) return 0;
    const float t = s * 1.001f;
    const int k = (__float_as_int(t) >> 23) - 126;      // t < 2^k
    return e + ((k + 1) >> 1);
  }
};

__device__ __forceinline__ NormAcc warp_norm(NormAcc a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int e2 = __shfl_xor_sync(0xffffffffu, a.e, o);
    const float s2 = __shfl_xor_sync(0xffffffffu, a.s, o);
    a.bad |= __shfl_xor_sync(0xffffffffu, a.bad, o);
    // the same order on both partners: the larger exponent first
    NormAcc lo = a;
    if (e2 > a.e || (e2 == a.e && s2 > a.s)) { lo.e = e2; lo.s = s2; lo.merge(a.e, a.s); }
    else lo.merge(e2, s2);
    a.e = lo.e;
    a.s = lo.s;
  }
  return a;
}

// x 2^(57 - e_n) rounded to an integer (|.| <= 2^57)
__device__ __forceinline__ long long fixed_point(double x, int en) {
  const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
  const int exf = static_cast<int>((bits >> 52) & 0x7FF);
  const unsigned long long mant = (bits & 0xFFFFFFFFFFFFFull) | (exf ? (1ull << 52) : 0ull);
  const int sh = (exf ? exf : 1) - 1075 + kBits - en;
  unsigned long long q;
  if (sh >= 0) {
    q = mant << (sh > 5 ? 5 : sh);      // |x| <= 2^(e_n): sh <= 5
  } else {
    const int rs = -sh;
    q = rs >= 64 ? 0ull : ((mant >> (rs - 1)) + 1ull) >> 1;
  }
  return (bits >> 63) ? -static_cast<long long>(q) : static_cast<long long>(q);
}

// the residues of eight consecutive integers modulo mod_at(l), as bfloat16
template <int SIDE>
__device__ __forceinline__ void store_residues(const int (&a0)[8], const int (&a1)[8], const int (&a2)[8],
                                               mg_t* __restrict__ out, size_t plane) {
#pragma unroll
  for (int l = 0; l < kModuli; ++l) {
    const int c0 = kPieces.c[SIDE][l][0], c1 = kPieces.c[SIDE][l][1], c2 = kPieces.c[SIDE][l][2];
    const int m = kPieces.m[l], h = m / 2;
    uint32_t w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int x = a0[j] * c0 + a1[j] * c1 + a2[j] * c2;
      const uint32_t y = static_cast<uint32_t>(x) + kPieces.shift[l];
      const int r = static_cast<int>(y - (__umulhi(y, kPieces.magic[l]) >> 8) * static_cast<uint32_t>(m)) - h;
      // exact small-integer conversion without the conversion unit
      w[j] = __float_as_uint(__int_as_float(0x4B400000 + r) - 12582912.0f);
    }
    uint4 u;
    u.x = __byte_perm(w[0], w[1], 0x7632);
    u.y = __byte_perm(w[2], w[3], 0x7632);
    u.z = __byte_perm(w[4], w[5], 0x7632);
    u.w = __byte_perm(w[6], w[7], 0x7632);
    *reinterpret_cast<uint4*>(out + static_cast<size_t>(l) * plane) = u;
  }
}

__device__ __forceinline__ void to_pieces(double x, int en, int& a0, int& a1, int& a2) {
  const long long q = en == kBad ? 0 : fixed_point(x, en);
  a0 = static_cast<int>(q & 0xFFFFF);
  a1 = static_cast<int>((q >> 20) & 0xFFFFF);
  a2 = static_cast<int>(q >> 40);
}

// One CTA per row with contiguous K: the row is staged in shared memory, its
// norm reduced, and each thread writes the residues of eight consecutive
// elements (16-byte stores, 512 bytes per warp and plane).
constexpr int kRowThreads = 128;

template <int SIDE>
__global__ void __launch_bounds__(kRowThreads) mg_split_rows(int rows, int K, int Kp, const double* __restrict__ src,
                                                             long long rs, long long bs, mg_t* __restrict__ planes,
                                                             size_t plane, int* __restrict__ exps) {
  extern __shared__ double row_s[];
  __shared__ int we[kRowThreads / 32], wbad[kRowThreads / 32];
  __shared__ float ws[kRowThreads / 32];
  const long long q = blockIdx.x;               // batch-major row
  const long long b = q / rows, r = q - b * rows;
  const double* x = src + b * bs + r * rs;
  NormAcc acc;
  for (int k = threadIdx.x; k < Kp; k += kRowThreads) {
    const double v = k < K ? x[k] : 0.0;
    row_s[k] = v;
    acc.add(v);
  }
  acc = warp_norm(acc);
  if ((threadIdx.x & 31) == 0) {
    we[threadIdx.x >> 5] = acc.e;
    ws[threadIdx.x >> 5] = acc.s;
    wbad[threadIdx.x >> 5] = acc.bad;
  }
  __syncthreads();
  NormAcc t;
#pragma unroll
  for (int w = 0; w < kRowThreads / 32; ++w) {
    t.merge(we[w], ws[w]);
    t.bad |= wbad[w];
  }
  const int en = t.exponent();
  if (threadIdx.x == 0) exps[q] = en;
  mg_t* out = planes + static_cast<size_t>(q) * Kp;
  for (int k0 = threadIdx.x * 8; k0 < Kp; k0 += kRowThreads * 8) {
    int a0[8], a1[8], a2[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) to_pieces(row_s[k0 + j], en, a0[j], a1[j], a2[j]);
    store_residues<SIDE>(a0, a1, a2, out + k0, plane);
  }
}

// Row norms of an operand with contiguous rows index (element k of row r at
// src + k ks + r): lanes along r, eight threads per row along K.
__global__ void __launch_bounds__(256) mg_norm_cols(int rows, int K, const double* __restrict__ src, long long ks,
                                                    long long bs, int* __restrict__ exps) {
  __shared__ int se[8][32], sbad[8][32];
  __shared__ float ss[8][32];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int r = blockIdx.x * 32 + lane;
  const long long b = blockIdx.y;
  NormAcc acc;
  if (r < rows) {
    const double* x = src + b * bs + r;
    for (int k = g; k < K; k += 8) acc.add(x[k * ks]);
  }
  se[g][lane] = acc.e;
  ss[g][lane] = acc.s;
  sbad[g][lane] = acc.bad;
  __syncthreads();
  if (g == 0 && r < rows) {
    NormAcc t;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      t.merge(se[w][lane], ss[w][lane]);
      t.bad |= sbad[w][lane];
    }
    exps[b * rows + r] = t.exponent();
  }
}

// Residues of such an operand, transposed through a 64 (K) x 32 (rows) tile.
template <int SIDE>
__global__ void __launch_bounds__(256) mg_split_cols(int rows, int K, int Kp, const double* __restrict__ src,
                                                     long long ks, long long bs, mg_t* __restrict__ planes,
                                                     size_t plane, const int* __restrict__ exps) {
  __shared__ double t[64][33];
  const int r0 = blockIdx.x * 32, k0 = blockIdx.y * 64;
  const long long b = blockIdx.z;
  const double* x = src + b * bs;
  for (int i = threadIdx.x; i < 64 * 32; i += 256) {
    const int k = i >> 5, r = i & 31;
    t[k][r] = (k0 + k < K && r0 + r < rows) ? x[(k0 + k) * ks + r0 + r] : 0.0;
  }
  __syncthreads();
  const int r = threadIdx.x >> 3, g = threadIdx.x & 7;
  if (r0 + r >= rows) return;
  const long long q = b * rows + r0 + r;
  const int en = exps[q];
  int a0[8], a1[8], a2[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) to_pieces(t[g * 8 + j][r], en, a0[j], a1[j], a2[j]);
  store_residues<SIDE>(a0, a1, a2, planes + static_cast<size_t>(q) * Kp + k0 + g * 8, plane);
}

// ---- the residue products -----------------------------------------------------

constexpr int BM = 128;
constexpr int BK = 64;            // bfloat16: one 128-byte swizzle row
constexpr int kChunkBlocks = 4;   // 256 terms per exact float32 accumulation

template <int BN>
struct MgCfg {
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_BYTES = BN * BK * 2;
  static constexpr int STAGE = A_BYTES + B_BYTES;
  static constexpr int STAGES = 4 * 48 * 1024 / STAGE;     // 192 KB of stage buffers
  static constexpr int NSLOT = 512 / BN;                   // chunk accumulators in TMEM
  static constexpr int EPI = 8;                            // epilogue warps: two per 32 TMEM lanes
  static constexpr int CW = BN / 2;                        // columns per epilogue warp
  static constexpr int THREADS = 64 + 32 * EPI;
  static constexpr int OUT_ROW = 80;                       // bytes of a staged output row: 32 residues and padding
  static constexpr int OUT = EPI * 32 * OUT_ROW;
  static constexpr size_t SMEM = 1024 + static_cast<size_t>(STAGES) * STAGE + OUT + (2 * STAGES + 2 * NSLOT) * 8 + 16;
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

struct MgArgs {
  int M, N, ldn, batch;
  int nk;                // K blocks
  int ntm, ntn, ntiles;
  int abatch, bbatch;    // 1: the operand has a plane per batch entry
  uint16_t* res;         // [modulus][batch][M][ldn]
};

__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("add.rn.f32x2 %0, %1, %2;"
      : "=l"(reinterpret_cast<unsigned long long&>(d))
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
  return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<unsigned long long&>(d))
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)),
        "l"(reinterpret_cast<unsigned long long&>(c)));
  return d;
}
// x modulo m for integers |x| <= 2^24 (inv = 1 / m rounded): x - q m with q within
// 1/2 + 2^-8 of x / m, so the remainder, below m / 2 + 3, is exact
__device__ __forceinline__ float2 mod2(float2 x, float m, float inv) {
  constexpr float kRound = 12582912.0f;   // 1.5 2^23: a sum with it is an integer
  const float2 t = fma2(x, make_float2(inv, inv), make_float2(kRound, kRound));
  const float2 q = add2(t, make_float2(-kRound, -kRound));
  return fma2(q, make_float2(-m, -m), x);
}

// Persistent, one CTA per SM, output tiles of all moduli and batch entries in
// one walk: warp 0 TMA producer, warp 1 MMA issue (one chunk of 256 terms per
// TMEM slot), warps 2..9 reduce the finished chunks modulo m_l, sum them (below
// 2^15 in float32) and write the sum's residue.  The drain of a chunk has to fit
// into the MMAs' time for the next: four packed float32 instructions per two
// elements in place of two conversions (A + B, 2200 AOs, 4 vectors: 1488 -> 1396 us in
// all four products).
template <int BN>
__global__ void __launch_bounds__(MgCfg<BN>::THREADS, 1)
    mg_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, MgArgs a, int* err) {
  using C = MgCfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(base + C::STAGES * C::STAGE + C::OUT);
  uint64_t* empty = full + C::STAGES;
  uint64_t* accf = empty + C::STAGES;
  uint64_t* acce = accf + C::NSLOT;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acce + C::NSLOT);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  auto tile_of = [&](int t, int& l, int& bz, int& m0, int& n0) {
    const int per = a.ntm * a.ntn;
    const int p = t / per;
    const int r = t - p * per;
    l = p / a.batch;
    bz = p - l * a.batch;
    m0 = (r / a.ntn) * BM;
    n0 = (r % a.ntn) * BN;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < C::NSLOT; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], 32 * C::EPI);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(tmem_slot, C::NSLOT * BN);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    long long g = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
      int l, bz, m0, n0;
      tile_of(t, l, bz, m0, n0);
      const int za = l * (a.abatch ? a.batch : 1) + (a.abatch ? bz : 0);
      const int zb = l * (a.bbatch ? a.batch : 1) + (a.bbatch ? bz : 0);
      for (int kb = 0; kb < a.nk; ++kb, ++g) {
        const int s = static_cast<int>(g % C::STAGES);
        if (g >= C::STAGES && !mbar_wait(&empty[s], static_cast<uint32_t>(((g / C::STAGES) + 1) & 1), err, 1)) {
          ok = false;
          break;
        }
        uint8_t* st = base + s * C::STAGE;
        mbar_expect_tx(&full[s], C::STAGE);
        tma_load_3d(st, &tmA, &full[s], kb * BK, m0, za);
        tma_load_3d(st + C::A_BYTES, &tmB, &full[s], kb * BK, n0, zb);
      }
    }
    // the copies still in flight complete before the CTA leaves (bounded)
    for (long long q = (g > C::STAGES ? g - C::STAGES : 0); q < g; ++q)
      mbar_wait(&empty[q % C::STAGES], static_cast<uint32_t>((q / C::STAGES) & 1), err, 0) || true;
  } else if (warp == 1 && lane == 0) {
    constexpr uint32_t idesc = idesc_f32acc(1, BM, BN);
    long long g = 0, q = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
      for (int kc = 0; kc < a.nk && ok; kc += kChunkBlocks, ++q) {
        const int slot = static_cast<int>(q % C::NSLOT);
        const long long use = q / C::NSLOT;
        if (use >= 1 && !mbar_wait(&acce[slot], static_cast<uint32_t>((use + 1) & 1), err, 4)) {
          ok = false;
          break;
        }
        fence_after_sync();
        const uint32_t acc = tmem + static_cast<uint32_t>(slot * BN);
        const int kend = min(kc + kChunkBlocks, a.nk);
        for (int kb = kc; kb < kend; ++kb, ++g) {
          const int s = static_cast<int>(g % C::STAGES);
          if (!mbar_wait(&full[s], static_cast<uint32_t>((g / C::STAGES) & 1), err, 2)) {
            ok = false;
            break;
          }
          fence_after_sync();
          uint8_t* st = base + s * C::STAGE;
          const uint32_t aa = smem_u32(st), bb = smem_u32(st + C::A_BYTES);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            mma_bf16(acc, sdesc(aa + kk * 32), sdesc(bb + kk * 32), idesc, (kb > kc || kk > 0) ? 1u : 0u);
          mma_commit(&empty[s]);
        }
        if (ok) mma_commit(&accf[slot]);
      }
    }
  } else if (warp >= 2) {
    const int lane_base = 32 * (warp % 4);
    const int colh = (warp - 2) / 4;
    long long q = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
      int l, bz, m0, n0;
      tile_of(t, l, bz, m0, n0);
      const float fm = kMods.m[l], inv = kMods.rec[l];
      float2 acc[C::CW / 2];
#pragma unroll
      for (int j = 0; j < C::CW / 2; ++j) acc[j] = make_float2(0.0f, 0.0f);
      for (int kc = 0; kc < a.nk; kc += kChunkBlocks, ++q) {
        const int slot = static_cast<int>(q % C::NSLOT);
        if (!mbar_wait(&accf[slot], static_cast<uint32_t>((q / C::NSLOT) & 1), err, 3)) {
          ok = false;
          break;
        }
        fence_after_sync();
        const uint32_t trow = tmem + static_cast<uint32_t>(slot * BN + colh * C::CW) +
                              (static_cast<uint32_t>(lane_base) << 16);
#pragma unroll
        for (int c0 = 0; c0 < C::CW; c0 += 16) {
          float v[16];
          tmem_ld16(trow + c0, v);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float2 x = make_float2(v[2 * j], v[2 * j + 1]);
            acc[c0 / 2 + j] = add2(acc[c0 / 2 + j], mod2(x, fm, inv));
          }
        }
        fence_before_sync();
        mbar_arrive(&acce[slot]);
      }
      if (!ok) break;
      // A thread holds one row: 32 columns at a time go through shared memory, so that a
      // warp's store covers whole sectors of eight rows.  Storing 16 bytes of 32 rows at a
      // time held back the next tile's drain (2200 AOs, 4 vectors: 1395 -> 1191 us in the four
      // products; 1125 without any store).
      uint8_t* stage = base + C::STAGES * C::STAGE + (warp - 2) * 32 * C::OUT_ROW;
      const int row0 = m0 + lane_base, col0 = n0 + colh * C::CW;
      uint16_t* out = a.res + (static_cast<size_t>(l * a.batch + bz) * a.M) * a.ldn;
#pragma unroll
      for (int c0 = 0; c0 < C::CW; c0 += 32) {
        uint32_t p[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          float2 r = mod2(acc[c0 / 2 + j], fm, inv);
          r.x += r.x < 0.0f ? fm : 0.0f;
          r.y += r.y < 0.0f ? fm : 0.0f;
          // 0 <= r < m: the low half of the bits of 2^23 + r
          p[j] = __byte_perm(__float_as_uint(r.x + 8388608.0f), __float_as_uint(r.y + 8388608.0f), 0x5410);
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<uint4*>(stage + lane * C::OUT_ROW + 16 * j) =
              make_uint4(p[4 * j], p[4 * j + 1], p[4 * j + 2], p[4 * j + 3]);
        __syncwarp();
        const int col = col0 + c0 + 8 * (lane & 3);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = 8 * i + (lane >> 2);
          const uint4 u = *reinterpret_cast<const uint4*>(stage + r * C::OUT_ROW + 16 * (lane & 3));
          if (row0 + r < a.M && col < a.ldn)   // ldn is a multiple of 16
            *reinterpret_cast<uint4*>(out + static_cast<size_t>(row0 + r) * a.ldn + col) = u;
        }
      }
    }
  }
  fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    fence_after_sync();
    tmem_dealloc(tmem, C::NSLOT * BN);
  }
}

// ---- the remainder theorem ------------------------------------------------------

struct CrtArgs {
  int M, N, ldn, batch;
  const uint16_t* res;
  const int *ea, *eb;       // row exponents of A [abatch][M] and B [bbatch][N]
  int abatch, bbatch;
  const double *A, *B;      // sources, for flagged rows
  long long ars, aks, abs_, brs, bks, bbs;
  int K;
  MgOut out;
};

// C' (13 weighted residues) to float64: C' = sum w_l (M / m_l) - k M with k the
// nearest integer of sum w_l / m_l (|C'| <= M / 4 keeps it unambiguous), then
// the leading 53 bits, rounded, times 2^shift
__device__ __forceinline__ double crt_value(const uint32_t (&w)[kModuli], int shift) {
  unsigned long long a[4];
  const uint32_t z = w[kModuli - 1];
  float f = static_cast<float>(z) * kMods.inv[kGroups];
#pragma unroll
  for (int j = 0; j < 4; ++j) a[j] = static_cast<unsigned long long>(z) * kMods.last[j];
#pragma unroll
  for (int g = 0; g < kGroups; ++g) {
    const uint32_t u = w[3 * g] * kMods.pair[g][0] + w[3 * g + 1] * kMods.pair[g][1] + w[3 * g + 2] * kMods.pair[g][2];
    f = fmaf(static_cast<float>(u), kMods.inv[g], f);
#pragma unroll
    for (int j = 0; j < 3; ++j) a[j] += static_cast<unsigned long long>(u) * kMods.word[g][j];   // < 2^63
  }
  constexpr u128 kM = mod_product();
  const u128 sum = static_cast<u128>(a[0]) + (static_cast<u128>(a[1]) << 32) + (static_cast<u128>(a[2]) << 64) +
                   (static_cast<u128>(a[3]) << 96);
  const u128 c = sum - static_cast<u128>(__float2uint_rn(f)) * kM;
  const bool neg = static_cast<long long>(static_cast<unsigned long long>(c >> 64)) < 0;
  const u128 mag = neg ? ~c + 1 : c;
  const unsigned long long hi = static_cast<unsigned long long>(mag >> 64), lo = static_cast<unsigned long long>(mag);
  if ((hi | lo) == 0ull) return 0.0;
  const int lz = hi ? __clzll(hi) : 64 + __clzll(lo);
  const unsigned long long top = static_cast<unsigned long long>((mag << lz) >> 64);
  const unsigned long long mant = (top >> 11) + ((top >> 10) & 1ull);   // 2^52 .. 2^53
  const int e = (128 - lz) - 53 + shift;                                // value = mant 2^e
  unsigned long long bits;
  if (e + 52 >= -1022 && e + 52 <= 1022) {
    bits = (static_cast<unsigned long long>(e + 52 + 1023) << 52) + (mant - (1ull << 52));
  } else {
    bits = static_cast<unsigned long long>(__double_as_longlong(ldexp(static_cast<double>(mant), e)));
  }
  return __longlong_as_double(static_cast<long long>(bits | (neg ? 1ull << 63 : 0ull)));
}

// four consecutive columns per thread
__global__ void __launch_bounds__(128) mg_crt_kernel(CrtArgs a) {
  const int c0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (c0 >= a.N) return;
  const long long row_all = blockIdx.y + static_cast<long long>(blockIdx.z) * gridDim.y;   // batch-major row
  if (row_all >= static_cast<long long>(a.batch) * a.M) return;
  const int b = static_cast<int>(row_all / a.M), row = static_cast<int>(row_all - static_cast<long long>(b) * a.M);
  const size_t plane = static_cast<size_t>(a.batch) * a.M * a.ldn;
  const uint16_t* p = a.res + static_cast<size_t>(row_all) * a.ldn + c0;
  uint2 v[kModuli];
#pragma unroll
  for (int l = 0; l < kModuli; ++l) v[l] = __ldg(reinterpret_cast<const uint2*>(p + l * plane));
  const int ea = a.ea[(a.abatch ? static_cast<long long>(b) * a.M : 0) + row];
  const int* ebp = a.eb + (a.bbatch ? static_cast<long long>(b) * a.N : 0);
  double* crow = a.out.C + b * a.out.sC + static_cast<long long>(row) * a.out.ldc;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int col = c0 + j;
    if (col >= a.N) break;
    const int eb = ebp[col];
    double y;
    if (ea == kBad || eb == kBad) {
      const double* x1 = a.A + (a.abatch ? b * a.abs_ : 0) + static_cast<long long>(row) * a.ars;
      const double* x2 = a.B + (a.bbatch ? b * a.bbs : 0) + static_cast<long long>(col) * a.brs;
      y = 0.0;
      for (int k = 0; k < a.K; ++k) y = fma(x1[k * a.aks], x2[k * a.bks], y);
    } else {
      uint32_t w[kModuli];
#pragma unroll
      for (int l = 0; l < kModuli; ++l) {
        const uint32_t two = j < 2 ? v[l].x : v[l].y;
        w[l] = (j & 1) ? two >> 16 : two & 0xFFFFu;
      }
      y = crt_value(w, ea + eb - 2 * kBits);
    }
    if (a.out.alpha != 1.0) y *= a.out.alpha;
    if (a.out.beta != 0.0) y = fma(a.out.beta, crow[col], y);
    if (a.out.X)
      y = fma(a.out.eps[a.out.o + col] - a.out.eps[row], a.out.X[b * a.out.sC + static_cast<long long>(row) * a.out.ldc + col], y);
    crow[col] = y;
  }
}

CUtensorMap make_map(const mg_t* ptr, int Kp, int rows, long long planes, int box_rows) {
  CUtensorMap m;
  cuuint64_t dims[3] = {static_cast<cuuint64_t>(Kp), static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(planes)};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(Kp) * 2, static_cast<cuuint64_t>(Kp) * rows * 2};
  cuuint32_t box[3] = {static_cast<cuuint32_t>(BK), static_cast<cuuint32_t>(box_rows), 1};
  cuuint32_t estr[3] = {1, 1, 1};
  if (reinterpret_cast<uintptr_t>(ptr) & 15) throw Error(XS_EINVAL, "residue planes not 16-byte aligned");
  CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<mg_t*>(ptr), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw Error(XS_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string(r) + ")");
  return m;
}

int num_sms() {
  static const int n = [] {
    int dev = 0, count = 0;
    XS_CUDA(cudaGetDevice(&dev));
    XS_CUDA(cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev));
    return count;
  }();
  return n;
}

template <int BN>
void launch_mg(cudaStream_t s, const MgOperand& A, const MgOperand& B, MgArgs a, int* err) {
  using C = MgCfg<BN>;
  static std::atomic<unsigned long long> smem{0};
  allow_smem(smem, mg_kernel<BN>, C::SMEM);
  const int Kp = mg_kp(A.K);
  const CUtensorMap ta = make_map(A.planes, Kp, A.rows, static_cast<long long>(kModuli) * A.batch, BM);
  const CUtensorMap tb = make_map(B.planes, Kp, B.rows, static_cast<long long>(kModuli) * B.batch, BN);
  a.nk = Kp / BK;
  a.ntm = (a.M + BM - 1) / BM;
  a.ntn = (a.N + BN - 1) / BN;
  a.ntiles = kModuli * a.batch * a.ntm * a.ntn;
  const int grid = std::min(a.ntiles, num_sms());
  mg_kernel<BN><<<grid, C::THREADS, C::SMEM, s>>>(ta, tb, a, err);
  XS_CHECK_LAUNCH();
}

template <int SIDE>
void split_side(cudaStream_t s, const MgOperand& op, MgPlanes& p) {
  const int Kp = mg_kp(op.K);
  const long long nrow = static_cast<long long>(op.batch) * op.rows;
  const size_t plane = static_cast<size_t>(nrow) * Kp;
  if (op.ks == 1) {
    const size_t smem = sizeof(double) * Kp;
    static std::atomic<unsigned long long> allowed{0};
    allow_smem(allowed, mg_split_rows<SIDE>, sizeof(double) * kMgMaxK);
    mg_split_rows<SIDE><<<static_cast<unsigned>(nrow), kRowThreads, smem, s>>>(
        op.rows, op.K, Kp, op.src, op.rs, op.bs, p.planes.get(), plane, p.exps.get());
    XS_CHECK_LAUNCH();
  } else {
    const unsigned gx = (op.rows + 31) / 32;
    mg_norm_cols<<<dim3(gx, op.batch), 256, 0, s>>>(op.rows, op.K, op.src, op.ks, op.bs, p.exps.get());
    XS_CHECK_LAUNCH();
    mg_split_cols<SIDE><<<dim3(gx, Kp / 64, op.batch), 256, 0, s>>>(op.rows, op.K, Kp, op.src, op.ks, op.bs,
                                                                   p.planes.get(), plane, p.exps.get());
    XS_CHECK_LAUNCH();
  }
}

}  // namespace

void mg_split(cudaStream_t s, int side, MgOperand& op, MgPlanes& p) {
  if (op.K < 1 || op.K > kMgMaxK || op.rows < 1 || op.batch < 1 || (op.rs != 1 && op.ks != 1))
    throw Error(XS_EINVAL, "mg_split: operand shape");
  p.planes.ensure(mg_plane_count(op.rows, op.K, op.batch));
  p.exps.ensure(static_cast<size_t>(op.batch) * op.rows);
  ProfScope ps(s, "mg_split", static_cast<double>(op.batch) * op.rows * op.K * (8.0 + 2.0 * kModuli), 0.0);
  if (side == 0) split_side<0>(s, op, p);
  else split_side<1>(s, op, p);
  op.planes = p.planes.get();
  op.exps = p.exps.get();
}

void mg_product(cudaStream_t s, const MgOperand& A, const MgOperand& B, int batch, const MgOut& out, MgWork& w,
                int* d_err) {
  const int M = A.rows, N = B.rows;
  if (A.K != B.K || (A.batch != 1 && A.batch != batch) || (B.batch != 1 && B.batch != batch))
    throw Error(XS_EINVAL, "mg_product: operand shapes");
  const int ldn = mg_ldn(N);
  w.res.ensure(static_cast<size_t>(kModuli) * batch * M * ldn);
  MgArgs a{};
  a.M = M;
  a.N = N;
  a.ldn = ldn;
  a.batch = batch;
  a.abatch = A.batch > 1 ? 1 : 0;
  a.bbatch = B.batch > 1 ? 1 : 0;
  a.res = w.res.get();
  {
    ProfScope ps(s, "mg_gemm", 0.0, 2.0 * kModuli * M * N * static_cast<double>(A.K) * batch);
    // waves of 256-wide tiles against waves of 128-wide ones, which cost 0.7 of them each
    // (four products, 128-wide -> 256-wide where the line is crossed: 561 AOs, 20 vectors
    // 375 -> 312 us, 600 AOs, 10 vectors 195 -> 179)
    const auto waves = [&](int bn) {
      const long long t = static_cast<long long>(kModuli) * batch * ((M + BM - 1) / BM) * ((N + bn - 1) / bn);
      return static_cast<double>((t + num_sms() - 1) / num_sms());
    };
    if (waves(256) <= 0.7 * waves(128)) launch_mg<256>(s, A, B, a, d_err);
    else launch_mg<128>(s, A, B, a, d_err);
  }
  CrtArgs c{};
  c.M = M;
  c.N = N;
  c.ldn = ldn;
  c.batch = batch;
  c.res = w.res.get();
  c.ea = A.exps;
  c.eb = B.exps;
  c.abatch = a.abatch;
  c.bbatch = a.bbatch;
  c.A = A.src;
  c.B = B.src;
  c.ars = A.rs;
  c.aks = A.ks;
  c.abs_ = A.bs;
  c.brs = B.rs;
  c.bks = B.ks;
  c.bbs = B.bs;
  c.K = A.K;
  c.out = out;
  const long long rows = static_cast<long long>(batch) * M;
  const unsigned gy = static_cast<unsigned>(std::min<long long>(rows, 32768));
  const dim3 grid(static_cast<unsigned>((N + 511) / 512), gy, static_cast<unsigned>((rows + gy - 1) / gy));
  ProfScope ps(s, "mg_crt", static_cast<double>(rows) * N * (2.0 * kModuli + 8.0), 0.0);
  mg_crt_kernel<<<grid, 128, 0, s>>>(c);
  XS_CHECK_LAUNCH();
}

}  // namespace xs
