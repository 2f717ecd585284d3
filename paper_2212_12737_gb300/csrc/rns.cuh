// Residue-number products on the BF16 tensor cores: FP64-class contractions of GDML_OZAKI contexts.
//
// The scheme is the modular form of Ozaki's error-free products (Ozaki, Uchino and Imamura,
// "Ozaki Scheme II: a GEMM-oriented emulation of floating-point matrix multiplication using an
// integer modular technique", 2025):
//
//   * row r of A and row c of B (both K entries) are scaled by powers of two and rounded to
//     integers x, y with |x|_2 < 2^tA, |y|_2 < 2^tB, so |x . y| < 2^(tA + tB) < P / 2 with
//     P = prod p_i over NM pairwise coprime moduli p_i <= 361;
//   * for each modulus the centred residues (|r| <= 181, exact in BF16) are multiplied on the
//     tensor cores; a sum over 512 K entries is an integer below 2^24, exact in the FP32
//     accumulator, and is reduced mod p_i before the next 512 entries are added;
//   * x . y follows from its NM residues by the Chinese remainder theorem:
//     x . y / P = frac(sum_i rho_i / p_i) with rho_i = (x . y) (P / p_i)^-1 mod p_i (the inverse
//     factor is folded into one operand's residues), summed in 76-bit fixed point.
//
// 14 products of residues up to 181 beat 13 of residues up to 256, which allow 256 exact K entries
// only: twice the reductions, 1.10 against 0.89 ms for T and U at n = 630k (zero operands).
// Against the sliced form (28 slice pairs, oz.cuh): nothing is truncated but the operands' rounding,
// and the matvec's error fell from 4.9-8.3e-15 to 3.3-4.7e-15 over N = 9 .. 48, M = 60 .. 5000
// (FP64 reference).  The product of P is chosen for 57 bits per operand: with 12 moduli up to 512
// (53 bits) the error rose to 2.1e-14 at M = 5000.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>

#include <vector>

#include "common.cuh"

namespace gdml {
namespace rns {

constexpr int kMaxMod = 14;
// pairwise coprime (361 = 19^2, 358 = 2 179, 355 = 5 71, 351 = 3^3 13, 343 = 7^3, 341 = 11 31, the
// others prime), largest first; residues reach at most 181
constexpr int kMods[kMaxMod] = {361, 359, 358, 355, 353, 351, 349, 347, 343, 341, 337, 331, 317, 313};

constexpr int kMvMods = 14;  // the matvec's: P = 2^117.9
constexpr int kMvBits = 57;  // both operands: 2^114 < P / 2
constexpr int kChunk = 512;  // K entries whose products of residues sum exactly in FP32
constexpr int kSumChunks = 149;  // chunks whose residues + 256 (at most 437 each) a 16-bit sum holds
constexpr int kDigit = 14;  // residues are formed from digits of 14 bits, four per integer
constexpr int kBad = -100000;  // scale of a row that holds a NaN or an infinity

template <int NM>
struct Crt {
  float p[NM], inv[NM];       // modulus, 1 / p
  float c1[NM], c2[NM], c3[NM];  // 2^14, 2^28, 2^42 mod p, centred
  int m[NM], fold[NM];           // modulus; (P / p_i)^-1 mod p_i
  uint32_t w2[NM], w1[NM], w0[NM];  // round(2^76 / p_i) = w2 2^44 + w1 2^12 + w0
  uint32_t o2, o1, o0;        // 256 sum_i round(2^76 / p_i) mod 2^76, the same limbs
  float pih, pil;             // P = 2^pexp (pih + pil), 1 <= pih < 2
  float ipih, ipil;           // 1 / (pih + pil)
  int pexp;
  constexpr Crt() : p(), inv(), c1(), c2(), c3(), m(), fold(), w2(), w1(), w0(), o2(0), o1(0), o0(0), pih(0), pil(0), ipih(0), ipil(0), pexp(0) {
    unsigned __int128 off = 0;
    for (int i = 0; i < NM; ++i) {
      const int n = kMods[i];
      m[i] = n;
      p[i] = (float)n;
      inv[i] = 1.0f / (float)n;
      long long e = 1;
      for (int b = 0; b < kDigit; ++b) e = e * 2 % n;
      const long long e2 = e * e % n, e3 = e2 * e % n;
      c1[i] = (float)(2 * e > n ? e - n : e);
      c2[i] = (float)(2 * e2 > n ? e2 - n : e2);
      c3[i] = (float)(2 * e3 > n ? e3 - n : e3);
      long long q = 1;
      for (int j = 0; j < NM; ++j)
        if (j != i) q = q * kMods[j] % n;
      int f = 1;
      while (q * f % n != 1) ++f;
      fold[i] = f;
      const unsigned __int128 one = (unsigned __int128)1 << 76;
      const unsigned __int128 w = (one + n / 2) / n;
      w2[i] = (uint32_t)(w >> 44);
      w1[i] = (uint32_t)(w >> 12);
      w0[i] = (uint32_t)(w & 0xFFF);
      off += 256 * w;
    }
    o2 = (uint32_t)(off >> 44);
    o1 = (uint32_t)(off >> 12);
    o0 = (uint32_t)(off & 0xFFF);
    // P in double-double: products of integers below 2^9, normalised to [1, 2)
    double h = 1.0, l = 0.0;
    for (int i = 0; i < NM; ++i) {
      const double f = (double)kMods[i];
      // split h so that both partial products are exact
      const double t = h * 134217729.0, hh = t - (t - h), hl = h - hh;
      const double a = hh * f, b = hl * f + l * f;
      h = a + b;
      l = b - (h - a);
      while (h >= 2.0) {
        h *= 0.5;
        l *= 0.5;
        ++pexp;
      }
    }
    pih = (float)h;
    pil = (float)((h - (double)pih) + l);
    const double inv_p = 1.0 / (h + l);
    ipih = (float)inv_p;
    ipil = (float)(inv_p - (double)ipih);
  }
};

// two independent entries per instruction (f32x2); a - b as one fused multiply-add by -1 (exact)
constexpr float kMagic = 12582912.f;  // 1.5 2^23: adding it rounds |x| < 2^22 to an integer
__device__ __forceinline__ float2 f2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f), a); }
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// centred residues of two integers given by digits, modulo p_i, as packed BF16.  Every product and
// sum is an integer below 2^24; the quotient's rounding error (< 0.002) leaves |r| <= p / 2 + 1/2.
template <int NM>
__device__ __forceinline__ uint32_t residue2(const Crt<NM>& C, int i, const float2 (&d)[4]) {
  float2 t = p_fma(d[1], f2(C.c1[i]), d[0]);
  t = p_fma(d[2], f2(C.c2[i]), t);
  t = p_fma(d[3], f2(C.c3[i]), t);
  const float2 q = p_add(p_fma(t, f2(C.inv[i]), f2(kMagic)), f2(-kMagic));
  const float2 r = p_fma(q, f2(-C.p[i]), t);
  const __nv_bfloat162 b = __floats2bfloat162_rn(r.x, r.y);
  return *reinterpret_cast<const uint32_t*>(&b);
}

}  // namespace rns

// One operand as residues: NM planes of rows x Kp BF16 (K-major, zero padded), and the power of
// two each row was scaled by (value = integer 2^-s)
struct RnsOperand {
  __nv_bfloat16* d = nullptr;
  int* s = nullptr;
  int64_t rows = 0, K = 0, Kp = 0;
  CUtensorMap map;
};

struct RnsMatvec {
  bool ready = false;
  int64_t M = 0;   // rows a (the geometries)
  int64_t MB = 0;  // training-side rows: M, or M S with S permutational symmetries (row b S + q)
  int N = 0, D = 0;
  int S = 1;
  const int* pis = nullptr;     // S x D descriptor-entry permutations (S > 1)
  const double* XcB = nullptr;  // MB x D centred training-side descriptors
  RnsOperand Xc1;  // T = Xc W^T: A, fixed
  RnsOperand W1;   //             B, per matvec
  RnsOperand A2;   // U = A W + beta Xc: A of the first product, fixed
  RnsOperand WT2;  //                    B of the first product, per matvec
  RnsOperand B2;   //                    A of the second (beta), per panel
  RnsOperand XT2;  //                    B of the second, fixed
  double* W = nullptr;      // M x D, MB x D: FP64 projections (S > 1)
  double* WB = nullptr;
  double* t = nullptr;
  int Dp = 0;               // D rounded up to even: rows of the float-pair arrays below, padded with zeros
  float2* G3 = nullptr;     // [M][3][Dp] Jacobian factors
  uint32_t* ij = nullptr;   // Dp: 3 i | 3 j << 16 of pair p
  float2* Wf = nullptr;     // [M][Dp] the projection (S = 1)
  unsigned* colmax = nullptr;  // copies x Dp: largest |W| of each descriptor (float bits), zero between matvecs
  float2* Xc2 = nullptr;    // [M][Dp] the centred descriptors
  float2* t2 = nullptr;     // t_b = xc_b . w_b over the mantissa of P
  float2* S2 = nullptr;     // M x ldT: c^2 S_ab times the mantissa of P
  int64_t P = 0;            // rows per panel: T, beta and U exist for these only (M, or a multiple of 256)
  uint16_t* Tp = nullptr;   // [slab][modulus][P][ldT] residues of T: sums over the chunks of residue + 256
  uint16_t* Up = nullptr;   // [slab of A W | slab of beta Xc][modulus][P][ldU]
  float2* JX = nullptr;     // 3 N M: J_a^T xc_a
  int64_t ldT = 0, ldU = 0;
  int bn1 = 256, bn2 = 256;     // columns per tile of the two products
  int g1 = 1, g2 = 1;           // 512-entry K chunks per unit (gdml_autotune)
  int64_t nch1 = 0, nch2 = 0;   // chunks of D and of MB
  int cap1 = 1, cap2 = 1;       // slabs (K groups) that Tp and Up hold
  int* err = nullptr;
  std::vector<void*> allocs;
};

// As oz_setup (oz.cuh): G (M x D x 3), Xc (M x D), A, S (M x MB; A's row stride ldA), XcB (MB x D)
gdml_status rns_setup(RnsMatvec& r, int64_t M, int N, int D, const double* G, const double* Xc, const double* A, int64_t ldA,
                      const double* S, double c, cudaStream_t st, int Ssym, const int* pis, const double* XcB);
// out = K v (+ lambda v); G, Xc: the FP64 Jacobian factors and centred descriptors (used when S > 1)
gdml_status rns_matvec(RnsMatvec& r, const double* G, const double* Xc, const double* v, double* out, int add_lambda,
                       double lam, cudaStream_t st);
gdml_status rns_check(RnsMatvec& r, cudaStream_t st);
void rns_destroy(RnsMatvec& r);
// K chunks per unit: the value used for a requested one, given the slabs that the buffers hold
int rns_chunks(int64_t nch, int g, int cap);
cudaError_t set_wait_limit_rns(uint32_t polls);

// ---- the products of the OZAKI preconditioner build: A B^T mod each p_i.  Operands: NM planes of
// Ra (Rb) rows x Kp BF16 residues, Kp a multiple of 64, neither with the CRT factor folded in
enum { RNS_FULL = 0, RNS_TRI = 1, RNS_LOWER = 2 };
struct RnsProduct {
  const __nv_bfloat16 *A = nullptr, *B = nullptr;
  int64_t Ra = 0, Rb = 0, Kp = 0;
  int64_t M = 0, N = 0;  // outputs: rows row0 .. row0 + M of A against rows 0 .. N of B
  int64_t row0 = 0;      // a multiple of 256 (0 unless RNS_LOWER)
  int shape = RNS_FULL;  // RNS_TRI: row c of B is zero past entry c; RNS_LOWER: only columns <= the row are wanted
  uint16_t* out = nullptr;  // [slab][modulus][M][ldo]: sums over the slab's chunks of residue + 256
  int64_t ldo = 0;          // a multiple of 16
  int bn = 256, chunks = 1, slabs = 1;  // columns per tile, chunks per unit, K groups
};
// tile and K groups for a product of these sizes (at most `cap` groups unless a unit can't hold the chunks)
void rns_product_shape(RnsProduct& q, int cap);
gdml_status rns_product(RnsProduct& q, int* err, cudaStream_t st);

// C = A B^T for a tall A (n x K, column-major: entry (r, j) at A[j n + r]) and B (NB x K, row-major,
// row stride ldb; lower triangular when tri_b, so K entries past each row's diagonal are skipped).
// rowsq = false: C stored column-major, out[c n + r] (and as FP32 at out32[c n + r] when out32 is not
// null); out may alias A.  rowsq = true: out[r] = sum_c C[r][c]^2 (n doubles).  Synchronises the stream.
gdml_status rns_gemm_tall(const double* A, int64_t n, int64_t K, const double* B, int64_t NB, int64_t ldb, bool tri_b,
                          bool rowsq, double* out, float* out32, cudaStream_t st);
// lower triangle of C = X X^T (k x k, FP64, row stride ldc) for X (k x K, row stride ldx).
// Synchronises the stream.
gdml_status rns_syrk_lower(const float* X, int64_t k, int64_t K, int64_t ldx, double* C, int64_t ldc, cudaStream_t st);
gdml_status rns_syrk_lower(const double* X, int64_t k, int64_t K, int64_t ldx, double* C, int64_t ldc, cudaStream_t st);

}  // namespace gdml
