// Residue-number matvec of GDML_OZAKI contexts (see rns.cuh for the scheme).  One matvec is six
// kernels: projection (W = J v, its row residues), column residues of W, the products' residues
// T, beta (T from its residues, beta's residues), U, back-projection; the last four per panel of rows.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "kernels.cuh"
#include "rns.cuh"
#include "tc.cuh"
#include "tc_gemm.cuh"

namespace gdml {

namespace {

using bf16 = __nv_bfloat16;
using rns::f2;
using rns::kMagic;
using rns::p_add;
using rns::p_fma;
using rns::p_mul;
using rns::p_sub;
using rns::residue2;

// ------------------------------------------------------------ double-float helpers
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {  // |a| >= |b| or a == 0
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}
// (h, l) += (bh, bl)
__device__ __forceinline__ void df_add(float& h, float& l, float bh, float bl) {
  float s, e;
  two_sum(h, bh, s, e);
  e = __fadd_rn(e, __fadd_rn(l, bl));
  fast_two_sum(s, e, h, l);
}
// (h, l) = (ah, al) (bh, bl)
__device__ __forceinline__ void df_mul(float ah, float al, float bh, float bl, float& h, float& l) {
  const float p = __fmul_rn(ah, bh);
  float e = fmaf(ah, bh, -p);
  e = fmaf(ah, bl, e);
  e = fmaf(al, bh, e);
  fast_two_sum(p, e, h, l);
}
__device__ __forceinline__ float2 split_d(double x) {
  const float hi = __double2float_rn(x);
  return make_float2(hi, __double2float_rn(x - (double)hi));
}
__device__ __forceinline__ float2 as_pair(double x) { return split_d(x); }
__device__ __forceinline__ float2 as_pair(float2 x) { return x; }
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((127 + k) << 23); }
// x 2^e, exact unless the result leaves the FP32 range; NaN for the scale of a bad row
__device__ __noinline__ float scale2_slow(float x, int e) {
  if (e > 4096 || e < -4096) return __int_as_float(0x7fffffff);
  while (e > 127) {
    x *= pow2f(127);
    e -= 127;
  }
  while (e < -126) {
    x *= pow2f(-126);
    e += 126;
  }
  return x * pow2f(e);
}

// Scale of a row whose largest magnitude has the bits m and whose K entries the other operand's
// row meets: 2^s |row|_2 <= 2^s m sqrt(K) < 2^bits.  NaN and infinity have the largest bits.
__device__ __forceinline__ int row_scale(unsigned m, float sqrtK, int bits) {
  if (m >= 0x7f800000u) return rns::kBad;
  const float f = __uint_as_float(m);
  if (f == 0.f) return 0;
  int ef = 0, ek = 0;
  const float pr = frexpf(f, &ef) * frexpf(sqrtK, &ek);  // < 1
  int e = ef + ek;
  if (pr < 0.49999f) --e;
  return bits - e;
}

// ------------------------------------------------------------ packed FP32 pairs (rns.cuh)
struct df2 {  // two double-float numbers h + l
  float2 h, l;
};
// in memory: hi, lo, hi, lo
__device__ __forceinline__ df2 as_df2(float4 x) { return {make_float2(x.x, x.z), make_float2(x.y, x.w)}; }
__device__ __forceinline__ float4 as_f4(df2 x) { return make_float4(x.h.x, x.l.x, x.h.y, x.l.y); }
__device__ __forceinline__ df2 pair2(float2 a, float2 b) {  // from two (hi, lo) pairs
  return {make_float2(a.x, b.x), make_float2(a.y, b.y)};
}
__device__ __forceinline__ df2 p_fast_two_sum(float2 a, float2 b) {  // |a| >= |b| or a == 0
  const float2 s = p_add(a, b);
  return {s, p_sub(b, p_sub(s, a))};
}
__device__ __forceinline__ df2 p_df_add(df2 a, df2 b) {
  const float2 s = p_add(a.h, b.h);
  const float2 bb = p_sub(s, a.h);
  const float2 e = p_add(p_sub(a.h, p_sub(s, bb)), p_sub(b.h, bb));
  return p_fast_two_sum(s, p_add(e, p_add(a.l, b.l)));
}
__device__ __forceinline__ df2 p_df_sub(df2 a, df2 b) {
  const float2 s = p_sub(a.h, b.h);
  const float2 bb = p_sub(s, a.h);  // -(b.h) as far as it entered s
  const float2 e = p_sub(p_sub(a.h, p_sub(s, bb)), p_add(b.h, bb));
  return p_fast_two_sum(s, p_add(e, p_sub(a.l, b.l)));
}
__device__ __forceinline__ df2 p_df_mul(df2 a, df2 b) {
  const float2 p = p_mul(a.h, b.h);
  float2 e = p_fma(a.h, b.h, p_mul(p, f2(-1.f)));
  e = p_fma(a.h, b.l, e);
  e = p_fma(a.l, b.h, e);
  return p_fast_two_sum(p, e);
}

// ------------------------------------------------------------ integers to residues
// Two entries (already scaled) rounded to integers of at most 57 bits and cut into digits of 14 bits:
// x = d[0] + d[1] 2^14 + d[2] 2^28 + d[3] 2^42, |d[0..2]| <= 2^13, |d[3]| <= 2^15.  Each step is
// exact: h - d 2^q is a multiple of h's ulp and either 0 or at least that ulp, so Fast2Sum
// renormalises the pair.
__device__ __forceinline__ void digits2(df2 x, float2 (&d)[4]) {
#pragma unroll
  for (int q = 3; q >= 1; --q) {
    const float up = (float)(1ull << (rns::kDigit * q));
    d[q] = p_add(p_fma(x.h, f2(1.f / up), f2(kMagic)), f2(-kMagic));
    x = p_fast_two_sum(p_fma(d[q], f2(-up), x.h), x.l);
  }
  // the last digit: h is below 2^13 and l below h's ulp
  d[0] = p_add(p_add(p_add(x.h, x.l), f2(kMagic)), f2(-kMagic));
}

// The fraction (x . y) / P of two neighbouring outputs, in units of 2^-43, from words of two 16-bit
// sums (each over at most rns::kSumChunks chunks of residue + 256, so that neither field carries into
// the other); several groups of chunks are added here, in wider sums.
struct CrtSum {
  uint64_t a1[2] = {0, 0}, a0[2] = {0, 0};
  uint32_t a2[2] = {0, 0};
  template <int NM>
  __device__ __forceinline__ void add(const rns::Crt<NM>& C, const uint32_t (&w)[NM]) {
    uint32_t s0[2] = {0, 0};  // (14 fields times 12 bits stay below 2^32)
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      const uint32_t u[2] = {w[i] & 0xffffu, w[i] >> 16};
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        s0[v] += u[v] * C.w0[i];
        a1[v] += (uint64_t)u[v] * C.w1[i];
        a2[v] += u[v] * C.w2[i];
      }
    }
#pragma unroll
    for (int v = 0; v < 2; ++v) a0[v] += s0[v];
  }
  template <int NM>
  __device__ __forceinline__ df2 fraction(const rns::Crt<NM>& C, uint32_t chunks) const {
    // minus the offset of 256 per residue and chunk
    const uint64_t off = ((uint64_t)(chunks * C.o2) << 32) + (uint64_t)chunks * C.o1;
    float g2[2], g1[2], g0[2];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int64_t f = (int64_t)((((uint64_t)a2[v] << 32) + a1[v]) - off) + (((int64_t)a0[v] - (int64_t)(chunks * C.o0)) >> 12);
      // three digits of 21, 22 and 21 bits, each exact in FP32
      g2[v] = __int_as_float(0x4b400000 + (int)(f >> 43));
      g1[v] = __uint_as_float(0x4b000000u | ((uint32_t)(f >> 21) & 0x3fffffu));
      g0[v] = __uint_as_float(0x4b000000u | ((uint32_t)f & 0x1fffffu));
    }
    const float2 h2 = p_add(make_float2(g2[0], g2[1]), f2(-kMagic)), h1 = p_add(make_float2(g1[0], g1[1]), f2(-8388608.f)),
                 h0 = p_add(make_float2(g0[0], g0[1]), f2(-8388608.f));
    df2 r = p_fast_two_sum(p_mul(h2, f2(4194304.f)), h1);  // units of 2^21 2^-64
    return p_fast_two_sum(r.h, p_fma(h0, f2(4.76837158203125e-7f), r.l));
  }
};
template <int NM>
__device__ __forceinline__ df2 crt_fraction(const rns::Crt<NM>& C, const uint32_t (&w)[NM], uint32_t chunks) {
  CrtSum s;
  s.add(C, w);
  return s.fraction(C, chunks);
}

// (h, l) 2^e for each entry
__device__ __forceinline__ df2 p_scale(df2 x, int e0, int e1) {
  if ((unsigned)(e0 + 126) <= 253u && (unsigned)(e1 + 126) <= 253u) {
    const float2 f = make_float2(pow2f(e0), pow2f(e1));
    return {p_mul(x.h, f), p_mul(x.l, f)};
  }
  return {make_float2(scale2_slow(x.h.x, e0), scale2_slow(x.h.y, e1)),
          make_float2(scale2_slow(x.l.x, e0), scale2_slow(x.l.y, e1))};
}

// ------------------------------------------------------------ operand kernels
// Largest bits of |x| over the CTA's threads (256 at most)
__device__ __forceinline__ unsigned cta_max_bits(unsigned m, unsigned* red) {
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  m = red[0];
  for (int w = 1; w < (int)blockDim.x >> 5; ++w) m = max(m, red[w]);
  return m;
}

__device__ __forceinline__ unsigned abs_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }

// The columns' largest magnitudes are kept in kColCopies arrays, row a's CTA raising the (a mod
// kColCopies)-th: with one array the CTAs of a round, which all see it cleared, queue up behind one
// another's atomics (projection at M = 1,000, D = 210: 22.8 us, 8.6 with 16).
constexpr int kColCopies = 16;

// *p = max(*p, b) among all CTAs.  Most entries do not raise it: a plain look first (a stale value is
// only smaller) spares L2 the atomics, which all fall on the same few lines
__device__ __forceinline__ void raise_max(unsigned* p, unsigned b) {
  if (b > __ldcg(p)) atomicMax(p, b);
}

// residues of two consecutive entries of a row scaled by 2^s, to d[i stride] for every modulus
template <int NM>
__device__ __forceinline__ void store2(df2 x, int s, bf16* __restrict__ d, int64_t stride) {
  constexpr rns::Crt<NM> C{};
  float2 dg[4];
  digits2(p_scale(x, s, s), dg);
#pragma unroll
  for (int i = 0; i < NM; ++i) *reinterpret_cast<uint32_t*>(d + i * stride) = residue2<NM>(C, i, dg);
}

// Fixed operands (set-up): rows of an FP64 matrix, rounded to integers of `bits` bits in FP64 and
// reduced in integer arithmetic; the residues carry the CRT factor.  One CTA per row.
template <int NM>
__global__ void __launch_bounds__(256) rns_fixed_rows_kernel(const double* __restrict__ X, int64_t ldx, int64_t K,
                                                             int64_t rows, int64_t Kp, int bits, bf16* __restrict__ d,
                                                             int* __restrict__ sc) {
  __shared__ unsigned red[8];
  const int64_t row = blockIdx.x;
  unsigned m = 0;
  for (int64_t k = threadIdx.x; k < K; k += 256) m = max(m, abs_bits(__double2float_ru(fabs(X[row * ldx + k]))));
  m = cta_max_bits(m, red);
  const int s = row_scale(m, sqrtf((float)K) * 1.0001f, bits);
  if (threadIdx.x == 0) sc[row] = s;
  constexpr rns::Crt<NM> C{};
  for (int64_t k = threadIdx.x; k < K; k += 256) {
    const long long x = s == rns::kBad ? 0 : llrint(scalbn(X[row * ldx + k], s));
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      const int p = C.m[i];
      int r = (int)(x % p) * C.fold[i] % p;
      if (2 * r > p) r -= p;
      if (2 * r < -p) r += p;
      d[((int64_t)i * rows + row) * Kp + k] = __float2bfloat16_rn((float)r);
    }
  }
}

// Rows of an FP64 matrix per matvec (the symmetric kernel's W on the training side): row residues,
// the columns' largest magnitudes, t as a float pair.  One CTA per row.
template <int NM>
__global__ void __launch_bounds__(256) rns_rows_kernel(const double* __restrict__ X, int64_t rows, int K, int64_t Kp,
                                                       int bits, bf16* __restrict__ d, int* __restrict__ sc,
                                                       unsigned* __restrict__ colmax, const double* __restrict__ t,
                                                       float2* __restrict__ t2) {
  __shared__ unsigned red[8];
  constexpr rns::Crt<NM> C{};
  const int64_t row = blockIdx.x;
  unsigned m = 0;
  colmax += (row % kColCopies) * ((K + 1) & ~1);
  for (int k = threadIdx.x; k < K; k += 256) {
    const unsigned b = abs_bits(__double2float_ru(fabs(X[row * K + k])));
    raise_max(&colmax[k], b);
    m = max(m, b);
  }
  m = cta_max_bits(m, red);
  const int s = row_scale(m, sqrtf((float)K) * 1.0001f, bits);
  if (threadIdx.x == 0) {
    sc[row] = s;
    t2[row] = split_d(t[row]);  // (t in units of P's mantissa: see rns_proj_kernel)
    float h, l;
    df_mul(t2[row].x, t2[row].y, C.ipih, C.ipil, h, l);
    t2[row] = make_float2(h, l);
  }
  for (int k = 2 * threadIdx.x; k < K; k += 512) {
    const float2 x0 = split_d(X[row * K + k]);
    const float2 x1 = k + 1 < K ? split_d(X[row * K + k + 1]) : make_float2(0.f, 0.f);
    store2<NM>(pair2(x0, x1), s, d + row * Kp + k, rows * Kp);
  }
}

// The projection W_a = J_a v_a, t_a = xc_a . w_a (the matvec's first step, Sec. 2.1) in
// double-float arithmetic (GB300's FP64 pipe runs at 1/64 of the FP32 rate), with row a's residues
// and the columns' largest magnitudes.  t is stored divided by the mantissa of P: T comes from its
// residues in those units.  One CTA per geometry; a thread takes two consecutive descriptors at a
// time in packed arithmetic (G3, Xc2, ij are laid out for that, their padding is zero), w staged in
// shared memory between the row's maximum and its residues.
template <int NM>
__global__ void __launch_bounds__(512) rns_proj_kernel(const float4* __restrict__ G3, const float4* __restrict__ Xc2,
                                                       const uint2* __restrict__ ij, const double* __restrict__ v,
                                                       int64_t M, int N, int Dp, float rootD, float4* __restrict__ Wf,
                                                       float2* __restrict__ t2, int64_t Kp, int bits,
                                                       bf16* __restrict__ d, int* __restrict__ sc,
                                                       unsigned* __restrict__ colmax) {
  extern __shared__ __align__(16) float2 sh[];  // Dp: w_a; 3N: v_a
  __shared__ unsigned red[16];
  __shared__ float2 red2[16];
  constexpr rns::Crt<NM> C{};
  const int64_t a = blockIdx.x;
  const int tid = threadIdx.x, B = 3 * N, nt = blockDim.x, H = Dp >> 1;
  float4* sw = reinterpret_cast<float4*>(sh);
  float2* sv = sh + Dp;
  const float4* Ga = G3 + a * 3 * H;
  const float4* Xa = Xc2 + a * H;
  colmax += (a % kColCopies) * Dp;
  // the first descriptors' operands in one round of loads with v
  const int q0 = min(tid, H - 1);
  float4 g[3] = {Ga[q0], Ga[H + q0], Ga[2 * H + q0]}, x = Xa[q0];
  uint2 pr = ij[q0], cm = __ldcg(reinterpret_cast<const uint2*>(colmax) + q0);
  grid_trigger();
  for (int l = tid; l < B; l += nt) sv[l] = split_d(v[a * B + l]);
  __syncthreads();
  df2 t{f2(0.f), f2(0.f)};
  unsigned m = 0;
  for (int q = tid; q < H; q += nt) {  // descriptors 2q, 2q + 1
    if (q != tid) {
      g[0] = Ga[q];
      g[1] = Ga[H + q];
      g[2] = Ga[2 * H + q];
      x = Xa[q];
      pr = ij[q];  // 3 i | 3 j << 16 of each
      cm = __ldcg(reinterpret_cast<const uint2*>(colmax) + q);
    }
    const float2 *vi0 = sv + (pr.x & 0xffffu), *vj0 = sv + (pr.x >> 16), *vi1 = sv + (pr.y & 0xffffu),
                 *vj1 = sv + (pr.y >> 16);
    df2 w{f2(0.f), f2(0.f)};
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // w += g_c (v_jc - v_ic)
      const df2 y = p_df_mul(as_df2(g[c]), p_df_sub(pair2(vj0[c], vj1[c]), pair2(vi0[c], vi1[c])));
      w = c == 0 ? y : p_df_add(w, y);
    }
    t = p_df_add(t, p_df_mul(as_df2(x), w));
    const float4 wf = as_f4(w);
    sw[q] = wf;
    Wf[a * H + q] = wf;
    const unsigned b0 = abs_bits(w.h.x), b1 = abs_bits(w.h.y);
    if (b0 > cm.x) atomicMax(&colmax[2 * q], b0);
    if (b1 > cm.y) atomicMax(&colmax[2 * q + 1], b1);
    m = max(m, max(b0, b1));
  }
  float th = t.h.x, tl = t.l.x;
  df_add(th, tl, t.h.y, t.l.y);
  for (int o = 16; o > 0; o >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, th, o), ol = __shfl_xor_sync(0xffffffffu, tl, o);
    df_add(th, tl, oh, ol);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((tid & 31) == 0) {
    red[tid >> 5] = m;
    red2[tid >> 5] = make_float2(th, tl);
  }
  __syncthreads();
  m = red[0];
  for (int w = 1; w < nt >> 5; ++w) m = max(m, red[w]);
  const int s = row_scale(m, rootD, bits);
  for (int q = tid; q < H; q += nt) store2<NM>(as_df2(sw[q]), s, d + a * Kp + 2 * q, M * Kp);
  if (tid == nt - 1) {
    sc[a] = s;
    th = red2[0].x;
    tl = red2[0].y;
    for (int w = 1; w < nt >> 5; ++w) df_add(th, tl, red2[w].x, red2[w].y);
    df_mul(th, tl, C.ipih, C.ipil, th, tl);
    t2[a] = make_float2(th, tl);
  }
}

// Column residues of W (rows b < MB, D columns): operand row d holds W[:, d] scaled by the
// column's largest magnitude.  One CTA per 32 rows x 32 columns through shared memory; a thread
// writes four consecutive entries of an operand row per modulus (8 bytes, 64 per row).
template <int NM, typename T>
__global__ void __launch_bounds__(256) rns_cols_kernel(const T* W, int64_t MB, int D, int ldW,
                                                       const unsigned* colmax, int64_t Kp, int64_t rows,
                                                       int bits, bf16* __restrict__ d, int* __restrict__ sc) {
  __shared__ float2 tile[32][33];
  const int64_t b0 = (int64_t)blockIdx.x * 32;
  const int d0 = blockIdx.y * 32;
  grid_trigger();
  grid_wait();
  {
    const int c = threadIdx.x & 31;
#pragma unroll
    for (int r0 = 0; r0 < 32; r0 += 8) {
      const int r = r0 + (threadIdx.x >> 5);
      tile[c][r] = b0 + r < MB && d0 + c < D ? as_pair(__ldcg(W + (b0 + r) * ldW + d0 + c)) : make_float2(0.f, 0.f);
    }
  }
  const int c = threadIdx.x >> 3, r = (threadIdx.x & 7) * 4;
  unsigned m = 0;
  if (d0 + c < D)
#pragma unroll
    for (int i = 0; i < kColCopies / 8; ++i) m = max(m, __ldcg(colmax + ((threadIdx.x & 7) + 8 * i) * ((D + 1) & ~1) + d0 + c));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int s = row_scale(m, sqrtf((float)MB) * 1.0001f, bits);
  __syncthreads();
  if (d0 + c >= D || b0 + r >= Kp) return;
  if (b0 == 0 && r == 0) sc[d0 + c] = s;
  constexpr rns::Crt<NM> C{};
  float2 da[4], db[4];
  digits2(p_scale(pair2(tile[c][r], tile[c][r + 1]), s, s), da);
  digits2(p_scale(pair2(tile[c][r + 2], tile[c][r + 3]), s, s), db);
  bf16* o = d + (int64_t)(d0 + c) * Kp + b0 + r;
  const int64_t stride = rows * Kp;
#pragma unroll
  for (int i = 0; i < NM; ++i)
    *reinterpret_cast<uint2*>(o + i * stride) = make_uint2(residue2<NM>(C, i, da), residue2<NM>(C, i, db));
}

// XT (cols + 1 rows of `rows` entries) = X^T, X rows x cols, and a last row of ones (32 x 32 tiles;
// set-up)
__global__ void rns_transpose_kernel(const double* __restrict__ X, int64_t rows, int64_t cols, double* __restrict__ XT) {
  __shared__ double tile[32][33];
  const int64_t r0 = (int64_t)blockIdx.y * 32, c0 = (int64_t)blockIdx.x * 32;
  for (int yy = threadIdx.y; yy < 32; yy += 8) {
    const int64_t r = r0 + yy, c = c0 + threadIdx.x;
    if (r < rows && c <= cols) tile[yy][threadIdx.x] = c < cols ? X[r * cols + c] : 1.0;
  }
  __syncthreads();
  for (int yy = threadIdx.y; yy < 32; yy += 8) {
    const int64_t c = c0 + yy, r = r0 + threadIdx.x;
    if (r < rows && c <= cols) XT[c * rows + r] = tile[threadIdx.x][yy];
  }
}

// S2 = c^2 S times the mantissa pm of P (set-up)
__global__ void rns_s2_kernel(const double* __restrict__ S, int64_t M, int64_t MB, int64_t ld, double c2pm,
                              float2* __restrict__ S2) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= M * MB) return;
  const int64_t a = i / MB;
  S2[a * ld + (i - a * MB)] = split_d(c2pm * S[i]);
}

// Set-up: G as float pairs in three planes per geometry ([a][c][Dp]) and Xc as float pairs ([a][Dp]),
// rows padded with zeros to Dp, a multiple of 2; ij[p] = 3 i | 3 j << 16 of pair p = (i, j)
__global__ void rns_planes_kernel(const double* __restrict__ G, const double* __restrict__ Xc, int64_t M, int D, int Dp,
                                  float2* __restrict__ G3, float2* __restrict__ Xc2, uint32_t* __restrict__ ij) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= M * D) return;
  const int64_t a = t / D;
  const int p = (int)(t - a * D);
  for (int c = 0; c < 3; ++c) G3[(a * 3 + c) * Dp + p] = split_d(G[3 * t + c]);
  Xc2[a * Dp + p] = split_d(Xc[t]);
  if (a == 0) {
    int i, j;
    pair_of(p, i, j);
    ij[p] = 3u * (uint32_t)i | 3u * (uint32_t)j << 16;
  }
}

// J_a^T xc_a as float pairs (set-up): the back-projection subtracts rowsum_a times it
__global__ void rns_jx_kernel(const double* __restrict__ G, const double* __restrict__ Xc, int64_t M, int N, int D,
                              float2* __restrict__ JX) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int B = 3 * N;
  if (t >= M * B) return;
  const int64_t a = t / B;
  const int o = (int)(t - a * B), i = o / 3, q = o - 3 * i;
  double s = 0.0;
  for (int j = 0; j < N; ++j) {
    if (j == i) continue;
    const int p = pair_idx(i, j);
    const double y = G[(a * D + p) * 3 + q] * Xc[a * D + p];
    s += i > j ? -y : y;
  }
  JX[t] = split_d(s);
}

// ------------------------------------------------------------ residue GEMM
// Units (slab, modulus, row tile, column tile), the column tile fastest, walked by persistent CTA
// pairs.  A slab is one K segment's group of 512-entry chunks.  Per unit a pair computes 256 rows x
// bn columns: k-blocks of 64 K entries through a TMA ring, each four M = 256, N = bn MMAs
// (cta_group::2: each CTA holds 128 rows of A, half the rows of B, and the accumulator of its 128
// rows).  A pair loads 64 bytes per SM and cycle of MMAs where a CTA alone on 128 x 256 loads 96, more
// than L2 delivers (~64).
// Two accumulators of 256 TMEM columns alternate: after each chunk (exact integers) the epilogue
// reduces it mod p and adds residue + 256 to packed 16-bit sums in registers while the other
// accumulator is being filled.
// What it takes to come near the MMAs' rate: the loops of the TMA and MMA warps short and
// warp-uniform, one mbarrier wait and one commit per k-block (T + U at n = 630k: 1.75 ms with two
// waits and looser loops, 1.05 so); 32-byte stores per lane (T 0.48 -> 0.35 ms); no release at cluster
// scope in the epilogue's arrivals.  At n = 630k T (5000 x 5000 x 861) takes 0.35 ms and U (5000 x 862
// x 2 5000) 0.70 ms: 1.8e15 BF16 flop/s, where the sliced products took 1.22 and 2.29 ms.
constexpr int kBM = 128;       // rows per CTA
constexpr int kKB = 64;        // K entries per k-block: one 128-byte swizzle span
constexpr int kKbChunk = 8;    // k-blocks per exact chunk of 512
constexpr int kATile = kBM * 128;
constexpr int kMaxSlots = 8;
constexpr int kRing = 224 * 1024;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 32 * (2 + kEpiWarps);  // warp 0 TMA, 1 MMA, 2.. epilogue
constexpr int kSmem = kRing + 1024 + 256;
constexpr int kMaxChunks = 96;  // per unit
static_assert(kMaxChunks <= rns::kSumChunks, "a unit's 16-bit sums");
static_assert(kSmem <= 227 * 1024, "shared memory per CTA");

struct GemmArgs {
  CUtensorMap a[2], b[2];  // per K segment
  float p[rns::kMaxMod], inv[rns::kMaxMod];
  int nmod, M, N, Rb;   // Ra, Rb: operand rows per modulus; row0: first row of A (per K segment)
  int Ra[2], row0[2];
  int bn, tn, tm;
  int nkb, kb_group, groups, slabs;  // k-blocks per segment and per slab; slabs = segments x groups
  int slots;                         // of the ring
  int64_t ldo;
  uint16_t* out;
  int* err;
  int units;
  // the builds' products (BUILD)
  int shape;    // RNS_FULL, RNS_TRI, RNS_LOWER
  int n_first;  // RNS_LOWER: column tiles of the first row of tiles
  int tiles;    // RNS_LOWER: tiles
};

struct Unit {
  int mod, m0, n0, seg, kb0, nk;
  int64_t plane;
};
template <bool BUILD>
__device__ __forceinline__ Unit unit_of(const GemmArgs& g, int u) {
  Unit x;
  int n, m;
  if (BUILD && g.shape == RNS_LOWER) {  // row m of tiles has n_first + m of them
    n = u % g.tiles;
    u /= g.tiles;
    m = 0;
    for (int w = g.n_first; n >= w; ++w, ++m) n -= w;
  } else if (BUILD) {  // columns outermost, the longest K first (RNS_TRI)
    const int rest = g.units / g.tn;
    n = g.tn - 1 - u / rest;
    u %= rest;
    m = u % g.tm;
    u /= g.tm;
  } else {
    n = u % g.tn;
    u /= g.tn;
    m = u % g.tm;
    u /= g.tm;
  }
  x.mod = u % g.nmod;
  const int sl = u / g.nmod;
  x.seg = sl / g.groups;
  x.kb0 = (sl - x.seg * g.groups) * g.kb_group;
  x.nk = min(g.kb_group, g.nkb - x.kb0);
  x.m0 = m * (2 * kBM);
  x.n0 = n * g.bn;
  // row c of B ends at its entry c
  if (BUILD && g.shape == RNS_TRI) x.nk = max(0, min(x.nk, (x.n0 + g.bn + kKB - 1) / kKB - x.kb0));
  x.plane = (int64_t)sl * g.nmod + x.mod;
  return x;
}

__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A TMA load into this CTA that completes on a barrier of the pair's leader; bytes > 0: first
// expects them on that barrier (the leader itself).  Executed by the warp's elected lane.
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, uint32_t leader_bar,
                                              uint32_t bytes, int x, int y) {
  asm volatile(
      "{\n .reg .pred e, f;\n elect.sync _|e, 0xffffffff;\n setp.ne.and.b32 f, %6, 0, e;\n"
      " @f mbarrier.arrive.expect_tx.shared::cta.b64 _, [%5], %6;\n"
      " @e cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, "
      "%4}], [%2];\n}\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(leader_bar), "r"(x), "r"(y), "r"(bar), "r"(bytes)
      : "memory");
}

// The four MMAs of a k-block (64 K entries: descriptors 2 apart), executed by the warp's elected
// lane.  The whole warp runs the surrounding code, so that the operands stay in uniform registers:
// under `if (lane == 0)` each MMA took ~65 cycles to issue.
__device__ __forceinline__ void mma4(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool acc) {
  asm volatile(
      "{\n .reg .pred e, p;\n .reg .b64 a1, a2, a3, b1, b2, b3;\n"
      " add.s64 a1, %1, 2;\n add.s64 a2, %1, 4;\n add.s64 a3, %1, 6;\n"
      " add.s64 b1, %2, 2;\n add.s64 b2, %2, 4;\n add.s64 b3, %2, 6;\n"
      " setp.ne.b32 p, %4, 0;\n elect.sync _|e, 0xffffffff;\n"
      " @e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n"
      " @e tcgen05.mma.cta_group::2.kind::f16 [%0], a1, b1, %3, 1;\n"
      " @e tcgen05.mma.cta_group::2.kind::f16 [%0], a2, b2, %3, 1;\n"
      " @e tcgen05.mma.cta_group::2.kind::f16 [%0], a3, b3, %3, 1;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc ? 1u : 0u)
      : "memory");
}
// the elected lane's MMAs so far have completed: arrive on this barrier of both CTAs
__device__ __forceinline__ void commit_pair(uint32_t bar) {
  asm volatile(
      "{\n .reg .pred e;\n .reg .b16 m;\n mov.b16 m, 3;\n elect.sync _|e, 0xffffffff;\n"
      " @e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], m;\n}\n" ::"r"(
          bar)
      : "memory");
}

// Bounded wait that also gives up once another role has (limit: polls).  Called by whole warps, of
// which the elected lane polls: the code around stays warp-uniform, so that the operands of copies
// and MMAs stay in uniform registers, and the polls of a CTA's 12 warps do not crowd out one another.
template <bool SLEEP>
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, uint32_t limit, volatile int* abort_flag) {
  for (uint32_t it = 0; it < limit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred e, p;\n mov.u32 %0, 0;\n elect.sync _|e, 0xffffffff;\n"
        " @e mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n @e selp.u32 %0, 1, 0, p;\n}\n"
        : "=&r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (__any_sync(0xffffffffu, done != 0)) return true;
    if ((it & 255) == 255 && __any_sync(0xffffffffu, *abort_flag != 0)) return false;
    if (SLEEP) __nanosleep(40);
  }
  return false;
}

// one thread's bounded wait for an arrival that is under way, given up where another role has failed
__device__ __forceinline__ bool wait_landed(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  const uint32_t addr = tc::smem_u32(bar);
  for (uint32_t it = 0; it < tc::kSpinLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
    if ((it & 255) == 255 && *abort_flag) return false;
  }
  return false;
}

__device__ __forceinline__ void ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

template <bool BUILD>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    rns_gemm_kernel(const __grid_constant__ GemmArgs g) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kRing);  // both CTAs' tiles of a k-block have landed (leader's)
  uint64_t* empty = full + kMaxSlots;                          // its MMAs have completed
  uint64_t* tfull = empty + kMaxSlots;                         // [2] a chunk's MMAs have completed
  uint64_t* tempty = tfull + 2;                                // [2] both CTAs' epilogues have read it (leader's)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);  // raised in both CTAs
  volatile int* peer = abort_flag + 1;  // [2] in the leader: k-blocks the other CTA copied; in the other: the leader's
                                        // k-blocks and chunks of MMAs
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // provably uniform
  const int bn = g.bn, slots = g.slots;
  uint32_t rank;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int units = g.units;
  const int u0 = blockIdx.x >> 1, du = gridDim.x >> 1;
  const int b_bytes = bn * 64;  // this CTA's half of a B tile
  uint8_t* smem_b = smem + slots * kATile;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxSlots; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&tfull[b], 1);
      tc::mbar_init(&tempty[b], 2 * kEpiWarps);
    }
    *abort_flag = 0;
    peer[0] = peer[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(tmem_slot)),
                 "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  tc::fence_before_sync();
  __syncthreads();
  cluster_sync();
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  // (both words are read by the other CTA after a cluster barrier, or earlier as a hint to give up)
  auto tell_peer = [&](volatile int* word, int x) {
    asm volatile("st.volatile.shared::cluster.u32 [%0], %1;" ::"r"(mapa(tc::smem_u32((const void*)word), rank ^ 1u)), "r"(x) : "memory");
  };
  auto fail_with = [&](int code) {
    atomicExch(g.err, code);
    *abort_flag = 1;
    tell_peer(abort_flag, 1);
  };
  int copied = 0;  // producer: k-blocks issued

  grid_trigger();
  grid_wait();
  const uint32_t limit = tc::g_wait_limit;
  const uint32_t full0 = tc::smem_u32(full), empty0 = tc::smem_u32(empty);
  const uint32_t tfull0 = tc::smem_u32(tfull), tempty0 = tc::smem_u32(tempty);
  // The loops below run once per k-block on one warp, ~5 cycles an instruction: they are kept short,
  // since a k-block's MMAs take 512 cycles at most.
  if (warp == 0) {
    // ---------------- TMA producer
    const uint32_t leader0 = mapa(full0, 0), a0 = tc::smem_u32(smem), b0 = tc::smem_u32(smem_b);
    const uint32_t tx = rank == 0 ? 2u * (uint32_t)(kATile + b_bytes) : 0u;
    int slot = 0;
    uint32_t ph = 1;
    bool ok = true;
    for (int u = u0; u < units && ok; u += du) {
      const Unit x = unit_of<BUILD>(g, u);
      const CUtensorMap *mA = &g.a[x.seg], *mB = &g.b[x.seg];
      const int ya = x.mod * g.Ra[x.seg] + g.row0[x.seg] + x.m0 + (int)rank * kBM, yb = x.mod * g.Rb + x.n0 + (int)rank * (bn >> 1);
      int kx = x.kb0 * kKB;
      for (int kb = 0; kb < x.nk; ++kb, kx += kKB) {
        ok = wait_bar<false>(empty0 + 8u * slot, ph, limit, abort_flag);
        if (!ok) break;
        tma_load_pair(a0 + slot * kATile, mA, full0 + 8u * slot, leader0 + 8u * slot, tx, kx, ya);
        tma_load_pair(b0 + slot * b_bytes, mB, full0 + 8u * slot, leader0 + 8u * slot, 0u, kx, yb);
        ++copied;
        if (++slot == slots) {
          slot = 0;
          ph ^= 1u;
        }
      }
    }
    if (lane == 0) {
      if (!ok) fail_with(tc::ERR_TIMEOUT_EMPTY);
      if (rank == 1) tell_peer(peer, copied);
      // the MMAs' arrivals on this CTA's barriers land before it exits (after a failure: see below)
      for (int i = max(0, copied - slots); i < copied && ok; ++i) ok = wait_landed(&empty[i % slots], (uint32_t)(i / slots) & 1u, abort_flag);
      if (!ok && !*abort_flag) fail_with(tc::ERR_TIMEOUT_DONE);
    }
    __syncwarp();
  } else if (warp == 1 && rank == 0) {
    // ---------------- MMA issuer
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(bn >> 3) << 17) | (16u << 24);  // M = 256
    const uint64_t adesc0 = tc::make_sw128_desc(tc::smem_u32(smem));  // linear in address / 16
    const uint64_t bdesc0 = tc::make_sw128_desc(tc::smem_u32(smem_b));
    const uint32_t bstep = (uint32_t)(b_bytes >> 4);
    int slot = 0, issued = 0, chunks = 0;  // chunks committed
    uint32_t ph = 0;
    bool ok = true;
    for (int u = u0; u < units && ok; u += du) {
      const Unit x = unit_of<BUILD>(g, u);
      for (int k0 = 0; k0 < x.nk; k0 += kKbChunk) {
        const int len = min(kKbChunk, x.nk - k0);
        const uint32_t t = (uint32_t)(chunks & 1), acc = tmem + t * 256u;
        ok = wait_bar<false>(tempty0 + 8u * t, ((uint32_t)(chunks >> 1) & 1u) ^ 1u, limit, abort_flag);
        for (int i = 0; i < len && ok; ++i) {
          ok = wait_bar<false>(full0 + 8u * slot, ph, limit, abort_flag);
          if (!ok) break;
          tc::fence_after_sync();
          mma4(acc, adesc0 + (uint64_t)(uint32_t)(slot * (kATile >> 4)), bdesc0 + (uint64_t)(slot * bstep), idesc, i > 0);
          commit_pair(empty0 + 8u * slot);
          ++issued;
          if (++slot == slots) {
            slot = 0;
            ph ^= 1u;
          }
        }
        if (!ok) break;
        commit_pair(tfull0 + 8u * t);
        ++chunks;
      }
    }
    if (lane == 0) {
      if (!ok) fail_with(tc::ERR_TIMEOUT_FULL);
      // every MMA and commit has completed before the tensor memory is released
      tell_peer(peer, issued);
      tell_peer(peer + 1, chunks);
      if (issued > 0) (void)tc::mbar_wait_bounded(&empty[(issued - 1) % slots], (uint32_t)((issued - 1) / slots) & 1u);
      if (chunks > 0) (void)tc::mbar_wait_bounded(&tfull[(chunks - 1) & 1], (uint32_t)((chunks - 1) >> 1) & 1u);
    }
    __syncwarp();
  } else if (warp >= 2) {
    // ---------------- epilogue: lanes = rows, each warp one half of the bn columns
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    const int c0 = half * (bn >> 1);
    const int ng = bn >> 5;  // groups of 16 columns
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0;
    int chunks = 0;
    const uint32_t tempty_leader = mapa(tempty0, 0);
    bool go = true;
    for (int u = u0; u < units && go; u += du) {
      const Unit x = unit_of<BUILD>(g, u);
      const float2 np2 = f2(-g.p[x.mod]), inv2 = f2(g.inv[x.mod]);
      uint32_t acc[8][8];  // packed sums of residue + 256: columns 2w and 2w + 1 of group q
#pragma unroll
      for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int w = 0; w < 8; ++w) acc[q][w] = 0u;
      for (int k0 = 0; k0 < x.nk; k0 += kKbChunk, ++chunks) {
        const uint32_t t = (uint32_t)(chunks & 1);
        if (!wait_bar<true>(tfull0 + 8u * t, (uint32_t)(chunks >> 1) & 1u, limit, abort_flag)) {
          if (lane == 0) fail_with(tc::ERR_TIMEOUT_DONE);
          go = false;
          break;
        }
        tc::fence_after_sync();
        const uint32_t base = lane_base + t * 256u;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (q >= ng) break;
          uint32_t v[16];
          ld16(base + 16 * q, v);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int w = 0; w < 8; ++w) {
            const float2 y = make_float2(__uint_as_float(v[2 * w]), __uint_as_float(v[2 * w + 1]));
            const float2 qq = __fadd2_rn(__ffma2_rn(y, inv2, f2(kMagic)), f2(-kMagic));
            // residue + 256 in the low 16 bits of the float
            const float2 r = __fadd2_rn(__ffma2_rn(qq, np2, y), f2(8388608.f + 256.f));
            acc[q][w] += __byte_perm(__float_as_uint(r.x), __float_as_uint(r.y), 0x5410);
          }
        }
        tc::fence_before_sync();
        __syncwarp();
        // (no release at cluster scope: that would wait for this thread's stores; the accumulator is
        // ordered by the tcgen05 fence)
        if (lane == 0)
          asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(tempty_leader + 8u * t) : "memory");
      }
      if (!go) break;
      const int row = x.m0 + (int)rank * kBM + quarter * 32 + lane;
      if (row < g.M) {
        const int64_t col = x.n0 + c0;
        uint16_t* o = g.out + (x.plane * g.M + row) * g.ldo + col;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (q >= ng || col + 16 * q >= g.ldo) break;
          // one whole 32-byte sector per lane (16-byte stores made T 30 % slower)
          asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(o + 16 * q), "r"(acc[q][0]),
                       "r"(acc[q][1]), "r"(acc[q][2]), "r"(acc[q][3]), "r"(acc[q][4]), "r"(acc[q][5]), "r"(acc[q][6]),
                       "r"(acc[q][7])
                       : "memory");
        }
      }
    }
  }
  __syncwarp();
  tc::fence_before_sync();
  __syncthreads();
  cluster_sync();  // no CTA of the pair leaves while the other's MMAs or arrivals reach it
  if (*abort_flag) {  // (of both CTAs, by now)  nothing in flight outlives the pair
    if (warp == 0 && lane == 0) {
      if (rank == 0) {  // copies of both CTAs land on the leader's barriers
        const int theirs = peer[0], n = max(copied, theirs);
        for (int i = max(0, n - slots); i < n; ++i) {
          uint64_t* bar = &full[i % slots];
          if (i >= copied) tc::mbar_expect_tx(bar, (uint32_t)(kATile + b_bytes));  // theirs alone
          if (i >= theirs)  // theirs was never issued
            asm volatile("mbarrier.complete_tx.shared::cta.b64 [%0], %1;" ::"r"(tc::smem_u32(bar)), "r"((uint32_t)(kATile + b_bytes)) : "memory");
          (void)tc::mbar_wait_bounded(bar, (uint32_t)(i / slots) & 1u);
        }
      } else {  // the leader's commits arrive here too
        const int n = peer[0], chunks = peer[1];
        for (int i = max(0, n - slots); i < n; ++i) (void)tc::mbar_wait_bounded(&empty[i % slots], (uint32_t)(i / slots) & 1u);
        for (int q = max(0, chunks - 2); q < chunks; ++q) (void)tc::mbar_wait_bounded(&tfull[q & 1], (uint32_t)(q >> 1) & 1u);
      }
    }
    __syncwarp();
    __syncthreads();
    cluster_sync();
  }
  if (warp == 1) {
    tc::fence_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
  }
}

// ------------------------------------------------------------ beta
// beta_ab = c^2 S_ab (T_ab - t_b) in double-float (T from its residues) and its row residues.  One
// CTA per row a, two columns per thread and step in packed arithmetic.  STAGE: beta is kept in shared
// memory between the row's maximum and its residues; else (rows of more than kBetaStage columns) it
// is formed twice.  Four CTAs of 256 threads per SM (64 registers) against three at 80; rows that fit the
// chip as CTAs of 128 threads run in one round (see row_threads).
constexpr int64_t kBetaStage = 24 * 1024;
template <int NM, bool STAGE>
__global__ void __launch_bounds__(256, 4) rns_beta_kernel(const uint16_t* Tp, int slabs, int chunks,
                                                          int64_t M, int64_t MB, int64_t ldT, int64_t Rd,
                                                          const int* __restrict__ sA, const int* sW,
                                                          const float2* __restrict__ S2, const float2* t2,
                                                          float rootMB, int64_t Kp, int bits, bf16* __restrict__ d,
                                                          int* __restrict__ sc) {
  extern __shared__ float4 sb[];
  __shared__ unsigned red[8];
  const int64_t a = blockIdx.x;
  const int tid = threadIdx.x;
  constexpr rns::Crt<NM> C{};
  const int ea = C.pexp - 43 - sA[a];
  const uint16_t* Ta = Tp + a * ldT;  // (uniform plane pointers + a 32-bit offset per thread)
  const int64_t plane = M * ldT;
  const float4* Sa = reinterpret_cast<const float4*>(S2 + a * ldT);
  const unsigned n = (unsigned)MB;
  grid_trigger();
  grid_wait();
  auto beta2 = [&](unsigned b) {  // columns b, b + 1 (b even)
    uint32_t w[NM];
#pragma unroll
    for (int i = 0; i < NM; ++i) w[i] = __ldcg(reinterpret_cast<const uint32_t*>(Ta + i * plane + b));
    const df2 S = as_df2(Sa[b >> 1]), t = as_df2(__ldcg(reinterpret_cast<const float4*>(t2) + (b >> 1)));
    const int2 e2 = __ldcg(reinterpret_cast<const int2*>(sW + b));
    for (int sl = 1; sl < slabs; ++sl)
#pragma unroll
      for (int i = 0; i < NM; ++i) w[i] += __ldcg(reinterpret_cast<const uint32_t*>(Ta + (sl * NM + i) * plane + b));
    df2 r = p_df_mul(S, p_df_sub(p_scale(crt_fraction<NM>(C, w, (uint32_t)chunks), ea - e2.x, ea - e2.y), t));
    if (b + 1 >= n) r.h.y = r.l.y = 0.f;
    return r;
  };
  unsigned m = 0;
  for (unsigned b = 2 * tid; b < n; b += 2 * blockDim.x) {
    const df2 r = beta2(b);
    if (STAGE) sb[b >> 1] = as_f4(r);
    m = max(m, max(abs_bits(r.h.x), abs_bits(r.h.y)));
  }
  m = cta_max_bits(m, red);  // contains a __syncthreads
  const int s = row_scale(m, rootMB, bits);
  if (tid == 0) sc[a] = s;
  bf16* da = d + a * Kp;
  const int64_t dplane = Rd * Kp;  // (of the operand: rows of a whole panel)
  for (unsigned b = 4 * tid; b < n; b += 4 * blockDim.x) {
    const df2 zero{f2(0.f), f2(0.f)};
    float2 dx[4], dy[4];
    digits2(p_scale(STAGE ? as_df2(sb[b >> 1]) : beta2(b), s, s), dx);
    digits2(b + 2 < n ? p_scale(STAGE ? as_df2(sb[(b >> 1) + 1]) : beta2(b + 2), s, s) : zero, dy);
#pragma unroll
    for (int i = 0; i < NM; ++i)
      *reinterpret_cast<uint2*>(da + i * dplane + b) = make_uint2(residue2<NM>(C, i, dx), residue2<NM>(C, i, dy));
  }
}

// ------------------------------------------------------------ back-projection
// (K v)_a = J_a^T (U_a - rowsum_a xc_a) (+ lambda v_a) in double-float arithmetic; U_a is the sum
// of the two products, each from its residues, rowsum_a = sum_b beta_ab the second product's column
// D (its operand's row of ones), and J_a^T xc_a comes from the set-up (JX).  One CTA per geometry:
// w_p = g_p u_p into shared memory, two consecutive descriptors per thread and step; then `lanes`
// lanes per atom sum shares of its N - 1 pair terms, all three coordinates (the derivative of x_p
// with respect to its first atom i > j carries the minus sign).  CTA 0 clears the column maxima for
// the next matvec.  A product's slabs are added as packed 16-bit sums; WIDE (more than kSumChunks chunks
// in all, MB > 76,288): `per_sum` slabs at a time, and these in the reconstruction's wider sums.
template <int NM, bool WIDE>
__global__ void __launch_bounds__(256, 4) rns_backproj_kernel(const uint16_t* Up, int slabs, int per_sum, int chunks,
                                                              int64_t M, int D, int Dp, int64_t ldU,
                                                              const int* __restrict__ sA, const int* sWT,
                                                              const int* sB, const int* __restrict__ sXT,
                                                              const float2* __restrict__ JX,
                                                              const float4* __restrict__ G3,
                                                              const double* __restrict__ v, int N, double lam,
                                                              int add_lambda, int lanes, unsigned* colmax,
                                                              double* __restrict__ out) {
  extern __shared__ float4 w4[];  // [3][Dp] pairs: the terms g_pc u_p
  __shared__ float2 rs;
  const int64_t a = blockIdx.x;
  const int tid = threadIdx.x, H = Dp >> 1;
  constexpr rns::Crt<NM> C{};
  grid_wait();
  const int ea = C.pexp - 43 - sA[a], eb = C.pexp - 43 - __ldcg(sB + a);
  if (a == 0)
    for (int p = tid; p < kColCopies * Dp; p += blockDim.x) colmax[p] = 0u;
  const int64_t plane = M * ldU;
  const uint16_t* Ua = Up + a * ldU;
  const float4* Ga = G3 + a * 3 * H;
  const df2 pm{f2(C.pih), f2(C.pil)};
  for (unsigned p = 2 * tid; p <= (unsigned)D; p += 2 * blockDim.x) {
    uint32_t w[2][NM];
    CrtSum sum[2];
    auto load = [&](int s0, int s1) {  // slabs s0 .. s1 - 1
#pragma unroll
      for (int sg = 0; sg < 2; ++sg)
#pragma unroll
        for (int i = 0; i < NM; ++i)
          w[sg][i] = __ldcg(reinterpret_cast<const uint32_t*>(Ua + (int64_t)((sg * slabs + s0) * NM + i) * plane + p));
      for (int sl = s0 + 1; sl < s1; ++sl)
#pragma unroll
        for (int sg = 0; sg < 2; ++sg)
#pragma unroll
          for (int i = 0; i < NM; ++i)
            w[sg][i] += __ldcg(reinterpret_cast<const uint32_t*>(Ua + (int64_t)((sg * slabs + sl) * NM + i) * plane + p));
    };
    const unsigned q = p >> 1, qg = min(q, (unsigned)H - 1u);
    const float4 g[3] = {Ga[qg], Ga[H + qg], Ga[2 * H + qg]};
    for (int s0 = 0; s0 < slabs; s0 += WIDE ? per_sum : slabs) {
      load(s0, WIDE ? min(s0 + per_sum, slabs) : slabs);
      sum[0].add(C, w[0]);
      sum[1].add(C, w[1]);
    }
    // (the scales of columns 0 .. D, padded to an even count)
    const int2 e0 = __ldcg(reinterpret_cast<const int2*>(sWT + p)), e1 = *reinterpret_cast<const int2*>(sXT + p);
    const df2 x = p_scale(sum[0].fraction(C, (uint32_t)chunks), ea - e0.x, ea - e0.y);
    const df2 y = p_scale(sum[1].fraction(C, (uint32_t)chunks), eb - e1.x, eb - e1.y);
    if (p == (unsigned)D) rs = make_float2(y.h.x, y.l.x);
    if (p + 1 == (unsigned)D) rs = make_float2(y.h.y, y.l.y);
    if (p < (unsigned)D) {
      const df2 u = p_df_mul(p_df_add(x, y), pm);
#pragma unroll
      for (int c = 0; c < 3; ++c) w4[c * H + q] = as_f4(p_df_mul(as_df2(g[c]), u));
    }
  }
  __syncthreads();
  const int sub = tid & (lanes - 1), per = (int)blockDim.x / lanes;
  const float2* w3 = reinterpret_cast<const float2*>(w4);
  for (int i0 = 0; i0 < N; i0 += per) {  // every lane group runs the same trip count
    const int i = i0 + tid / lanes;
    df2 xy{f2(0.f), f2(0.f)}, zz{f2(0.f), f2(0.f)};  // coordinates 0 and 1; 2
    if (i < N) {
      const int below = i * (i - 1) / 2;
      for (int j = sub; j < N; j += lanes) {
        if (j == i) continue;
        const float sg = i > j ? -1.f : 1.f;
        const float2* w = w3 + (i > j ? below + j : j * (j - 1) / 2 + i);
        const df2 x = pair2(w[0], w[Dp]), z = pair2(w[2 * Dp], make_float2(0.f, 0.f));
        xy = p_df_add(xy, {p_mul(x.h, f2(sg)), p_mul(x.l, f2(sg))});
        zz = p_df_add(zz, {p_mul(z.h, f2(sg)), p_mul(z.l, f2(sg))});
      }
      if (sub == lanes - 1) {  // - rowsum J^T xc
        const float2* J = JX + (a * N + i) * 3;
        const df2 r = p_df_mul({f2(rs.x), f2(rs.y)}, pm);
        xy = p_df_sub(xy, p_df_mul(r, pair2(J[0], J[1])));
        zz = p_df_sub(zz, p_df_mul(r, pair2(J[2], make_float2(0.f, 0.f))));
      }
    }
    for (int k = 1; k < lanes; k <<= 1) {
      df2 o, q;
      o.h = make_float2(__shfl_xor_sync(0xffffffffu, xy.h.x, k), __shfl_xor_sync(0xffffffffu, xy.h.y, k));
      o.l = make_float2(__shfl_xor_sync(0xffffffffu, xy.l.x, k), __shfl_xor_sync(0xffffffffu, xy.l.y, k));
      q.h = make_float2(__shfl_xor_sync(0xffffffffu, zz.h.x, k), 0.f);
      q.l = make_float2(__shfl_xor_sync(0xffffffffu, zz.l.x, k), 0.f);
      xy = p_df_add(xy, o);
      zz = p_df_add(zz, q);
    }
    if (i < N && sub < 3) {  // lanes 0 .. 2 hold the same sums: one coordinate each
      const int64_t o = (a * N + i) * 3 + sub;
      double s = sub == 0 ? (double)xy.h.x + (double)xy.l.x : sub == 1 ? (double)xy.h.y + (double)xy.l.y
                                                                       : (double)zz.h.x + (double)zz.l.x;
      if (add_lambda) s = fma(lam, v[o], s);
      out[o] = s;
    }
  }
}

}  // namespace

// ------------------------------------------------------------ host side
#define RNS_TRY(x)                \
  do {                            \
    gdml_status _s = (x);         \
    if (_s != GDML_OK) return _s; \
  } while (0)

template <typename T>
static gdml_status rns_alloc(RnsMatvec& r, T** p, size_t count, cudaStream_t st) {
  void* v = nullptr;
  const size_t bytes = std::max<size_t>(count, 1) * sizeof(T);
  if (cudaMalloc(&v, bytes) != cudaSuccess) {
    (void)cudaGetLastError();
    return fail(GDML_ERR_OOM, "residue buffers: cudaMalloc failed");
  }
  r.allocs.push_back(v);
  *p = static_cast<T*>(v);
  if (cudaMemsetAsync(v, 0, bytes, st) != cudaSuccess) return fail(GDML_ERR_CUDA, "residue buffer memset");
  return GDML_OK;
}

static gdml_status make_operand(RnsMatvec& r, RnsOperand& op, int64_t rows, int64_t K, int box_rows, cudaStream_t st) {
  op.rows = rows;
  op.K = K;
  op.Kp = cdiv(K, kKB) * kKB;
  RNS_TRY(rns_alloc(r, &op.d, (size_t)(rns::kMvMods * rows * op.Kp), st));
  RNS_TRY(rns_alloc(r, &op.s, (size_t)rows + 1, st));  // (read in pairs)
  if (!make_kmajor_map(&op.map, op.d, true, (uint64_t)op.Kp, (uint64_t)(rns::kMvMods * rows), (uint64_t)op.Kp,
                       (uint32_t)box_rows))
    return fail(GDML_ERR_CUDA, "cuTensorMapEncodeTiled failed (residue operand)");
  return GDML_OK;
}

int rns_chunks(int64_t nch, int g, int cap) {
  nch = std::max<int64_t>(nch, 1);
  const int64_t lo = cdiv(nch, std::max(cap, 1));  // fewer chunks per unit need more slabs than there are
  return (int)std::min<int64_t>(std::min<int64_t>(nch, kMaxChunks), std::max<int64_t>(lo, g));
}

// Columns per tile and K chunks per unit for an M x N product of nkb k-blocks over `planes`
// independent planes: the fewest cycles of the busiest pair, whole rounds of units x (a unit's
// k-blocks + ~2000 cycles: the ring's start, the last drain, the store).  A k-block takes 2 bn cycles
// of MMAs, 256 + bn of loads at 64 bytes per cycle, and ~300 to wait for and issue.
static void gemm_shape(int64_t M, int64_t N, int64_t nkb, int64_t planes, int cap, int* bn_out, int* g_out) {
  const int64_t pairs = std::max(num_sms() / 2, 1), nch = cdiv(nkb, kKbChunk);
  double best = 1e300;
  for (int64_t bn = 32; bn <= 256; bn += 32) {
    const int64_t tn = cdiv(N, bn);
    if (bn > 32 && cdiv(N, bn - 32) == tn) continue;  // a narrower tile covers N as well
    for (int64_t sl = 1; sl <= std::min<int64_t>(cap, nch); ++sl) {
      const int64_t g = cdiv(nch, sl);
      if (g > kMaxChunks && sl < std::min<int64_t>(cap, nch)) continue;
      const int64_t units = cdiv(M, 2 * kBM) * tn * planes * cdiv(nch, g);
      const double kb = (double)std::min<int64_t>(nkb, g * kKbChunk);
      const double step = std::max(std::max(2.0 * bn, 256.0 + bn), 300.0);
      const double cost = (double)cdiv(units, pairs) * (kb * step + 2000.0) + 600.0 * (double)(cdiv(nch, g) - 1);
      if (cost < best * 0.999) {
        best = cost;
        *bn_out = (int)bn;
        *g_out = (int)g;
      }
    }
  }
}

// residues of A B^T (or of both segments' products) into out
template <bool BUILD>
static gdml_status launch_gemm(GemmArgs& g, int segs, int chunks, bool pdl, cudaStream_t st) {
  if (!allow_smem(rns_gemm_kernel<BUILD>, kSmem)) return fail(GDML_ERR_CUDA, "cudaFuncSetAttribute(residue gemm)");
  for (int i = 0; i < rns::kMaxMod; ++i) {
    g.p[i] = (float)rns::kMods[i];
    g.inv[i] = 1.0f / (float)rns::kMods[i];
  }
  g.nmod = rns::kMvMods;
  g.tn = (int)cdiv(g.N, g.bn);
  g.tm = (int)cdiv(g.M, 2 * kBM);
  g.kb_group = chunks * kKbChunk;
  g.groups = (int)cdiv(g.nkb, g.kb_group);
  g.slabs = segs * g.groups;
  g.slots = std::min(kMaxSlots, kRing / (kATile + g.bn * 64));
  int64_t tiles = (int64_t)g.tm * g.tn;
  if (BUILD && g.shape == RNS_LOWER) {
    g.n_first = g.row0[0] / (2 * kBM) + 1;
    tiles = 0;
    for (int m = 0; m < g.tm; ++m) tiles += g.n_first + m;
    g.tiles = (int)tiles;
  }
  const int64_t units = (int64_t)g.slabs * g.nmod * tiles;
  if (chunks > kMaxChunks) return fail(GDML_ERR_ARG, "residue gemm: too many K chunks per unit");
  if (units > INT32_MAX / 2) return fail(GDML_ERR_ARG, "residue gemm: too many tiles");
  g.units = (int)units;
  const unsigned grid = 2u * (unsigned)std::min<int64_t>(units, std::max(num_sms() / 2, 1));
  { launch_after(pdl, rns_gemm_kernel<BUILD>, grid, kThreads, kSmem, st, g); count_launch(); }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(GDML_ERR_CUDA, std::string("residue gemm launch: ") + cudaGetErrorString(e));
  return GDML_OK;
}

// rows row0[s] .. row0[s] + M of segment s's A
static gdml_status rns_gemm(const RnsOperand* A, const RnsOperand* B, const int64_t* row0, int64_t M, int segs, int bn,
                            int chunks, uint16_t* out, int64_t ldo, int* err, bool pdl, cudaStream_t st, int* slabs_out) {
  GemmArgs g{};
  for (int s = 0; s < 2; ++s) {
    g.a[s] = A[s < segs ? s : 0].map;
    g.b[s] = B[s < segs ? s : 0].map;
    g.Ra[s] = (int)A[s < segs ? s : 0].rows;
    g.row0[s] = (int)row0[s < segs ? s : 0];
  }
  g.M = (int)M;
  g.N = g.Rb = (int)B[0].rows;
  g.bn = bn;
  g.nkb = (int)(A[0].Kp / kKB);
  g.ldo = ldo;
  g.out = out;
  g.err = err;
  RNS_TRY(launch_gemm<false>(g, segs, chunks, pdl, st));
  if (slabs_out) *slabs_out = g.groups;
  return GDML_OK;
}

gdml_status rns_product(RnsProduct& q, int* err, cudaStream_t st) {
  GemmArgs g{};
  if (!make_kmajor_map(&g.a[0], q.A, true, (uint64_t)q.Kp, (uint64_t)(rns::kMvMods * q.Ra), (uint64_t)q.Kp, kBM) ||
      !make_kmajor_map(&g.b[0], q.B, true, (uint64_t)q.Kp, (uint64_t)(rns::kMvMods * q.Rb), (uint64_t)q.Kp,
                       (uint32_t)q.bn / 2))
    return fail(GDML_ERR_CUDA, "cuTensorMapEncodeTiled failed (residue product)");
  g.a[1] = g.a[0];
  g.b[1] = g.b[0];
  g.M = (int)q.M;
  g.N = (int)q.N;
  g.Ra[0] = (int)q.Ra;
  g.Rb = (int)q.Rb;
  g.bn = q.bn;
  g.nkb = (int)(q.Kp / kKB);
  g.ldo = q.ldo;
  g.out = q.out;
  g.err = err;
  g.shape = q.shape;
  g.row0[0] = (int)q.row0;
  return launch_gemm<true>(g, 1, q.chunks, false, st);
}

void rns_product_shape(RnsProduct& q, int cap) {
  int bn = 256, g = 1;
  gemm_shape(q.M, q.N, q.Kp / kKB, rns::kMvMods, cap, &bn, &g);
  if (q.shape == RNS_LOWER && bn != 256) {  // square tiles: the diagonal's fall on the rows' last
    bn = 256;
    const int64_t nch = cdiv(q.Kp, rns::kChunk);
    const int64_t units = cdiv(q.M, 2 * kBM) * cdiv(q.N, 256) * rns::kMvMods;
    g = (int)cdiv(nch, std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(cap, nch), num_sms() / 2 / units)));
  }
  q.bn = bn;
  q.chunks = std::min(std::max(g, 1), kMaxChunks);
  q.slabs = (int)cdiv(cdiv(q.Kp, rns::kChunk), q.chunks);
}

template <typename F>
static gdml_status big_smem(F* fn, size_t bytes) {
  return allow_smem(fn, bytes) ? GDML_OK : fail(GDML_ERR_CUDA, "cudaFuncSetAttribute(residue matvec)");
}

// Bytes of T, beta and U at a time.  With 2 GB the rounds of units that end each panel cost 4 to 9 % at M = 8,000 to
// 20,000 (12,000 rows, D = 210: 4.41 -> 4.83 ms)
constexpr int64_t kPanelBytes = (int64_t)8 << 30;

gdml_status rns_setup(RnsMatvec& r, int64_t M, int N, int D, const double* G, const double* Xc, const double* A, int64_t ldA,
                      const double* S, double c, cudaStream_t st, int Ssym, const int* pis, const double* XcB) {
  constexpr int NM = rns::kMvMods;
  if (Ssym < 1 || (Ssym > 1 && (!pis || !XcB))) return fail(GDML_ERR_ARG, "residue setup: bad symmetry arguments");
  const int64_t MB = M * Ssym;
  // (beta's kernel adds all K groups of T as packed 16-bit sums)
  if (MB > (int64_t)1 << 24 || D > rns::kSumChunks * rns::kChunk) return fail(GDML_ERR_ARG, "system too large for the residue path");
  r.M = M;
  r.MB = MB;
  r.N = N;
  r.D = D;
  r.S = Ssym;
  r.pis = pis;
  r.XcB = Ssym > 1 ? XcB : Xc;
  r.ldT = cdiv(MB, 16) * 16;
  r.ldU = cdiv(D + 1, 16) * 16;
  r.Dp = 2 * (int)cdiv(D, 2);
  r.nch1 = cdiv(D, kKB * kKbChunk);
  r.nch2 = cdiv(MB, kKB * kKbChunk);
  // K groups kept in HBM: more of them only where the products are small
  auto slab_cap = [](int64_t entries, int64_t nch) {
    return (int)std::max<int64_t>(cdiv(nch, kMaxChunks), std::min<int64_t>(std::min<int64_t>(nch, 4), ((int64_t)1 << 29) / (2 * NM * std::max<int64_t>(entries, 1))));
  };
  // T, beta and U exist for a panel of rows at a time: 56 bytes per pair of rows and training rows, which
  // with the 68 that stay (S, [A | beta] and T in FP64, c^2 S, A's residues) would be more than the 76 of
  // sliced operands; within kPanelBytes (M = 12,300 at D = 210) all rows are one panel
  {
    const int64_t row = 2 * NM * (cdiv(r.nch1, kMaxChunks) * r.ldT + cdiv(MB, kKB) * kKB + 2 * cdiv(r.nch2, kMaxChunks) * r.ldU);
    const int64_t fit = std::max<int64_t>(1, kPanelBytes / row / 256) * 256;
    r.P = M <= fit ? M : cdiv(cdiv(M, cdiv(M, fit)), 256) * 256;
  }
  r.cap1 = slab_cap(r.P * r.ldT, r.nch1);
  r.cap2 = slab_cap(2 * r.P * r.ldU, r.nch2);
  gemm_shape(r.P, MB, cdiv(D, kKB), NM, r.cap1, &r.bn1, &r.g1);
  gemm_shape(r.P, D + 1, cdiv(MB, kKB), 2 * NM, r.cap2, &r.bn2, &r.g2);
  RNS_TRY(make_operand(r, r.Xc1, M, D, kBM, st));
  RNS_TRY(make_operand(r, r.W1, MB, D, r.bn1 / 2, st));
  RNS_TRY(make_operand(r, r.A2, M, MB, kBM, st));
  RNS_TRY(make_operand(r, r.WT2, D + 1, MB, r.bn2 / 2, st));  // row D: zeros
  RNS_TRY(make_operand(r, r.B2, r.P, MB, kBM, st));
  RNS_TRY(make_operand(r, r.XT2, D + 1, MB, r.bn2 / 2, st));  // row D: ones
  RNS_TRY(rns_alloc(r, &r.G3, (size_t)(3 * M * r.Dp), st));
  RNS_TRY(rns_alloc(r, &r.Xc2, (size_t)(M * r.Dp), st));
  RNS_TRY(rns_alloc(r, &r.ij, (size_t)r.Dp, st));
  RNS_TRY(rns_alloc(r, &r.colmax, (size_t)(kColCopies * r.Dp), st));
  RNS_TRY(rns_alloc(r, &r.t2, (size_t)r.ldT, st));
  RNS_TRY(rns_alloc(r, &r.S2, (size_t)(M * r.ldT), st));
  RNS_TRY(rns_alloc(r, &r.Tp, (size_t)(r.cap1 * NM * r.P * r.ldT), st));
  RNS_TRY(rns_alloc(r, &r.Up, (size_t)(2 * r.cap2 * NM * r.P * r.ldU), st));
  RNS_TRY(rns_alloc(r, &r.JX, (size_t)(3 * M * N), st));
  RNS_TRY(rns_alloc(r, &r.err, 1, st));
  if (Ssym > 1) {
    RNS_TRY(rns_alloc(r, &r.W, (size_t)(M * D), st));
    RNS_TRY(rns_alloc(r, &r.WB, (size_t)(MB * D), st));
    RNS_TRY(rns_alloc(r, &r.t, (size_t)MB, st));
  } else {
    RNS_TRY(rns_alloc(r, &r.Wf, (size_t)(M * r.Dp), st));
  }
  auto fixed = [&](const double* X, int64_t ldx, RnsOperand& op) {
    rns_fixed_rows_kernel<NM><<<(unsigned)op.rows, 256, 0, st>>>(X, ldx, op.K, op.rows, op.Kp, rns::kMvBits, op.d, op.s);
    count_launch();
  };
  fixed(Xc, D, r.Xc1);
  fixed(A, ldA, r.A2);
  // the transposed descriptors go where T's residues will be, if these take more room
  double *XT = reinterpret_cast<double*>(r.Tp), *own = nullptr;
  if ((size_t)(r.cap1 * NM * r.P * r.ldT) * sizeof(uint16_t) < (size_t)(MB * (D + 1)) * sizeof(double)) {
    if (cudaMalloc(&own, (size_t)(MB * (D + 1)) * sizeof(double)) != cudaSuccess) {
      (void)cudaGetLastError();
      return fail(GDML_ERR_OOM, "residue set-up scratch");
    }
    XT = own;
  }
  { rns_transpose_kernel<<<dim3((unsigned)cdiv(D + 1, 32), (unsigned)cdiv(MB, 32)), dim3(32, 8), 0, st>>>(r.XcB, MB, D, XT); count_launch(); }
  fixed(XT, MB, r.XT2);  // D + 1 rows
  { rns_planes_kernel<<<(unsigned)cdiv(M * D, 256), 256, 0, st>>>(G, Xc, M, D, r.Dp, r.G3, r.Xc2, r.ij); count_launch(); }
  { rns_jx_kernel<<<(unsigned)cdiv(3 * M * N, 256), 256, 0, st>>>(G, Xc, M, N, D, r.JX); count_launch(); }
  constexpr rns::Crt<NM> C{};
  { rns_s2_kernel<<<(unsigned)cdiv(M * MB, 256), 256, 0, st>>>(S, M, MB, r.ldT, c * c * ((double)C.pih + (double)C.pil), r.S2); count_launch(); }
  const bool bad = cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess;
  if (own) cudaFree(own);
  if (bad) return fail(GDML_ERR_CUDA, "residue setup kernels");
  r.ready = true;
  return GDML_OK;
}

// Threads per row of the beta and back-projection kernels (64 registers, `smem` bytes a row): 128 where a
// row has no work for more, or where that makes all M rows resident at once and 256 do not; else 256.
// Back-projection of M = 1,000 rows, D = 210: 13.3 us, 20.3 with 256 threads in three CTAs per SM; beta of
// 1,000 columns 18.9 and 20.2; of 6,000 columns (48 KB a row, so four CTAs either way) 128 threads took 16 us longer.
static int row_threads(int64_t M, int64_t pairs, size_t smem) {
  const int64_t sms = num_sms(), fit = std::min<int64_t>(8, (int64_t)(227 * 1024 / (smem + 2048)));
  if (pairs <= 128) return 128;
  return M > std::min<int64_t>(4, fit) * sms && M <= fit * sms ? 128 : 256;
}

// Whether the matvec's kernels may start while the one before them drains (each waits for it before it
// reads, and reads what a kernel of the same matvec wrote past L1, never as read-only data): about 1.5 us of
// launch and start-up per kernel.  Outside capture only, and where a kernel's rows are resident at once:
// M = 200, D = 36 28.3 us, 38.6 without; M = 1,000, D = 210 92.9 and 98.9; but M = 5,000, D = 861 1,660 and
// 1,588, and a captured solve at M = 1,000 8.96 and 8.85 ms.
static bool chained(int64_t M, cudaStream_t st) {
  return M <= 8 * (int64_t)num_sms() && not_capturing(st);
}

gdml_status rns_matvec(RnsMatvec& r, const double* G, const double* Xc, const double* v, double* out, int add_lambda,
                       double lam, cudaStream_t st) {
  constexpr int NM = rns::kMvMods;
  constexpr int bits = rns::kMvBits;
  if (!r.ready) return fail(GDML_ERR_STATE, "residue matvec not set up");
  const int64_t M = r.M, MB = r.MB;
  const int D = r.D;
  const bool pdl = chained(M, st);
  const float rootD = std::sqrt((float)D) * 1.0001f, rootMB = std::sqrt((float)MB) * 1.0001f;
  const dim3 gc((unsigned)cdiv(MB, 32), (unsigned)cdiv(D, 32));
  const size_t proj_sm = (size_t)(3 * r.N + r.Dp) * sizeof(float2);
  const size_t beta_sm = MB <= kBetaStage ? (size_t)r.ldT * sizeof(float2) : 0, back_sm = 3 * (size_t)r.Dp * sizeof(float2);
  auto* beta = MB <= kBetaStage ? rns_beta_kernel<NM, true> : rns_beta_kernel<NM, false>;
  const bool wide = r.nch2 > rns::kSumChunks;
  const int per_sum = rns::kSumChunks / rns_chunks(r.nch2, r.g2, r.cap2);
  auto* backproj = wide ? rns_backproj_kernel<NM, true> : rns_backproj_kernel<NM, false>;
  RNS_TRY(big_smem(rns_proj_kernel<NM>, proj_sm));
  RNS_TRY(big_smem(beta, beta_sm));
  RNS_TRY(big_smem(backproj, back_sm));
  if (r.S > 1) {  // w_b = J_b v_b, then row b S + q = P_q w_b with t = xc_(bS+q) . w_(bS+q)
    launch_proj(G, Xc, v, M, r.N, D, r.W, D, r.t, st);
    launch_sym_gather(r.W, M, D, r.pis, r.S, r.XcB, r.WB, r.t, st);
    { rns_rows_kernel<NM><<<(unsigned)MB, 256, 0, st>>>(r.WB, MB, D, r.W1.Kp, bits, r.W1.d, r.W1.s, r.colmax, r.t, r.t2); count_launch(); }
    { launch_after(pdl, rns_cols_kernel<NM, double>, gc, 256, 0, st, r.WB, MB, D, D, r.colmax, r.WT2.Kp, D + 1, bits, r.WT2.d, r.WT2.s); count_launch(); }
  } else {
    const int nt = (int)std::min<int64_t>(512, std::max<int64_t>(64, cdiv(cdiv(D, 2), 32) * 32));
    { rns_proj_kernel<NM><<<(unsigned)M, nt, proj_sm, st>>>((const float4*)r.G3, (const float4*)r.Xc2, (const uint2*)r.ij, v, M, r.N, r.Dp, rootD, (float4*)r.Wf, r.t2, r.W1.Kp, bits, r.W1.d, r.W1.s, r.colmax); count_launch(); }
    { launch_after(pdl, rns_cols_kernel<NM, float2>, gc, 256, 0, st, r.Wf, MB, D, r.Dp, r.colmax, r.WT2.Kp, D + 1, bits, r.WT2.d, r.WT2.s); count_launch(); }
  }
  for (int64_t a0 = 0; a0 < M; a0 += r.P) {  // panels of rows
    const int64_t rows = std::min(r.P, M - a0);
    int s1 = 0, s2 = 0;
    RNS_TRY(rns_gemm(&r.Xc1, &r.W1, &a0, rows, 1, r.bn1, rns_chunks(r.nch1, r.g1, r.cap1), r.Tp, r.ldT, r.err, pdl, st, &s1));
    const int nr = row_threads(rows, cdiv(MB, 2), beta_sm);
    { launch_after(pdl, beta, (unsigned)rows, nr, beta_sm, st, r.Tp, s1, (int)r.nch1, rows, MB, r.ldT, r.P, r.Xc1.s + a0, r.W1.s, r.S2 + a0 * r.ldT, r.t2, rootMB, r.B2.Kp, bits, r.B2.d, r.B2.s); count_launch(); }
    const RnsOperand a[2] = {r.A2, r.B2}, b[2] = {r.WT2, r.XT2};
    const int64_t row0[2] = {a0, 0};
    RNS_TRY(rns_gemm(a, b, row0, rows, 2, r.bn2, rns_chunks(r.nch2, r.g2, r.cap2), r.Up, r.ldU, r.err, pdl, st, &s2));
    const int nb = row_threads(rows, cdiv(D + 1, 2), back_sm);
    int lanes = 4;  // per atom in the last step: as many as the threads give, up to 16
    while (lanes < 16 && 2 * lanes * r.N <= nb) lanes *= 2;
    const int64_t c0 = a0 * 3 * r.N;
    { launch_after(pdl, backproj, (unsigned)rows, nb, back_sm, st, r.Up, s2, per_sum, (int)r.nch2, rows, D, r.Dp, r.ldU, r.A2.s + a0, r.WT2.s, r.B2.s, r.XT2.s, r.JX + c0, (const float4*)(r.G3 + a0 * 3 * r.Dp), v + c0, r.N, lam, add_lambda, lanes, r.colmax, out + c0); count_launch(); }
  }
  if (cudaGetLastError() != cudaSuccess) return fail(GDML_ERR_CUDA, "residue matvec kernels");
  return GDML_OK;
}

gdml_status rns_check(RnsMatvec& r, cudaStream_t st) {
  if (!r.ready) return GDML_OK;
  int h = 0;
  if (cudaMemcpyAsync(&h, r.err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return fail(GDML_ERR_CUDA, "reading the residue gemm's error word");
  if (h) {
    cudaMemsetAsync(r.err, 0, sizeof(int), st);
    return fail(GDML_ERR_TIMEOUT, "a residue gemm pipeline wait timed out (code " + std::to_string(h) + ")");
  }
  return GDML_OK;
}

void rns_destroy(RnsMatvec& r) {
  for (void* p : r.allocs) cudaFree(p);
  r.allocs.clear();
  r.ready = false;
}

cudaError_t set_wait_limit_rns(uint32_t polls) { return tc::set_wait_limit_here(polls); }

}  // namespace gdml
