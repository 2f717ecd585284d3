// Products of the OZAKI preconditioner build on the residue GEMM (see rns.cuh for the scheme):
//   K_nk L_kk^-T and the leverage scores' row norms (tall A, triangular B), and the Gram matrices
//   L^T L and X^T X (lower triangle).
// Operands are rounded to integers of 57 bits below max sqrt(K) of their row; the GEMM leaves the
// products' residues, and the output kernels reconstruct them in 96-bit fixed point and round once
// to FP64.  The sliced form (7 slices of 7 bits below each 256-entry chunk's largest magnitude) kept 49.
//
// n = 126,126, k = 1,500 with leverage scores (three tall products, five Gram matrices): 73 ms sliced
// with all level sums in one CTA's tensor memory (17 ms a tall product), 34 ms so: 16.4 ms of GEMM
// (bounded by its tensor-core rate at 256 x 256 tiles), 9.4 ms of operands and 8.3 ms of outputs, whose
// kernels run at 3 to 5 TB/s on their 28 bytes of residues per entry.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "kernels.cuh"
#include "rns.cuh"

namespace gdml {

namespace {

using bf16 = __nv_bfloat16;
constexpr int NM = rns::kMvMods;
// bytes of residues (operand panel and outputs) at a time: 34 ms of products at n = 126,126, k = 1,500;
// with half of it, which L2 would hold, 39 ms (fewer tiles per launch)
constexpr int64_t kScratch = (int64_t)256 << 20;
constexpr int64_t kKPanel = 16384;                // K entries of a Gram product at a time (sqrt(K) costs 7 bits)

// Weights of the reconstruction: frac(x / P) = frac(sum_i r_i frac(fold_i / p_i)), in units of 2^-96
struct Crt96 {
  uint64_t h[NM];
  uint32_t l[NM];
  uint64_t oh;  // 256 times their sum: the offset of a chunk's residue + 256
  uint32_t ol;
  long long pm;  // P = pm 2^pexp
  int pexp;
  constexpr Crt96() : h(), l(), oh(0), ol(0), pm(0), pexp(0) {
    const rns::Crt<NM> c{};
    unsigned __int128 off = 0;
    for (int i = 0; i < NM; ++i) {
      const unsigned __int128 one = (unsigned __int128)1 << 96;
      const unsigned __int128 w = (one * (unsigned)c.fold[i] + (unsigned)c.m[i] / 2) / (unsigned)c.m[i] % one;
      h[i] = (uint64_t)(w >> 32);
      l[i] = (uint32_t)w;
      off += 256 * w;
    }
    oh = (uint64_t)(off >> 32);
    ol = (uint32_t)off;
    unsigned __int128 P = 1;  // 118 bits
    for (int i = 0; i < NM; ++i) P *= (unsigned)c.m[i];
    pm = (long long)(uint64_t)(P >> 55);
    pexp = 55;
  }
};

// The FP64 pipe does under two operations per cycle and SM, so conversions and products there would
// outlast an entry's 28 bytes of residues: numbers are taken apart and put together as integers
// (outputs of 3,072 x 1,500: 75 -> 64 us; operands 38 us either way).

// x = return value 2^e (53 or 24 bits and the sign); x finite
__device__ __forceinline__ long long take_apart(double x, int& e) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)((uint64_t)b >> 52) & 0x7ff;
  e = max(ex, 1) - 1075;
  const long long m = (b & 0xfffffffffffffll) | (ex ? 1ll << 52 : 0);
  return b < 0 ? -m : m;
}
__device__ __forceinline__ long long take_apart(float x, int& e) {
  const int b = __float_as_int(x), ex = (b >> 23) & 0xff;
  e = max(ex, 1) - 150;
  const int m = (b & 0x7fffff) | (ex ? 1 << 23 : 0);
  return b < 0 ? -m : m;
}
// v 2^e rounded to FP64
__device__ __forceinline__ double put_together(long long v, int e) {
  const uint64_t a = (uint64_t)(v < 0 ? -v : v);
  if (a == 0) return 0.0;
  const int lz = __clzll((long long)a), ex = 1023 + 63 - lz + e;
  if (ex < 1 || ex > 2045) return scalbn((double)v, e);
  const uint64_t m = a << lz;
  // (a carry out of the mantissa raises the exponent)
  const uint64_t b = ((uint64_t)(ex - 1) << 52) + (m >> 11) + ((m >> 10) & 1u);
  return __longlong_as_double((long long)(b | (v < 0 ? 1ull << 63 : 0)));
}

// Scale of a row of K entries whose largest magnitude has the high word m: 2^s max sqrt(K) < 2^kMvBits
__device__ __forceinline__ int scale_of(unsigned m, double rootK) {
  if (m >= 0x7fefffffu) return rns::kBad;  // NaN or infinity (or within an ulp of it)
  if (m < 0x00100000u) return 0;           // zero (or denormal: rounds to zero)
  const double b = __hiloint2double((int)m + 1, 0) * 0.5 * rootK;
  const unsigned hb = (unsigned)__double2hiint(b);
  if (hb >= 0x7ff00000u) return rns::kBad;
  return rns::kMvBits - ((int)(hb >> 20) - 1022 + 1);  // b < 2^(exponent + 1)
}

__device__ __forceinline__ unsigned high_abs(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ unsigned high_abs(float x) { return (unsigned)__float_as_int(x) & 0x7fffffffu; }
__device__ __forceinline__ unsigned double_high(unsigned m, double) { return m; }
__device__ __forceinline__ unsigned double_high(unsigned m, float) {  // of a float's bits
  return m >= 0x7f800000u ? 0x7ff00000u : (unsigned)__double2hiint((double)__uint_as_float(m));
}

// the integer nearest x 2^s (|.| <= 2^57), cut into digits of 14 bits
template <typename T>
__device__ __forceinline__ void to_digits(T x, int s, float (&d)[4]) {
  int e;
  long long v = take_apart(x, e);
  e += s;
  v = e >= 0 ? v << min(e, 57) : e > -60 ? (v + (1ll << (-e - 1))) >> -e : 0;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int t = ((int)(uint32_t)v << 18) >> 18;
    d[q] = (float)t;
    v = (v - t) >> rns::kDigit;
  }
  d[3] = (float)(int)v;
}

template <typename T>
__device__ __forceinline__ void store_residues(T x0, T x1, int s, bf16* __restrict__ d, int64_t stride) {
  constexpr rns::Crt<NM> C{};
  float a[4] = {0.f, 0.f, 0.f, 0.f}, b[4] = {0.f, 0.f, 0.f, 0.f};
  if (s != rns::kBad) {
    to_digits(x0, s, a);
    to_digits(x1, s, b);
  }
  const float2 dg[4] = {make_float2(a[0], b[0]), make_float2(a[1], b[1]), make_float2(a[2], b[2]), make_float2(a[3], b[3])};
#pragma unroll
  for (int i = 0; i < NM; ++i) *reinterpret_cast<uint32_t*>(d + i * stride) = rns::residue2<NM>(C, i, dg);
}

// Scales of the rows of a row-major matrix: one CTA per row
template <typename T>
__global__ void __launch_bounds__(256) row_scales_kernel(const T* __restrict__ X, int64_t ldx, int64_t K, double rootK,
                                                         int* __restrict__ sc) {
  __shared__ unsigned red[8];
  const T* x = X + (int64_t)blockIdx.x * ldx;
  unsigned m = 0;
#pragma unroll 4
  for (int64_t k = threadIdx.x; k < K; k += 256) m = max(m, high_abs(x[k]));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) m = max(m, red[w]);
    sc[blockIdx.x] = scale_of(double_high(m, T(0)), rootK);
  }
}

// Residues of the rows of a row-major matrix: 512 entries per CTA
template <typename T>
__global__ void __launch_bounds__(256) row_residues_kernel(const T* __restrict__ X, int64_t ldx, int64_t K, int64_t Kp,
                                                           int64_t rows, const int* __restrict__ sc,
                                                           bf16* __restrict__ d) {
  const int64_t row = blockIdx.x, k = ((int64_t)blockIdx.y * 256 + threadIdx.x) * 2;
  if (k >= Kp) return;
  const T* x = X + row * ldx;
  const T x0 = k < K ? x[k] : T(0), x1 = k + 1 < K ? x[k + 1] : T(0);
  store_residues(x0, x1, sc[row], d + row * Kp + k, rows * Kp);
}

// Scales of rows r0 .. r0 + rows of a column-major matrix: 32 rows per CTA
__global__ void __launch_bounds__(1024) col_scales_kernel(const double* __restrict__ A, int64_t ld, int64_t r0,
                                                         int64_t rows, int64_t K, double rootK, int* __restrict__ sc) {
  __shared__ unsigned red[32][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t r = (int64_t)blockIdx.x * 32 + lane;
  unsigned m = 0;
  if (r < rows)
#pragma unroll 8
    for (int64_t k = w; k < K; k += 32) m = max(m, high_abs(A[k * ld + r0 + r]));
  red[w][lane] = m;
  __syncthreads();
  if (w == 0 && r < rows) {
    for (int i = 1; i < 32; ++i) m = max(m, red[i][lane]);
    sc[r] = scale_of(m, rootK);
  }
}

// Residues of those rows: a tile of 32 rows x 64 entries per CTA, transposed in shared memory so that
// reads run down the columns and writes along the rows (128 bytes each)
__global__ void __launch_bounds__(256) col_residues_kernel(const double* __restrict__ A, int64_t ld, int64_t r0,
                                                           int64_t rows, int64_t K, int64_t Kp, int64_t R,
                                                           const int* __restrict__ sc, bf16* __restrict__ d) {
  __shared__ double tile[32][65];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t rb = (int64_t)blockIdx.x * 32, k0 = (int64_t)blockIdx.y * 64;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int kk = w + 8 * i;
    const int64_t k = k0 + kk;
    tile[lane][kk] = rb + lane < rows && k < K ? A[k * ld + r0 + rb + lane] : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = w + 8 * i;
    if (rb + r >= rows) break;
    store_residues(tile[r][2 * lane], tile[r][2 * lane + 1], sc[rb + r], d + (rb + r) * Kp + k0 + 2 * lane, R * Kp);
  }
}

// ---- outputs
struct OutArgs {
  const uint16_t* u;  // [slab][modulus][rows][ldo]
  int slabs;
  int64_t rows, ldo, N;
  int nch;           // chunks of K
  int tri_bn;        // > 0: RNS_TRI with this many columns per tile
  const int *sa, *sb;
};
__device__ __forceinline__ int chunks_of(const OutArgs& g, int64_t c) {
  if (!g.tri_bn) return g.nch;
  return (int)min((int64_t)g.nch, ((c / g.tri_bn + 1) * g.tri_bn + rns::kChunk - 1) / rns::kChunk);
}
// products of row r with columns c (even) and c + 1
__device__ __forceinline__ double2 value2(const OutArgs& g, int64_t r, int64_t c, int sa) {
  constexpr Crt96 C{};
  const int64_t plane = g.rows * g.ldo;
  const uint16_t* u = g.u + r * g.ldo + c;
  uint32_t w[NM];
  uint64_t hi[2] = {0, 0}, lo[2] = {0, 0};
  for (int sl = 0; sl < g.slabs; ++sl) {
#pragma unroll
    for (int i = 0; i < NM; ++i) w[i] = __ldcs(reinterpret_cast<const uint32_t*>(u + ((int64_t)sl * NM + i) * plane));
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      const uint32_t x[2] = {w[i] & 0xffffu, w[i] >> 16};
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        lo[v] += (uint64_t)x[v] * C.l[i];
        hi[v] += (uint64_t)x[v] * C.h[i];
      }
    }
  }
  const int64_t nch = chunks_of(g, c);
  double y[2];
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    const int64_t f =
        (int64_t)(hi[v] - (uint64_t)nch * C.oh + (uint64_t)((int64_t)(lo[v] - (uint64_t)nch * C.ol) >> 32));
    const int sb = c + v < g.N ? g.sb[c + v] : 0;
    y[v] = sa == rns::kBad || sb == rns::kBad ? __longlong_as_double(0x7ff8000000000000ll)
                                              : put_together(__mul64hi(f, C.pm), C.pexp - sa - sb);
  }
  return make_double2(y[0], y[1]);
}

// C column-major (and as FP32): 32 rows x 64 columns per CTA, transposed in shared memory
__global__ void __launch_bounds__(256) out_cols_kernel(const OutArgs g, int64_t ldc, double* __restrict__ C,
                                                       float* __restrict__ C32) {
  __shared__ double tile[64][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * 32, c0 = (int64_t)blockIdx.y * 64;
  const int64_t c = c0 + 2 * lane;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t r = r0 + w + 8 * i;
    if (r < g.rows && c < g.N) {
      const double2 y = value2(g, r, c, g.sa[r]);
      tile[2 * lane][w + 8 * i] = y.x;
      tile[2 * lane + 1][w + 8 * i] = y.y;
    }
  }
  __syncthreads();
  const int64_t r = r0 + lane;
  if (r < g.rows)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int64_t cc = c0 + w + 8 * i;
      if (cc >= g.N) break;
      const double y = tile[w + 8 * i][lane];
      C[cc * ldc + r] = y;
      if (C32) C32[cc * ldc + r] = (float)y;
    }
}

// out[r] = sum_c C[r][c]^2: one warp per row
__global__ void __launch_bounds__(256) out_rowsq_kernel(const OutArgs g, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (r >= g.rows) return;
  const int sa = g.sa[r];
  double s = 0.0;
  for (int64_t c = 2 * lane; c < g.N; c += 64) {
    const double2 y = value2(g, r, c, sa);
    s = fma(y.x, y.x, s);
    if (c + 1 < g.N) s = fma(y.y, y.y, s);
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[r] = s;
}

// Entries at and below the diagonal of rows row0 .. of C (row-major); add: to what is there (the next
// K panel).  8 rows x 64 columns per CTA
__global__ void __launch_bounds__(256) out_lower_kernel(const OutArgs g, int64_t row0, int add, double* __restrict__ C,
                                                        int64_t ldc) {
  const int64_t r = (int64_t)blockIdx.y * 8 + (threadIdx.x >> 5), c = (int64_t)blockIdx.x * 64 + 2 * (threadIdx.x & 31);
  if (r >= g.rows || c > row0 + r) return;
  const double2 y = value2(g, r, c, g.sa[r]);
  double* o = C + (row0 + r) * ldc + c;
  o[0] = add ? o[0] + y.x : y.x;
  if (c + 1 <= row0 + r) o[1] = add ? o[1] + y.y : y.y;
}

struct Buffers {  // freed with the stream idle
  cudaStream_t st;
  std::vector<void*> p;
  ~Buffers() {
    cudaStreamSynchronize(st);
    for (void* q : p) cudaFree(q);
  }
  template <typename T>
  bool get(T** out, int64_t count) {
    void* v = nullptr;
    if (cudaMalloc(&v, (size_t)std::max<int64_t>(count, 1) * sizeof(T)) != cudaSuccess) {
      (void)cudaGetLastError();
      return false;
    }
    p.push_back(v);
    *out = static_cast<T*>(v);
    return true;
  }
};

double root_of(int64_t K) { return std::sqrt((double)K) * (1.0 + 1e-9); }
int64_t pad(int64_t x, int64_t m) { return cdiv(x, m) * m; }

template <typename T>
void rows_to_residues(const T* X, int64_t ldx, int64_t K, int64_t Kp, int64_t rows, int* sc, bf16* d, cudaStream_t st) {
  { row_scales_kernel<T><<<(unsigned)rows, 256, 0, st>>>(X, ldx, K, root_of(K), sc); count_launch(); }
  { row_residues_kernel<T><<<dim3((unsigned)rows, (unsigned)cdiv(Kp, 512)), 256, 0, st>>>(X, ldx, K, Kp, rows, sc, d); count_launch(); }
}

gdml_status finish(int* err, cudaStream_t st, const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(GDML_ERR_CUDA, std::string(what) + " launch: " + cudaGetErrorString(e));
  int h = 0;
  if (cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return fail(GDML_ERR_CUDA, std::string(what) + ": synchronise");
  if (h) return fail(GDML_ERR_TIMEOUT, std::string(what) + ": a tcgen05 pipeline wait timed out (code " + std::to_string(h) + ")");
  return GDML_OK;
}

}  // namespace

gdml_status rns_gemm_tall(const double* A, int64_t n, int64_t K, const double* B, int64_t NB, int64_t ldb, bool tri_b,
                          bool rowsq, double* out, float* out32, cudaStream_t st) {
  if (n <= 0 || K <= 0 || NB <= 0 || !A || !B || !out) return fail(GDML_ERR_ARG, "rns_gemm_tall: bad arguments");
  if (NB > ((int64_t)1 << 24) || K > ((int64_t)1 << 24)) return fail(GDML_ERR_ARG, "rns_gemm_tall: sizes too large");
  const char* what = "residue tall gemm";
  RnsProduct q;
  q.Kp = pad(K, 64);
  q.ldo = pad(NB, 16);
  q.shape = tri_b ? RNS_TRI : RNS_FULL;
  q.N = q.Rb = NB;
  // rows per panel: whole tiles whose residues, in and out, fit the scratch
  const int64_t per_row = 2 * NM * (q.Kp + q.ldo);
  int64_t P = std::max<int64_t>(256, std::min<int64_t>(pad(n, 256), kScratch / per_row / 256 * 256));
  q.M = std::min(P, n);
  rns_product_shape(q, 1);
  if (q.slabs > 1) P = std::max<int64_t>(256, std::min<int64_t>(P, kScratch / (2 * NM * (q.Kp + q.slabs * q.ldo)) / 256 * 256));
  Buffers buf{st, {}};
  bf16 *a = nullptr, *b = nullptr;
  int *sa = nullptr, *sb = nullptr, *err = nullptr;
  if (!buf.get(&b, NM * NB * q.Kp) || !buf.get(&a, NM * P * q.Kp) || !buf.get(&q.out, (int64_t)q.slabs * NM * P * q.ldo) ||
      !buf.get(&sa, P) || !buf.get(&sb, NB) || !buf.get(&err, 1))
    return fail(GDML_ERR_OOM, std::string(what) + ": cudaMalloc failed");
  if (cudaMemsetAsync(err, 0, sizeof(int), st) != cudaSuccess) return fail(GDML_ERR_CUDA, what);
  rows_to_residues(B, ldb, K, q.Kp, NB, sb, b, st);
  q.A = a;
  q.B = b;
  q.Ra = P;
  for (int64_t p0 = 0; p0 < n; p0 += P) {
    q.M = std::min(P, n - p0);
    const unsigned rt = (unsigned)cdiv(q.M, 32);
    { col_scales_kernel<<<rt, 1024, 0, st>>>(A, n, p0, q.M, K, root_of(K), sa); count_launch(); }
    { col_residues_kernel<<<dim3(rt, (unsigned)(q.Kp / 64)), 256, 0, st>>>(A, n, p0, q.M, K, q.Kp, P, sa, a); count_launch(); }
    const gdml_status s = rns_product(q, err, st);
    if (s != GDML_OK) return s;
    const OutArgs o{q.out, q.slabs, q.M, q.ldo, NB, (int)cdiv(q.Kp, rns::kChunk), tri_b ? q.bn : 0, sa, sb};
    if (rowsq) {
      out_rowsq_kernel<<<(unsigned)cdiv(q.M, 8), 256, 0, st>>>(o, out + p0);
      count_launch();
    } else {
      out_cols_kernel<<<dim3(rt, (unsigned)cdiv(NB, 64)), 256, 0, st>>>(o, n, out + p0, out32 ? out32 + p0 : nullptr);
      count_launch();
    }
  }
  return finish(err, st, what);
}

template <typename T>
static gdml_status syrk(const T* X, int64_t k, int64_t K, int64_t ldx, double* C, int64_t ldc, cudaStream_t st) {
  if (k <= 0 || K <= 0) return fail(GDML_ERR_ARG, "rns_syrk_lower: empty sizes");
  const char* what = "residue syrk";
  const int64_t kp = std::min(pad(K, 64), std::min(kKPanel, std::max<int64_t>(rns::kChunk, 4 * kScratch / (2 * NM * k) / 512 * 512)));
  const int64_t np = cdiv(K, kp), Kpan = np == 1 ? kp : pad(cdiv(K, np), 512);  // K entries of a panel
  RnsProduct q;
  q.shape = RNS_LOWER;
  q.Kp = pad(std::min(K, Kpan), 64);
  q.ldo = pad(k, 16);
  // rows of C at a time, and K groups where the tiles are few
  const int64_t P = std::max<int64_t>(256, std::min<int64_t>(pad(k, 256), 2 * kScratch / (2 * NM * q.ldo) / 256 * 256));
  q.M = std::min(P, k);
  q.N = k;
  rns_product_shape(q, (int)std::max<int64_t>(1, 2 * kScratch / (2 * NM * q.ldo * P)));
  Buffers buf{st, {}};
  bf16* a = nullptr;
  int *sc = nullptr, *err = nullptr;
  if (!buf.get(&a, NM * k * q.Kp) || !buf.get(&q.out, (int64_t)q.slabs * NM * P * q.ldo) || !buf.get(&sc, k) || !buf.get(&err, 1))
    return fail(GDML_ERR_OOM, std::string(what) + ": cudaMalloc failed");
  if (cudaMemsetAsync(err, 0, sizeof(int), st) != cudaSuccess) return fail(GDML_ERR_CUDA, what);
  q.A = q.B = a;
  q.Ra = q.Rb = k;
  for (int64_t k0 = 0; k0 < K; k0 += Kpan) {
    const int64_t kn = std::min(Kpan, K - k0);
    q.Kp = pad(kn, 64);
    q.slabs = (int)cdiv(cdiv(q.Kp, rns::kChunk), q.chunks);
    rows_to_residues(X + k0, ldx, kn, q.Kp, k, sc, a, st);
    for (int64_t r0 = 0; r0 < k; r0 += P) {
      q.row0 = r0;
      q.M = std::min(P, k - r0);
      q.N = r0 + q.M;
      const gdml_status s = rns_product(q, err, st);
      if (s != GDML_OK) return s;
      const OutArgs o{q.out, q.slabs, q.M, q.ldo, q.N, (int)cdiv(q.Kp, rns::kChunk), 0, sc + r0, sc};
      out_lower_kernel<<<dim3((unsigned)cdiv(q.N, 64), (unsigned)cdiv(q.M, 8)), 256, 0, st>>>(o, r0, k0 > 0, C, ldc);
      count_launch();
    }
  }
  return finish(err, st, what);
}

gdml_status rns_syrk_lower(const float* X, int64_t k, int64_t K, int64_t ldx, double* C, int64_t ldc, cudaStream_t st) {
  return syrk(X, k, K, ldx, C, ldc, st);
}
gdml_status rns_syrk_lower(const double* X, int64_t k, int64_t K, int64_t ldx, double* C, int64_t ldc, cudaStream_t st) {
  return syrk(X, k, K, ldx, C, ldc, st);
}

}  // namespace gdml
