// gdml_matvec_noalloc: the FP64 force-kernel matvec without a context and
// without any device allocation, for callers that cannot call cudaMalloc.
//
// All working memory (descriptors, Jacobian factors, projections) lives in one file-scope __device__ array sized for
// M <= kNoAllocMaxM geometries of N <= kNoAllocMaxN atoms.  Host code never
// names the array directly: the first call on a device looks up its device
// address with cudaGetSymbolAddress (with that device current) and caches it
// per device; that first call should therefore happen before any stream
// capture.  The cached address belongs to the device's primary context: it
// does not survive cudaDeviceReset, and calls made under another context of
// the same device must not use this entry point.  A stream of another device
// than the current one is rejected.  Every call overwrites the whole region
// it uses before reading it, so nothing has to start at zero; calls that
// overlap on the GPU (different streams, or different host threads on one
// device) race on the array.
#include <mutex>

#include "common.cuh"
#include "kernels.cuh"

namespace gdml {
namespace {

constexpr int64_t kNoAllocMaxM = 128;
constexpr int kNoAllocMaxN = 24;
constexpr int kNoAllocMaxD = kNoAllocMaxN * (kNoAllocMaxN - 1) / 2;
// X, W, 3 G: 5 M D
constexpr int64_t kNoAllocDoubles = 5 * kNoAllocMaxM * kNoAllocMaxD;

static __device__ __align__(256) double g_noalloc_scratch[kNoAllocDoubles];  // 1.4 MB per device

constexpr int kMaxDevices = 64;
std::mutex g_mu;
double* g_scratch_addr[kMaxDevices] = {};

gdml_status scratch_address(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(GDML_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return fail(GDML_ERR_ARG, "device index out of range");
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_scratch_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
      return fail(GDML_ERR_CUDA, std::string("cudaGetSymbolAddress(scratch): ") + cudaGetErrorString(e));
    g_scratch_addr[dev] = static_cast<double*>(p);
  }
  *out = g_scratch_addr[dev];
  return GDML_OK;
}

// Two launches, one CTA per geometry in each, are the whole matvec: at these sizes (M <= 128) the
// chain of eight kernels it replaced spent its time on launches and on tiles that left all but one SM
// idle (N = 6, M = 24: 125 us, 22 us as two).
//
// Geometry a: descriptors x_a, Jacobian factors g_a and w_a = J_a v_a.
__global__ void __launch_bounds__(128) noalloc_geom_kernel(const double* __restrict__ R, const double* __restrict__ v,
                                                           int N, int D, double* __restrict__ X,
                                                           double* __restrict__ G, double* __restrict__ W) {
  __shared__ double r[2][3 * kNoAllocMaxN];  // R_a, v_a
  const int64_t a = blockIdx.x;
  const int B = 3 * N, tid = threadIdx.x;
  for (int l = tid; l < B; l += 128) {
    r[0][l] = R[a * B + l];
    r[1][l] = v[a * B + l];
  }
  __syncthreads();
  for (int p = tid; p < D; p += 128) {
    int i, j;
    pair_of(p, i, j);
    double d[3], d2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      d[c] = r[0][3 * i + c] - r[0][3 * j + c];
      d2 = fma(d[c], d[c], d2);
    }
    const double inv = 1.0 / sqrt(d2), inv3 = inv / d2;
    double w = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double g = d[c] * inv3;
      G[(a * 3 + c) * D + p] = g;
      w = fma(-g, r[1][3 * i + c] - r[1][3 * j + c], w);
    }
    X[a * D + p] = inv;
    W[a * D + p] = w;
  }
}

// Row a of the kernel: r_ab and (x_a - x_b) . w_b for every b (one warp per b), A_ab and
// beta_ab = c^2 S_ab (x_a - x_b) . w_b, then u_a = sum_b A_ab w_b + beta_ab (x_b - x_a) (descriptors over
// the threads, geometries in groups where there are few descriptors) and
// (K v)_a = J_a^T u_a (+ lambda v_a).
constexpr int kRowThreads = 512;
__global__ void __launch_bounds__(kRowThreads) noalloc_row_kernel(const double* __restrict__ X,
                                                                  const double* __restrict__ G,
                                                                  const double* __restrict__ W,
                                                                  const double* __restrict__ v, int64_t M, int N, int D,
                                                                  double c, double lam, int add_lambda,
                                                                  double* __restrict__ out) {
  __shared__ double xa[kNoAllocMaxD], A[kNoAllocMaxM], beta[kNoAllocMaxM], part[kRowThreads], u[kNoAllocMaxD];
  const int64_t a = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n = (int)M;
  for (int p = tid; p < D; p += kRowThreads) xa[p] = X[a * D + p];
  __syncthreads();
  const double c2_3 = c * c / 3.0;
  for (int b = warp; b < n; b += kRowThreads / 32) {
    double r2 = 0.0, T = 0.0;
    for (int p = lane; p < D; p += 32) {
      const double d = xa[p] - X[(int64_t)b * D + p];
      r2 = fma(d, d, r2);
      T = fma(d, W[(int64_t)b * D + p], T);
    }
    for (int o = 16; o > 0; o >>= 1) {
      r2 += __shfl_xor_sync(0xffffffffu, r2, o);
      T += __shfl_xor_sync(0xffffffffu, T, o);
    }
    if (lane == 0) {
      const double r = b == (int)a ? 0.0 : sqrt(r2);
      const double s = c2_3 * exp(-c * r);
      A[b] = s * (1.0 + c * r);
      beta[b] = c * c * s * T;
    }
  }
  __syncthreads();
  const int groups = max(1, kRowThreads / (32 * ((D + 31) / 32)));  // of geometries
  const int width = kRowThreads / groups;
  const int grp = tid / width;
  for (int p0 = 0; p0 < D; p0 += width) {
    const int p = p0 + tid - grp * width;
    double s = 0.0;
    if (grp < groups && p < D)
      for (int b = grp; b < n; b += groups)
        s = fma(A[b], W[(int64_t)b * D + p], fma(beta[b], X[(int64_t)b * D + p] - xa[p], s));
    part[tid] = s;
    __syncthreads();
    if (grp == 0 && p < D) {
      for (int g = 1; g < groups; ++g) s += part[g * width + tid];
      u[p] = s;
    }
    __syncthreads();
  }
  const int B = 3 * N;
  for (int o = tid >> 2; o < B; o += kRowThreads / 4) {  // four lanes per output
    const int i = o / 3, q = o - 3 * i, sub = tid & 3;
    double s = 0.0;
    for (int j = sub; j < N; j += 4) {
      if (j == i) continue;
      const int p = pair_idx(i, j);
      const double y = G[(a * 3 + q) * D + p] * u[p];
      s += i > j ? -y : y;  // dx_p/dR_i = -g_p if i is the first atom of p, else +g_p
    }
    const unsigned lanes = 0xfu << (lane & ~3);
    s += __shfl_xor_sync(lanes, s, 1);
    s += __shfl_xor_sync(lanes, s, 2);
    if (sub == 0) {
      if (add_lambda) s = fma(lam, v[a * B + o], s);
      out[a * B + o] = s;
    }
  }
}

}  // namespace
}  // namespace gdml

using namespace gdml;

extern "C" gdml_status gdml_matvec_noalloc(const double* R_dev, int64_t M, int32_t N, double sigma, double lambda,
                                           const double* v_dev, double* out_dev, int32_t add_lambda,
                                           void* cuda_stream) {
  clear_msg();
  if (!R_dev || !v_dev || !out_dev || v_dev == out_dev) return fail(GDML_ERR_ARG, "matvec_noalloc: bad pointers");
  if (M < 1 || M > kNoAllocMaxM || N < 2 || N > kNoAllocMaxN)
    return fail(GDML_ERR_ARG, "matvec_noalloc: needs 1 <= M <= " + std::to_string(kNoAllocMaxM) +
                                  " geometries and 2 <= N <= " + std::to_string(kNoAllocMaxN) + " atoms");
  if (!(sigma > 0.0) || !(lambda >= 0.0)) return fail(GDML_ERR_ARG, "matvec_noalloc: need sigma > 0, lambda >= 0");
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (st) {  // the scratch address is the current device's: the stream must belong to it
    int cur = 0, sdev = 0;
    cudaError_t e = cudaGetDevice(&cur);
    if (e == cudaSuccess) e = cudaStreamGetDevice(st, &sdev);
    if (e != cudaSuccess) return fail(GDML_ERR_CUDA, std::string("matvec_noalloc: ") + cudaGetErrorString(e));
    if (sdev != cur)
      return fail(GDML_ERR_ARG, "matvec_noalloc: the stream belongs to device " + std::to_string(sdev) +
                                    " but device " + std::to_string(cur) + " is current");
  }
  double* base = nullptr;
  gdml_status s = scratch_address(&base);
  if (s != GDML_OK) return s;
  const int D = N * (N - 1) / 2;
  const double c = std::sqrt(5.0) / sigma;
  double* X = base;
  double* W = X + M * D;
  double* G = W + M * D;
  { noalloc_geom_kernel<<<(unsigned)M, 128, 0, st>>>(R_dev, v_dev, N, D, X, G, W); count_launch(); }
  { noalloc_row_kernel<<<(unsigned)M, kRowThreads, 0, st>>>(X, G, W, v_dev, M, N, D, c, lambda, add_lambda ? 1 : 0, out_dev); count_launch(); }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(GDML_ERR_CUDA, std::string("matvec_noalloc: ") + cudaGetErrorString(e));
  return GDML_OK;
}
