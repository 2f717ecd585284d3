// Geometry-side kernels of the force-kernel matvec (Sec. 2.1), FP64.
//
//  desc_jac   x_{a,p} = 1/|R_i - R_j|,  g_{a,p} = (R_i - R_j)/|R_i - R_j|^3  (p <-> (i, j), i > j)
//  center     xc_a = x_a - mean_b x_b   (the kernel only sees differences x_a - x_b,
//             so centring is exact and keeps the low-precision contractions small)
//  dist_tab   r_ab = |x_a - x_b|, S_ab = (c^2/3) e^{-c r_ab}, A_ab = S_ab (1 + c r_ab)
//  kdiag      diag(K)_{a,(i,q)} = (c^2/3) sum_{p owns i} g_{a,p,q}^2   (K_aa = (c^2/3) J_a^T J_a)
//  proj       w_a = J_a v_a:  w_{a,p} = -g_{a,p} . (v_{a,i} - v_{a,j});  t_a = xc_a . w_a
//  beta       beta_ab = c^2 S_ab (T_ab - t_b), T = Xc W^T; rowsum_a = sum_b beta_ab
//  backproj   (K v)_a = J_a^T u'_a with u'_a = U_a - rowsum_a xc_a, plus lambda v
//  kcol       columns K[:, c] = J_a^T H_ab J_b e_l for a list of column indices c = b*3N + l
//  center_like   query descriptors centred on the training centre (force prediction; dist_tab
//             also makes the tables of query geometries against the training set)
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"
#include "rns.cuh"

namespace gdml {

__global__ void desc_jac_kernel(const double* __restrict__ R, int64_t M, int N, int D,
                                double* __restrict__ X, double* __restrict__ G) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= M * D) return;
  int64_t a = t / D;
  int p = (int)(t - a * D);
  int i, j;
  pair_of(p, i, j);
  const double* Ra = R + a * N * 3;
  double dx = Ra[3 * i] - Ra[3 * j], dy = Ra[3 * i + 1] - Ra[3 * j + 1], dz = Ra[3 * i + 2] - Ra[3 * j + 2];
  double r2 = dx * dx + dy * dy + dz * dz;
  double r = sqrt(r2);
  double inv_r = 1.0 / r;
  double inv_r3 = inv_r / r2;
  X[t] = inv_r;
  G[3 * t] = dx * inv_r3;
  G[3 * t + 1] = dy * inv_r3;
  G[3 * t + 2] = dz * inv_r3;
}

// column means of X in a fixed order, then Xc = X - mean
__global__ void center_kernel(const double* __restrict__ X, int64_t M, int D, double* __restrict__ Xc) {
  __shared__ double part[8][33];
  const int col = blockIdx.x * 32 + (threadIdx.x & 31);
  const int row0 = threadIdx.x >> 5;  // 0..7
  double s = 0.0;
  if (col < D)
    for (int64_t a = row0; a < M; a += 8) s += X[a * D + col];
  part[row0][threadIdx.x & 31] = s;
  __syncthreads();
  double mean = 0.0;
  for (int r = 0; r < 8; ++r) mean += part[r][threadIdx.x & 31];
  mean /= (double)M;
  if (col < D)
    for (int64_t a = row0; a < M; a += 8) Xc[a * D + col] = X[a * D + col] - mean;
}

// S_ab, A_ab from r_ab = |x_a - x_b| for rows x_a of Xa against rows x_b of X, r straight from
// differences (no Gram-matrix cancellation); S has row stride M, A row stride ldA.  same: Xa is X
// (r_aa = 0 exactly).  8 U x 32 outputs per CTA of 256 threads, U per thread; bound by the FP64 pipe
// (two operations per entry and pair), so U is the one that spreads the tiles most evenly (Q = 300
// against M = 1000, D = 210: 398 us with U = 4, 290 us with U = 1).
template <int U>
__global__ void dist_tab_kernel(const double* __restrict__ Xa, int64_t Q, const double* __restrict__ X, int64_t M,
                                int D, double c, int same, double* __restrict__ S, double* __restrict__ A,
                                int64_t ldA) {
  __shared__ double xa[8 * U][33], xb[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // ty 0..7
  const int64_t a0 = (int64_t)blockIdx.y * (8 * U), b0 = (int64_t)blockIdx.x * 32;
  double acc[U];
#pragma unroll
  for (int u = 0; u < U; ++u) acc[u] = 0.0;
  for (int p0 = 0; p0 < D; p0 += 32) {
    const int p = p0 + tx;
    for (int rr = ty; rr < 32; rr += 8) {
      const int64_t ra = a0 + rr, rb = b0 + rr;
      if (rr < 8 * U) xa[rr][tx] = (ra < Q && p < D) ? Xa[ra * D + p] : 0.0;
      xb[rr][tx] = (rb < M && p < D) ? X[rb * D + p] : 0.0;
    }
    __syncthreads();
    const int qn = min(32, D - p0);
#pragma unroll 4
    for (int q = 0; q < qn; ++q) {
      const double vb = xb[tx][q];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const double d = xa[ty + 8 * u][q] - vb;
        acc[u] = fma(d, d, acc[u]);
      }
    }
    __syncthreads();
  }
  const double c2_3 = c * c / 3.0;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t a = a0 + ty + 8 * u, b = b0 + tx;
    if (a < Q && b < M) {
      const double r = (same && a == b) ? 0.0 : sqrt(acc[u]);
      const double s = c2_3 * exp(-c * r);
      S[a * M + b] = s;
      A[a * ldA + b] = s * (1.0 + c * r);
    }
  }
}

// Xqc = Xq - mu, mu = X_0 - Xc_0: query descriptors centred on the training set's centre,
// so that (xq - mu) . w_b - xc_b . w_b = (x_q - x_b) . w_b
__global__ void center_like_kernel(const double* __restrict__ Xq, int64_t Q, int D, const double* __restrict__ X,
                                   const double* __restrict__ Xc, double* __restrict__ Xqc) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= Q * D) return;
  const int p = (int)(t % D);
  Xqc[t] = Xq[t] - (X[p] - Xc[p]);
}

__global__ void kdiag_kernel(const double* __restrict__ G, int64_t M, int N, int D, double c2_3,
                             double* __restrict__ diag) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int B = 3 * N;
  if (t >= M * B) return;
  int64_t a = t / B;
  int l = (int)(t - a * B), i = l / 3, q = l - 3 * (l / 3);
  const double* Ga = G + a * D * 3;
  double s = 0.0;
  // branch-free so that the loads of successive j are independent and in flight together
#pragma unroll 4
  for (int j = 0; j < N; ++j) {
    const bool skip = j == i;
    const double gl = Ga[3 * (skip ? 0 : pair_idx(i, j)) + q];  // always a valid address
    const double g = skip ? 0.0 : gl;
    s = fma(g, g, s);
  }
  diag[t] = c2_3 * s;
}

// W_a = J_a v_a and t_a = xc_a . w_a; one CTA per geometry, one descriptor p per thread (a
// second round when D exceeds the block): the G loads are issued before v_a is staged, the
// pair (i, j) of p decoded in FP32, and t_a reduced in a fixed order (shuffle tree, then warps).
__global__ void __launch_bounds__(1024) proj_cta_kernel(const double* __restrict__ G, const double* __restrict__ Xc,
                                                        const double* __restrict__ v, int64_t M, int N, int D,
                                                        double* __restrict__ W, int64_t ldW, double* __restrict__ t) {
  extern __shared__ double sv[];  // 3N
  __shared__ double red[32];
  const int64_t a = blockIdx.x;
  const int B = 3 * N;
  const double* Ga = G + a * D * 3;
  int p = threadIdx.x;
  double g0 = 0.0, g1 = 0.0, g2 = 0.0, xc = 0.0;
  if (p < D) {
    g0 = Ga[3 * p];
    g1 = Ga[3 * p + 1];
    g2 = Ga[3 * p + 2];
    xc = Xc[a * D + p];
  }
  for (int l = threadIdx.x; l < B; l += blockDim.x) sv[l] = v[a * B + l];
  __syncthreads();
  double part = 0.0;
  for (; p < D; p += blockDim.x) {
    if (p >= (int)blockDim.x) {  // later rounds (D > blockDim)
      g0 = Ga[3 * p];
      g1 = Ga[3 * p + 1];
      g2 = Ga[3 * p + 2];
      xc = Xc[a * D + p];
    }
    int i, j;
    pair_of(p, i, j);
    const double w = -(g0 * (sv[3 * i] - sv[3 * j]) + g1 * (sv[3 * i + 1] - sv[3 * j + 1]) +
                       g2 * (sv[3 * i + 2] - sv[3 * j + 2]));
    W[a * ldW + p] = w;
    part = fma(xc, w, part);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if (lane == 0) red[warp] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    t[a] = s;
  }
}

// beta_ab = c^2 S_ab (T_ab - t_b) into Pb[a*ldP + b]; rowsum_a = sum_b beta_ab
template <int THREADS>
__global__ void beta_kernel(const double* __restrict__ T, const double* __restrict__ S,
                            const double* __restrict__ t, int64_t M, double c2,
                            double* __restrict__ Pb, int64_t ldP, double* __restrict__ rowsum) {
  __shared__ double red[THREADS / 32];
  const int64_t a = blockIdx.x;
  double part = 0.0;
  for (int64_t b = threadIdx.x; b < M; b += THREADS) {
    double beta = c2 * S[a * M + b] * (T[a * M + b] - t[b]);
    Pb[a * ldP + b] = beta;
    part += beta;
  }
  double s = block_sum<THREADS>(part, red);
  if (threadIdx.x == 0) rowsum[a] = s;
}

// (K v)_a = J_a^T (U_a - rowsum_a xc_a) (+ lambda v_a). One CTA per geometry.
template <typename TU>
__global__ void backproj_kernel(const TU* __restrict__ U, int64_t ldU, int splits, int64_t split_stride,
                                const double* __restrict__ rowsum,
                                const double* __restrict__ Xc, const double* __restrict__ G,
                                const double* __restrict__ v, int N, int D, double lam, int add_lambda,
                                double* __restrict__ out) {
  extern __shared__ double sh_u[];  // D
  const int64_t a = blockIdx.x;
  const double rs = rowsum[a];
  for (int p = threadIdx.x; p < D; p += blockDim.x) {
    double u = 0.0;
    for (int s = 0; s < splits; ++s) u += (double)U[s * split_stride + a * ldU + p];
    sh_u[p] = u - rs * Xc[a * D + p];
  }
  __syncthreads();
  const int B = 3 * N;
  const double* Ga = G + a * D * 3;
  for (int l = threadIdx.x; l < B; l += blockDim.x) {
    int i = l / 3, q = l - 3 * i;
    double s = 0.0;
#pragma unroll 4
    for (int j = 0; j < N; ++j) {  // branch-free: independent loads of successive j
      const bool skip = j == i;
      const int p = skip ? 0 : pair_idx(i, j);
      const double gj = Ga[3 * p + q] * sh_u[p];
      s += skip ? 0.0 : ((i > j) ? -gj : gj);  // dx_p/dR_i = -g_p if i is the first atom of p, else +g_p
    }
    if (add_lambda) s = fma(lam, v[a * B + l], s);
    out[a * B + l] = s;
  }
}

// Columns of K: out[c*n + a*3N + l'] = (J_a^T H_ab J_b e_l)_{l'} for cols[c] = b*3N + l.
// grid (M, ceil(ncols/colsPerCta)); CTA handles target geometry a for several columns.
__global__ void kcol_kernel(const int64_t* __restrict__ cols, int64_t ncols, int colsPerCta,
                            const double* __restrict__ X, const double* __restrict__ G,
                            const double* __restrict__ S, const double* __restrict__ A, int64_t ldA,
                            int64_t M, int N, int D, double c2, double* __restrict__ out, int64_t ldo,
                            const int* __restrict__ stop_flag) {
  if (stop_flag && *stop_flag) return;
  extern __shared__ double sh[];
  double* delta = sh;       // D
  double* u = sh + D;       // D
  double* wsp = sh + 2 * D; // N (w on the pairs (i, j), indexed by partner j)
  __shared__ double s_dot;
  const int64_t a = blockIdx.x;
  const int B = 3 * N;
  const double* Xa = X + a * D;
  const double* Ga = G + a * D * 3;
  int64_t c_begin = (int64_t)blockIdx.y * colsPerCta;
  int64_t c_end = c_begin + colsPerCta < ncols ? c_begin + colsPerCta : ncols;
  int64_t last_b = -1;
  for (int64_t c = c_begin; c < c_end; ++c) {
    const int64_t col = cols[c];
    const int64_t b = col / B;
    const int l = (int)(col - b * B), i = l / 3, q = l - 3 * i;
    const double* Xb = X + b * D;
    const double* Gb = G + b * D * 3;
    __syncthreads();
    if (b != last_b) {
      for (int p = threadIdx.x; p < D; p += blockDim.x) delta[p] = Xa[p] - Xb[p];
      last_b = b;
    }
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
      double w = 0.0;
      if (j != i) {
        int p = pair_idx(i, j);
        w = (i > j) ? -Gb[3 * p + q] : Gb[3 * p + q];  // (J_b e_l)_p
      }
      wsp[j] = w;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int j = 0; j < N; ++j)
        if (j != i) s = fma(delta[pair_idx(i, j)], wsp[j], s);
      s_dot = s;
    }
    __syncthreads();
    const double Sab = S[a * M + b], Aab = A[a * ldA + b];
    const double coef = -c2 * Sab * s_dot;
    for (int p = threadIdx.x; p < D; p += blockDim.x) u[p] = coef * delta[p];
    __syncthreads();
    for (int j = threadIdx.x; j < N; j += blockDim.x)
      if (j != i) u[pair_idx(i, j)] += Aab * wsp[j];
    __syncthreads();
    for (int l2 = threadIdx.x; l2 < B; l2 += blockDim.x) {
      int i2 = l2 / 3, q2 = l2 - 3 * i2;
      double s = 0.0;
#pragma unroll 4
      for (int j = 0; j < N; ++j) {
        const bool skip = j == i2;
        const int p = skip ? 0 : pair_idx(i2, j);
        const double gj = Ga[3 * p + q2] * u[p];
        s += skip ? 0.0 : ((i2 > j) ? -gj : gj);
      }
      out[c * ldo + a * B + l2] = s;
    }
  }
}

// Same columns, one warp per geometry a (W warps per CTA, grid (ceil(M/W), ncols)).
// All operands of a geometry (x_a, its Jacobian factors g_a) and of the column's
// geometry b (x_b, w = J_b e_l) are first staged in shared memory with independent,
// coalesced loads; the warp then forms s = delta_(i,.) . w (shuffle reduction),
// u = coef delta + A_ab w on the pairs of atom i, and the 3N outputs J_a^T u from
// shared memory only.  Shared memory: D + N doubles per CTA plus 5 D per warp.
__global__ void __launch_bounds__(256) kcol_warp_kernel(const int64_t* __restrict__ cols,
                                                        const double* __restrict__ X, const double* __restrict__ G,
                                                        const double* __restrict__ S, const double* __restrict__ A,
                                                        int64_t ldA, int64_t M, int N, int D, double c2,
                                                        double* __restrict__ out, int64_t ldo,
                                                        const int* __restrict__ stop_flag) {
  if (stop_flag && *stop_flag) return;
  extern __shared__ double shw[];
  const int W = blockDim.x >> 5;
  double* wsp = shw;            // N: (J_b e_l) on the pairs (i, j), indexed by partner j
  double* sxb = shw + N;        // D: x_b
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* sxa = shw + N + D + (size_t)warp * 5 * D;  // D: x_a
  double* u = sxa + D;                                 // D
  double* sga = u + D;                                 // 3 D: g_a
  const int64_t c = blockIdx.y;
  const int64_t col = cols[c];
  const int B = 3 * N;
  const int64_t b = col / B;
  const int l = (int)(col - b * B), i = l / 3, q = l - 3 * i;
  const double* Xb = X + b * D;
  const double* Gb = G + b * D * 3;
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    double w = 0.0;
    if (j != i) {
      const int p = pair_idx(i, j);
      w = (i > j) ? -Gb[3 * p + q] : Gb[3 * p + q];
    }
    wsp[j] = w;
  }
  for (int p = threadIdx.x; p < D; p += blockDim.x) sxb[p] = Xb[p];
  const int64_t a = (int64_t)blockIdx.x * W + warp;
  const bool live = a < M;
  if (live) {  // eight independent loads in flight per lane, then the shared-memory stores
    const double* Xa = X + a * D;
    const double* Ga = G + a * D * 3;
    for (int e0 = lane; e0 < 4 * D; e0 += 32 * 8) {
      double tmp[8];
#pragma unroll
      for (int u8 = 0; u8 < 8; ++u8) {
        const int e = e0 + 32 * u8;
        tmp[u8] = e < D ? Xa[e] : (e < 4 * D ? Ga[e - D] : 0.0);
      }
#pragma unroll
      for (int u8 = 0; u8 < 8; ++u8) {
        const int e = e0 + 32 * u8;
        if (e < D)
          sxa[e] = tmp[u8];
        else if (e < 4 * D)
          sga[e - D] = tmp[u8];
      }
    }
  }
  __syncthreads();
  if (!live) return;
  double sd = 0.0;
  for (int j = lane; j < N; j += 32)
    if (j != i) {
      const int p = pair_idx(i, j);
      sd = fma(sxa[p] - sxb[p], wsp[j], sd);
    }
  for (int o = 16; o > 0; o >>= 1) sd += __shfl_xor_sync(0xffffffffu, sd, o);
  const double Aab = A[a * ldA + b];
  const double coef = -c2 * S[a * M + b] * sd;
  for (int p = lane; p < D; p += 32) u[p] = coef * (sxa[p] - sxb[p]);
  __syncwarp();
  for (int j = lane; j < N; j += 32)
    if (j != i) u[pair_idx(i, j)] += Aab * wsp[j];
  __syncwarp();
  for (int l2 = lane; l2 < B; l2 += 32) {
    const int i2 = l2 / 3, q2 = l2 - 3 * i2;
    double s = 0.0;
    for (int j = 0; j < N; ++j) {
      const bool skip = j == i2;
      const int p = skip ? 0 : pair_idx(i2, j);
      const double gj = sga[3 * p + q2] * u[p];
      s += skip ? 0.0 : ((i2 > j) ? -gj : gj);
    }
    out[c * ldo + a * B + l2] = s;
  }
}

// ---- double-float helpers for the kernel column (pairs (hi, lo) of FP32 on the FP32 lanes)
__device__ __forceinline__ float2 dfk_split(double x) {
  const float h = __double2float_rn(x);
  return make_float2(h, __double2float_rn(x - (double)h));
}
__device__ __forceinline__ float2 dfk_add(float2 a, float2 b) {  // a + b
  const float s = __fadd_rn(a.x, b.x);
  const float v = __fsub_rn(s, a.x);
  float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, v)), __fsub_rn(b.x, v));
  e = __fadd_rn(e, __fadd_rn(a.y, b.y));
  const float h = __fadd_rn(s, e);
  return make_float2(h, __fsub_rn(e, __fsub_rn(h, s)));
}
__device__ __forceinline__ float2 dfk_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 dfk_mul(float2 a, float2 b) {  // a b
  const float p = __fmul_rn(a.x, b.x);
  float e = fmaf(a.x, b.x, -p);
  e = fmaf(a.x, b.y, e);
  e = fmaf(a.y, b.x, e);
  const float h = __fadd_rn(p, e);
  return make_float2(h, __fsub_rn(e, __fsub_rn(h, p)));
}

// Kernel columns in double-float on the FP32 lanes (DF64/OZAKI contexts): the algebra of
// kcol_warp_kernel with x and g read as float pairs (split once per context) and c^2 S_ab,
// A_ab split on the fly.  GB300's FP64 pipe is a small fraction of its FP32 lanes and the
// FP64 form of this kernel was bound by it; the column is accurate to ~1e-14 of its terms,
// the class of the double-float Schur sums it meets in Algorithm 1.  S and A are symmetric:
// column b is read as row b.  One warp per geometry a, W warps per CTA.
//
// Algorithm 1 (released not null): the grid starts beside the step before and waits for it here; its first
// thread then releases `step`, so that the Schur step that starts beside THIS grid, and acquires it, sees
// what the step before wrote (a grid sees what it waited for; one that a trigger started does not).
__global__ void __launch_bounds__(256) kcol_df_kernel(const int64_t* cols,
                                                      const float2* __restrict__ X2, const float2* __restrict__ G2,
                                                      const double* __restrict__ S, const double* __restrict__ A,
                                                      int64_t ldA, int64_t M, int N, int D, double c2,
                                                      double* __restrict__ out, int64_t ldo,
                                                      const int* stop_flag, unsigned* released, unsigned step) {
  extern __shared__ float2 shf[];
  const int W = blockDim.x >> 5;
  float2* wsp = shf;        // N: +-g_b on the pairs (i, j), indexed by partner j
  float2* sxb = shf + N;    // D: x_b
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* sxa = shf + N + D + (size_t)warp * 5 * D;  // D: x_a - x_b
  float2* u = sxa + D;                                 // D
  float2* sga = u + D;                                 // 3 D: g_a
  const int64_t c = blockIdx.y;
  const int B = 3 * N;
  const int64_t a = (int64_t)blockIdx.x * W + warp;
  const bool live = a < M;
  float2 sab = make_float2(0.f, 0.f), aab = sab;
  // geometry a's operands do not depend on the pivot: their loads go first, before the step that
  // selects it has ended
  if (live) {  // eight independent loads in flight per lane, then the shared-memory stores
    const float2* Xa = X2 + a * D;
    const float2* Ga = G2 + a * D * 3;
    for (int e0 = lane; e0 < 4 * D; e0 += 32 * 8) {
      float2 tmp[8];
#pragma unroll
      for (int u8 = 0; u8 < 8; ++u8) {
        const int e = e0 + 32 * u8;
        tmp[u8] = e < D ? Xa[e] : (e < 4 * D ? Ga[e - D] : make_float2(0.f, 0.f));
      }
#pragma unroll
      for (int u8 = 0; u8 < 8; ++u8) {
        const int e = e0 + 32 * u8;
        if (e < D)
          sxa[e] = tmp[u8];
        else if (e < 4 * D)
          sga[e - D] = tmp[u8];
      }
    }
  }
  grid_wait();
  if (released && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0)
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(released), "r"(step) : "memory");
  if (stop_flag && __ldcg(stop_flag)) return;
  grid_trigger();  // (after the wait and the release: the next kernel needs not poll)
  const int64_t col = __ldcg(cols + c);
  const int64_t b = col / B;
  const int l = (int)(col - b * B), i = l / 3, q = l - 3 * i;
  const float2* Xb = X2 + b * D;
  const float2* Gb = G2 + b * D * 3;
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    float2 w = make_float2(0.f, 0.f);
    if (j != i) {
      const float2 g = Gb[3 * pair_idx(i, j) + q];
      w = (i > j) ? dfk_neg(g) : g;
    }
    wsp[j] = w;
  }
  for (int p = threadIdx.x; p < D; p += blockDim.x) sxb[p] = Xb[p];
  if (live && lane == 0) {
    sab = dfk_mul(dfk_split(c2), dfk_split(S[b * M + a]));
    aab = dfk_split(A[b * ldA + a]);
  }
  __syncthreads();
  if (!live) return;
  sab = make_float2(__shfl_sync(0xffffffffu, sab.x, 0), __shfl_sync(0xffffffffu, sab.y, 0));
  aab = make_float2(__shfl_sync(0xffffffffu, aab.x, 0), __shfl_sync(0xffffffffu, aab.y, 0));
  for (int p = lane; p < D; p += 32) sxa[p] = dfk_add(sxa[p], dfk_neg(sxb[p]));  // x_a - x_b
  __syncwarp();
  float2 sd = make_float2(0.f, 0.f);
  for (int j = lane; j < N; j += 32)
    if (j != i) sd = dfk_add(sd, dfk_mul(sxa[pair_idx(i, j)], wsp[j]));
  for (int o = 16; o > 0; o >>= 1)
    sd = dfk_add(sd, make_float2(__shfl_xor_sync(0xffffffffu, sd.x, o), __shfl_xor_sync(0xffffffffu, sd.y, o)));
  const float2 coef = dfk_neg(dfk_mul(sab, sd));
  for (int p = lane; p < D; p += 32) u[p] = dfk_mul(coef, sxa[p]);
  __syncwarp();
  for (int j = lane; j < N; j += 32)
    if (j != i) {
      const int p = pair_idx(i, j);
      u[p] = dfk_add(u[p], dfk_mul(aab, wsp[j]));
    }
  __syncwarp();
  for (int l2 = lane; l2 < B; l2 += 32) {
    const int i2 = l2 / 3, q2 = l2 - 3 * i2;
    float2 s2 = make_float2(0.f, 0.f);
    for (int j = 0; j < N; ++j) {
      if (j == i2) continue;
      const int p = pair_idx(i2, j);
      const float2 gj = dfk_mul(sga[3 * p + q2], u[p]);
      s2 = dfk_add(s2, (i2 > j) ? dfk_neg(gj) : gj);
    }
    out[c * ldo + a * B + l2] = (double)s2.x + (double)s2.y;
  }
}

// Many kernel columns at once (the Nystrom factor's K_nk, Eq. 5), in double-float like kcol_df_kernel:
//   K[a, col] = J_a^T (A_ab w + coef (x_a - x_b)),  coef = -c^2 S_ab (x_a - x_b) . w,  w = J_b e_col.
// Per entry the second term is a sum of N - 1 products, bound by the FP32 lanes, so it decides the
// layout: a warp takes one atom of NA geometries a against 64 columns, two per lane in packed
// arithmetic (the sums are compensated and combined in FP64), g_a and x_a as broadcasts from shared
// memory, x_b from an array transposed to columns.  w has N - 1 entries (the pairs of one atom), so
// the first term and coef take one pass over them per (a, column).
// N = 42, M = 1001, 1500 columns: 26.7 ms as one warp per (a, column) gathering pairs from shared
// memory, 5.1 ms so.
constexpr int kColBlock = 128;   // columns per CTA
constexpr int kColBatch = 2048;  // columns per launch (their transposed operands: (D + 2 N) float pairs each)

// the columns' operands: XP[p][column pair] (hi, hi, lo, lo), W[j][column] = +-g_b on the pairs (i, j)
// of the column's atom i, XG[j][column] = x_b there
__global__ void kcol_prep_kernel(const int64_t* __restrict__ cols, int64_t ncols, int64_t LC,
                                 const float2* __restrict__ X2, const float2* __restrict__ G2, int N, int D,
                                 float4* __restrict__ XP, float2* __restrict__ W, float2* __restrict__ XG) {
  const int64_t cp = blockIdx.x;
  const int64_t ca = min(2 * cp, ncols - 1), cb = min(2 * cp + 1, ncols - 1);  // (padding repeats the last)
  const int B = 3 * N;
  const int64_t col[2] = {cols[ca], cols[cb]};
  const float2 *x0 = X2 + col[0] / B * D, *x1 = X2 + col[1] / B * D;
  for (int p = threadIdx.x; p < D; p += blockDim.x) {
    const float2 u = x0[p], v = x1[p];
    XP[p * (LC >> 1) + cp] = make_float4(u.x, v.x, u.y, v.y);
  }
  for (int e = threadIdx.x; e < 2 * N; e += blockDim.x) {
    const int h = e >= N ? 1 : 0, j = e - h * N;
    const int64_t b = col[h] / B;
    const int l = (int)(col[h] - b * B), i = l / 3, q = l - 3 * i;
    float2 w = make_float2(0.f, 0.f), x = w;
    if (j != i) {
      const int p = pair_idx(i, j);
      const float2 g = G2[(b * D + p) * 3 + q];
      w = i > j ? dfk_neg(g) : g;
      x = X2[b * D + p];
    }
    W[j * LC + 2 * cp + h] = w;
    XG[j * LC + 2 * cp + h] = x;
  }
}

__device__ __forceinline__ double dfk_double(float2 a) { return (double)a.x + (double)a.y; }

struct df2c {  // compensated sums of two columns
  float2 h, l;
};
// s += g d, g the same for both columns
__device__ __forceinline__ void mac2(df2c& s, float gh, float gl, float2 dh, float2 dl) {
  using namespace rns;
  const float2 p = p_mul(f2(gh), dh);
  float2 e = p_fma(f2(gh), dh, p_mul(p, f2(-1.f)));
  e = p_fma(f2(gh), dl, e);
  e = p_fma(f2(gl), dh, e);
  const float2 t = p_add(s.h, p), bb = p_sub(t, s.h);
  s.l = p_add(s.l, p_add(p_add(p_sub(s.h, p_sub(t, bb)), p_sub(p, bb)), e));
  s.h = t;
}
// (dh, dl) = a - x or x - a for the two columns x
template <bool NEG>
__device__ __forceinline__ void diff2(float ah, float al, float4 x, float2& dh, float2& dl) {
  using namespace rns;
  const float2 xh = make_float2(x.x, x.y), xl = make_float2(x.z, x.w);
  const float2 uh = NEG ? xh : f2(ah), vh = NEG ? f2(ah) : xh, ul = NEG ? xl : f2(al), vl = NEG ? f2(al) : xl;
  const float2 s = p_sub(uh, vh), bb = p_sub(s, uh);
  const float2 e = p_add(p_sub(p_sub(uh, p_sub(s, bb)), p_add(vh, bb)), p_sub(ul, vl));
  dh = p_add(s, e);
  dl = p_sub(e, p_sub(dh, s));
}

template <int NA>
__global__ void __launch_bounds__(256) kcol_bulk_df_kernel(const int64_t* __restrict__ cols, int64_t ncols, int64_t LC,
                                                           const float4* __restrict__ XP, const float2* __restrict__ W,
                                                           const float2* __restrict__ XG,
                                                           const float2* __restrict__ X2,
                                                           const float2* __restrict__ G2,
                                                           const double* __restrict__ S,
                                                           const double* __restrict__ A, int64_t ldA, int64_t M,
                                                           int N, int D, double c2, double* __restrict__ out,
                                                           int64_t ldo) {
  extern __shared__ float4 shb[];
  __shared__ double s_coef[NA][kColBlock], s_aab[NA][kColBlock], s_self[NA][3][kColBlock];
  __shared__ int s_atom[kColBlock];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int B = 3 * N;
  const int64_t a0 = (int64_t)blockIdx.x * NA, c0 = (int64_t)blockIdx.y * kColBlock;
  // pair p of geometry a: (g_0, g_1), (g_2, x_a)
  for (int e = tid; e < NA * D; e += 256) {
    const int ai = e >= D ? 1 : 0, p = e - ai * D;
    const int64_t r = min(a0 + ai, M - 1) * D + p;
    const float2 g0 = G2[3 * r], g1 = G2[3 * r + 1], g2 = G2[3 * r + 2], x = X2[r];
    shb[2 * e] = make_float4(g0.x, g0.y, g1.x, g1.y);
    shb[2 * e + 1] = make_float4(g2.x, g2.y, x.x, x.y);
  }
  __syncthreads();
  if (tid < NA * kColBlock) {  // one thread per (a, column)
    const int ai = tid / kColBlock, cl = tid % kColBlock;
    const int64_t c = c0 + cl, a = min(a0 + ai, M - 1);
    const int64_t col = cols[min(c, ncols - 1)], b = col / B;
    const int i = (int)(col - b * B) / 3;
    const float4* sg = shb + 2 * ai * D;
    float2 sd = make_float2(0.f, 0.f), self[3] = {sd, sd, sd};
    if (c < LC)
      for (int j = 0; j < N; ++j) {
        if (j == i) continue;
        const int p = pair_idx(i, j);
        const float4 ga = sg[2 * p], gb = sg[2 * p + 1];
        const float2 w = W[j * LC + c], x = XG[j * LC + c];
        sd = dfk_add(sd, dfk_mul(dfk_add(make_float2(gb.z, gb.w), dfk_neg(x)), w));
        const float2 v = i > j ? dfk_neg(w) : w;
        self[0] = dfk_add(self[0], dfk_mul(make_float2(ga.x, ga.y), v));
        self[1] = dfk_add(self[1], dfk_mul(make_float2(ga.z, ga.w), v));
        self[2] = dfk_add(self[2], dfk_mul(make_float2(gb.x, gb.y), v));
      }
    const double aab = A[b * ldA + a];
    s_coef[ai][cl] = -(c2 * S[b * M + a]) * dfk_double(sd);
    s_aab[ai][cl] = aab;
#pragma unroll
    for (int q = 0; q < 3; ++q) s_self[ai][q][cl] = aab * dfk_double(self[q]);
    if (ai == 0) s_atom[cl] = i;
  }
  __syncthreads();
  const int64_t hc = LC >> 1;
  for (int task = warp; task < 2 * N; task += 8) {  // (64 columns, atom)
    const int chunk = task >= N ? 1 : 0, i = task - chunk * N;
    const int64_t cb = c0 + 64 * chunk;
    if (cb >= ncols) break;
    const float4* xp = XP + (cb >> 1) + lane;
    df2c y[NA][3];
#pragma unroll
    for (int k = 0; k < NA; ++k)
#pragma unroll
      for (int q = 0; q < 3; ++q) y[k][q] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    auto term = [&](int p, auto neg) {
      const float4 x = xp[p * hc];
#pragma unroll
      for (int k = 0; k < NA; ++k) {
        const float4 ga = shb[2 * (k * D + p)], gb = shb[2 * (k * D + p) + 1];
        float2 dh, dl;
        diff2<decltype(neg)::value>(gb.z, gb.w, x, dh, dl);
        mac2(y[k][0], ga.x, ga.y, dh, dl);
        mac2(y[k][1], ga.z, ga.w, dh, dl);
        mac2(y[k][2], gb.x, gb.y, dh, dl);
      }
    };
    // J_a^T has +g on the pairs' first atoms, -g on their second
#pragma unroll 2
    for (int j = 0; j < i; ++j) term(pair_idx(i, j), std::true_type{});
#pragma unroll 2
    for (int j = i + 1; j < N; ++j) term(pair_idx(i, j), std::false_type{});
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int cl = 64 * chunk + 2 * lane + v;
      if (c0 + cl >= ncols) break;
      const int ic = s_atom[cl];
      const double w = ic == i ? 0.0 : (i > ic ? -1.0 : 1.0) * dfk_double(W[i * LC + c0 + cl]);
      const int p = ic == i ? 0 : pair_idx(i, ic);
#pragma unroll
      for (int k = 0; k < NA; ++k) {
        if (a0 + k >= M) break;
        const float4 ga = shb[2 * (k * D + p)], gb = shb[2 * (k * D + p) + 1];
        const float2 g[3] = {make_float2(ga.x, ga.y), make_float2(ga.z, ga.w), make_float2(gb.x, gb.y)};
        double* o = out + (c0 + cl) * ldo + (a0 + k) * B + 3 * i;
        const double coef = s_coef[k][cl], aw = s_aab[k][cl] * w;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const double t = ic == i ? s_self[k][q][cl] : aw * dfk_double(g[q]);
          o[q] = fma(coef, dfk_double(v ? make_float2(y[k][q].h.y, y[k][q].l.y) : make_float2(y[k][q].h.x, y[k][q].l.x)), t);
        }
      }
    }
  }
}

int64_t kcol_bulk_scratch(int64_t ncols, int N, int D) {
  return std::min<int64_t>(kColBatch, cdiv(ncols, kColBlock) * kColBlock) * (D + 2 * (int64_t)N);
}

template <int NA>
static bool kcol_bulk(const int64_t* cols, int64_t ncols, const float2* X2, const float2* G2, const double* S,
                      const double* A, int64_t ldA, int64_t M, int N, int D, double c, double* out, int64_t ldo,
                      float2* scratch, cudaStream_t st) {
  const size_t smem = 2 * NA * (size_t)D * sizeof(float4);
  if (!allow_smem(kcol_bulk_df_kernel<NA>, smem)) return false;
  for (int64_t c0 = 0; c0 < ncols; c0 += kColBatch) {
    const int64_t nc = std::min<int64_t>(kColBatch, ncols - c0), LC = cdiv(nc, kColBlock) * kColBlock;
    float4* XP = reinterpret_cast<float4*>(scratch);
    float2 *W = scratch + LC * D, *XG = W + LC * N;
    { kcol_prep_kernel<<<(unsigned)(LC / 2), 128, 0, st>>>(cols + c0, nc, LC, X2, G2, N, D, XP, W, XG); count_launch(); }
    const dim3 g((unsigned)cdiv(M, NA), (unsigned)(LC / kColBlock));
    { kcol_bulk_df_kernel<NA><<<g, 256, smem, st>>>(cols + c0, nc, LC, XP, W, XG, X2, G2, S, A, ldA, M, N, D, c * c, out + c0 * ldo, ldo); count_launch(); }
  }
  return true;
}

// Two geometries per CTA halve the loads of x_b; one where their 32 bytes per pair and geometry leave no
// room for two (D > 3400) or where two would leave SMs without a CTA
bool launch_kcol_bulk_df(const int64_t* cols, int64_t ncols, const float2* X2, const float2* G2, const double* S,
                         const double* A, int64_t ldA, int64_t M, int N, int D, double c, double* out, int64_t ldo,
                         float2* scratch, cudaStream_t st) {
  const size_t one = 2 * (size_t)D * sizeof(float4), most = 212 * 1024;
  if (one > most || ncols < 1 || M > 2147483647) return false;
  if (2 * one <= most && cdiv(M, 2) * cdiv(ncols, kColBlock) >= num_sms())
    return kcol_bulk<2>(cols, ncols, X2, G2, S, A, ldA, M, N, D, c, out, ldo, scratch, st);
  return kcol_bulk<1>(cols, ncols, X2, G2, S, A, ldA, M, N, D, c, out, ldo, scratch, st);
}

bool launch_kcol_df(const int64_t* cols, int64_t ncols, const float2* X2, const float2* G2, const double* S,
                    const double* A, int64_t ldA, int64_t M, int N, int D, double c, double* out, int64_t ldo,
                    const int* stop_flag, cudaStream_t st, unsigned* released, unsigned step) {
  const size_t per_warp = 5 * (size_t)D * sizeof(float2), fixed = ((size_t)N + D) * sizeof(float2);
  int W = (int)std::min<size_t>(8, (200 * 1024 - std::min<size_t>(fixed, 200 * 1024)) / per_warp);
  if (W < 1 || ncols > 65535) return false;
  const int sms = num_sms();
  const int64_t want = std::max<int64_t>(1, M * ncols / (2 * (int64_t)sms));
  if (want < W) W = (int)want;
  const size_t wsmem = fixed + W * per_warp;
  (void)allow_smem(kcol_df_kernel, wsmem);
  dim3 g((unsigned)cdiv(M, W), (unsigned)ncols);
  // stop_flag: Algorithm 1's step, which follows the previous one without waiting for it to drain
  { launch_after(stop_flag != nullptr, kcol_df_kernel, g, 32 * W, wsmem, st, cols, X2, G2, S, A, ldA, M, N, D, c * c, out, ldo, stop_flag, released, step); count_launch(); }
  return true;
}

// ---------------------------------------------------------------- launchers
void launch_desc_jac(const double* R, int64_t M, int N, int D, double* X, double* G, cudaStream_t st) {
  int64_t tot = M * D;
  { desc_jac_kernel<<<(unsigned)cdiv(tot, 256), 256, 0, st>>>(R, M, N, D, X, G); count_launch(); }
}
void launch_center(const double* X, int64_t M, int D, double* Xc, cudaStream_t st) {
  { center_kernel<<<(unsigned)cdiv(D, 32), 256, 0, st>>>(X, M, D, Xc); count_launch(); }
}
static void dist_tab(const double* Xa, int64_t Q, const double* X, int64_t M, int D, double c, int same, double* S,
                     double* A, int64_t ldA, cudaStream_t st) {
  int best = 4;
  int64_t best_work = INT64_MAX;
  for (int u : {4, 2, 1}) {
    const int64_t ta = cdiv(Q, 8 * u);
    if (u < 4 && ta > 65535) break;
    const int64_t work = cdiv(ta * cdiv(M, 32), num_sms()) * u;
    if (work < best_work) {
      best_work = work;
      best = u;
    }
  }
  const dim3 grid((unsigned)cdiv(M, 32), (unsigned)cdiv(Q, 8 * best));
  if (best == 4) dist_tab_kernel<4><<<grid, 256, 0, st>>>(Xa, Q, X, M, D, c, same, S, A, ldA);
  else if (best == 2) dist_tab_kernel<2><<<grid, 256, 0, st>>>(Xa, Q, X, M, D, c, same, S, A, ldA);
  else dist_tab_kernel<1><<<grid, 256, 0, st>>>(Xa, Q, X, M, D, c, same, S, A, ldA);
  count_launch();
}
void launch_dist_tab(const double* X, int64_t M, int D, double c, double* S, double* A, int64_t ldA,
                     cudaStream_t st) {
  dist_tab(X, M, X, M, D, c, 1, S, A, ldA, st);
}
void launch_kdiag(const double* G, int64_t M, int N, int D, double c, double* diag, cudaStream_t st) {
  int64_t tot = M * 3 * N;
  { kdiag_kernel<<<(unsigned)cdiv(tot, 256), 256, 0, st>>>(G, M, N, D, c * c / 3.0, diag); count_launch(); }
}
void launch_proj(const double* G, const double* Xc, const double* v, int64_t M, int N, int D, double* W,
                 int64_t ldW, double* t, cudaStream_t st) {
  const unsigned threads = (unsigned)std::min<int64_t>(1024, 32 * cdiv(D, 32));
  { proj_cta_kernel<<<(unsigned)M, threads, 3 * N * sizeof(double), st>>>(G, Xc, v, M, N, D, W, ldW, t); count_launch(); }
}
void launch_beta(const double* T, const double* S, const double* t, int64_t M, double c, double* Pb,
                 int64_t ldP, double* rowsum, cudaStream_t st) {
  { beta_kernel<256><<<(unsigned)M, 256, 0, st>>>(T, S, t, M, c * c, Pb, ldP, rowsum); count_launch(); }
}
void launch_beta_rows(const double* T, const double* S, const double* t, int64_t rows, int64_t M, double c,
                      double* Pb, int64_t ldP, double* rowsum, cudaStream_t st) {
  { beta_kernel<256><<<(unsigned)rows, 256, 0, st>>>(T, S, t, M, c * c, Pb, ldP, rowsum); count_launch(); }
}
void launch_dist_tab_cross(const double* Xq, int64_t Q, const double* X, int64_t M, int D, double c, double* S,
                           double* A, int64_t ldA, cudaStream_t st) {
  dist_tab(Xq, Q, X, M, D, c, 0, S, A, ldA, st);
}
void launch_center_like(const double* Xq, int64_t Q, int D, const double* X, const double* Xc, double* Xqc,
                        cudaStream_t st) {
  { center_like_kernel<<<(unsigned)cdiv(Q * D, 256), 256, 0, st>>>(Xq, Q, D, X, Xc, Xqc); count_launch(); }
}
template <typename TU>
void launch_backproj(const TU* U, int64_t ldU, int splits, int64_t split_stride, const double* rowsum,
                     const double* Xc, const double* G, const double* v, int64_t M, int N, int D, double lam,
                     int add_lambda, double* out, cudaStream_t st) {
  const size_t smem = D * sizeof(double);
  (void)allow_smem(backproj_kernel<TU>, smem);
  { backproj_kernel<TU><<<(unsigned)M, 128, smem, st>>>(U, ldU, splits, split_stride, rowsum, Xc, G, v, N, D,
                                                       lam, add_lambda, out); count_launch(); }
}
template void launch_backproj<double>(const double*, int64_t, int, int64_t, const double*, const double*,
                                      const double*, const double*, int64_t, int, int, double, int, double*,
                                      cudaStream_t);
template void launch_backproj<float>(const float*, int64_t, int, int64_t, const double*, const double*,
                                     const double*, const double*, int64_t, int, int, double, int, double*,
                                     cudaStream_t);

void launch_kcol(const int64_t* cols, int64_t ncols, const double* X, const double* G, const double* S,
                 const double* A, int64_t ldA, int64_t M, int N, int D, double c, double* out, int64_t ldo,
                 const int* stop_flag, cudaStream_t st) {
  // warps per CTA so that the staged operands fit in 200 KB of shared memory
  const size_t per_warp = 5 * (size_t)D * sizeof(double), fixed = ((size_t)N + D) * sizeof(double);
  int W = (int)std::min<size_t>(8, (200 * 1024 - std::min<size_t>(fixed, 200 * 1024)) / per_warp);
  {  // few columns (one per Algorithm 1 step): fewer warps per CTA so the grid covers every SM twice
    const int sms = num_sms();
    const int64_t want = std::max<int64_t>(1, M * ncols / (2 * (int64_t)sms));
    if (want < W) W = (int)want;
  }
  if (W >= 1 && ncols <= 65535) {
    const size_t wsmem = fixed + W * per_warp;
    (void)allow_smem(kcol_warp_kernel, wsmem);
    dim3 g((unsigned)cdiv(M, W), (unsigned)ncols);
    { kcol_warp_kernel<<<g, 32 * W, wsmem, st>>>(cols, X, G, S, A, ldA, M, N, D, c * c, out, ldo, stop_flag); count_launch(); }
    return;
  }
  const int per = 8;
  dim3 grid((unsigned)M, (unsigned)cdiv(ncols, per));
  size_t smem = (2 * (size_t)D + N) * sizeof(double);
  (void)allow_smem(kcol_kernel, smem);
  { kcol_kernel<<<grid, 128, smem, st>>>(cols, ncols, per, X, G, S, A, ldA, M, N, D, c * c, out, ldo, stop_flag); count_launch(); }
}

// *flag = 1 if any of the count values is not finite (NaN or infinite)
__global__ void check_finite_kernel(const double* __restrict__ a, int64_t count, int* __restrict__ flag) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    if (!isfinite(a[i])) {
      *flag = 1;
      return;
    }
}

void launch_check_finite(const double* a, int64_t count, int* flag, cudaStream_t st) {
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(cdiv(count, 256), 4 * num_sms()));
  { check_finite_kernel<<<grid, 256, 0, st>>>(a, count, flag); count_launch(); }
}

// ---------------------------------------------------------------- permutational symmetries
// A symmetry group of S atom permutations acts on the descriptor by pis (S x D: pi_q(p) = the
// pair index of (sigma_q(i), sigma_q(j)) for p = (i, j)) and pinv (its inverse per q).  The
// symmetric force kernel is K_ab = sum_q J_a^T H(x_a, P_q x_b) P_q J_b with (P_q x)_p = x_pi_q(p);
// its training side holds row b S + q = P_q applied to geometry b.

// out[b S + q][p] = in[b][pi_q(p)] for the M rows of `in`; with xcB, also
// t[b S + q] = xcB[b S + q] . out[b S + q].  One CTA (256 threads) per output row.
__global__ void __launch_bounds__(256) sym_gather_kernel(const double* __restrict__ in, int D,
                                                         const int* __restrict__ pis, int S,
                                                         const double* __restrict__ xcB, double* __restrict__ out,
                                                         double* __restrict__ t) {
  __shared__ double red[8];
  const int64_t row = blockIdx.x;
  const int64_t b = row / S;
  const int q = (int)(row - b * S);
  const int* pi = pis + (int64_t)q * D;
  double part = 0.0;
  for (int p = threadIdx.x; p < D; p += blockDim.x) {
    const double v = in[b * D + pi[p]];
    out[row * D + p] = v;
    if (xcB) part = fma(xcB[row * D + p], v, part);
  }
  if (xcB) {
    part = block_sum<256>(part, red);
    if (threadIdx.x == 0) t[row] = part;
  }
}

void launch_sym_gather(const double* in, int64_t M, int D, const int* pis, int S, const double* xcB, double* out,
                       double* t, cudaStream_t st) {
  { sym_gather_kernel<<<(unsigned)(M * S), 256, 0, st>>>(in, D, pis, S, xcB, out, t); count_launch(); }
}

// the value of u = J_a e_l on descriptor entry pp (zero unless pp pairs atom i with another):
// u_(i,j) = -g_(i,j),c for i > j and +g_(i,j),c for i < j
__device__ __forceinline__ double jac_col_at(const double* __restrict__ g, int pp, int i, int cc) {
  int I, J;
  pair_of(pp, I, J);  // I > J
  if (I == i) return -g[3 * pp + cc];
  if (J == i) return g[3 * pp + cc];
  return 0.0;
}

// diag(K) with symmetries: for column l = 3 i + cc of geometry a, with u = J_a e_l,
//   diag_{a,l} = sum_q u^T H(x_a, P_q x_a) P_q u = sum_q A_q (u . P_q u) - c^2 S_q (u . d_q)(P_q u . d_q),
// d_q = x_a - P_q x_a, (P_q u)_p = u_pi(p), so (P_q u) . d = sum_p' u_p' d_pinv(p').
// One CTA (256 threads) per geometry: d_q and its norm by a CTA reduction, then thread l sums
// over the N - 1 pairs of atom i.
__global__ void __launch_bounds__(256) kdiag_sym_kernel(const double* __restrict__ X, const double* __restrict__ G,
                                                        int N, int D, const int* __restrict__ pis,
                                                        const int* __restrict__ pinv, int S, double c,
                                                        double* __restrict__ diag) {
  extern __shared__ double sdq[];  // D
  __shared__ double red[8];
  __shared__ double s_r;
  const int64_t a = blockIdx.x;
  const double* Xa = X + a * D;
  const double* Ga = G + a * D * 3;
  const int B = 3 * N;
  double acc[2] = {0.0, 0.0};  // B <= 384: l = threadIdx.x, threadIdx.x + 256
  for (int q = 0; q < S; ++q) {
    const int* pi = pis + (int64_t)q * D;
    const int* pv = pinv + (int64_t)q * D;
    double part = 0.0;
    for (int p = threadIdx.x; p < D; p += blockDim.x) {
      const double d = Xa[p] - Xa[pi[p]];
      sdq[p] = d;
      part = fma(d, d, part);
    }
    part = block_sum<256>(part, red);  // synchronises: sdq is complete
    if (threadIdx.x == 0) s_r = sqrt(part);
    __syncthreads();
    const double r = s_r;
    const double Sv = (c * c / 3.0) * exp(-c * r), Av = Sv * (1.0 + c * r);
    for (int k = 0; k < 2; ++k) {
      const int l = threadIdx.x + 256 * k;
      if (l >= B) break;
      const int i = l / 3, cc = l - 3 * i;
      double ud = 0.0, vd = 0.0, uv = 0.0;
      for (int j = 0; j < N; ++j) {
        if (j == i) continue;
        const int pp = pair_idx(i, j);
        const double u = (i > j) ? -Ga[3 * pp + cc] : Ga[3 * pp + cc];
        ud = fma(u, sdq[pp], ud);
        vd = fma(u, sdq[pv[pp]], vd);
        uv = fma(u, jac_col_at(Ga, pi[pp], i, cc), uv);
      }
      acc[k] += Av * uv - c * c * Sv * ud * vd;
    }
    __syncthreads();  // sdq is rewritten for the next symmetry
  }
  for (int k = 0; k < 2; ++k) {
    const int l = threadIdx.x + 256 * k;
    if (l < B) diag[a * B + l] = acc[k];
  }
}

void launch_kdiag_sym(const double* X, const double* G, int64_t M, int N, int D, const int* pis, const int* pinv,
                      int S, double c, double* diag, cudaStream_t st) {
  const size_t smem = (size_t)D * sizeof(double);
  (void)allow_smem(kdiag_sym_kernel, smem);
  { kdiag_sym_kernel<<<(unsigned)M, 256, smem, st>>>(X, G, N, D, pis, pinv, S, c, diag); count_launch(); }
}

// Kernel columns with symmetries: column (b, l = 3 i + cc), u = J_b e_l, for every geometry a
//   K[a, col] = J_a^T sum_q [A_q w_q - c^2 S_q (d_q . w_q) d_q],
// w_q = P_q u ((w_q)_pinv(p') = u_p'), d_q = x_a - P_q x_b, S_q and A_q from the context's
// tables at (a, b S + q).  One warp per (geometry a, column), W warps per CTA; FP64.
__global__ void __launch_bounds__(256) kcol_sym_kernel(const int64_t* __restrict__ cols,
                                                       const double* __restrict__ X, const double* __restrict__ G,
                                                       const double* __restrict__ Stab,
                                                       const double* __restrict__ Atab, int64_t ldA, int64_t M,
                                                       int64_t MB, int N, int D, const int* __restrict__ pis,
                                                       const int* __restrict__ pinv, int S, double c2,
                                                       double* __restrict__ out, int64_t ldo,
                                                       const int* __restrict__ stop_flag) {
  if (stop_flag && *stop_flag) return;
  extern __shared__ double shs[];
  const int W = blockDim.x >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* ub = shs + (size_t)warp * (N + 6 * (size_t)D);  // N: u on the pairs (i, j), by partner j
  double* xa = ub + N;                                    // D
  double* ga = xa + D;                                    // 3 D
  double* dq = ga + 3 * D;                                // D
  double* uacc = dq + D;                                  // D
  const int64_t c = blockIdx.y;
  const int64_t col = cols[c];
  const int B = 3 * N;
  const int64_t b = col / B;
  const int l = (int)(col - b * B), i = l / 3, cc = l - 3 * i;
  const int64_t a = (int64_t)blockIdx.x * W + warp;
  if (a >= M) return;  // warp-level work only below
  const double* Xa = X + a * D;
  const double* Ga = G + a * D * 3;
  const double* Xb = X + b * D;
  const double* Gb = G + b * D * 3;
  for (int j = lane; j < N; j += 32) {
    double u = 0.0;
    if (j != i) {
      const int pp = pair_idx(i, j);
      u = (i > j) ? -Gb[3 * pp + cc] : Gb[3 * pp + cc];
    }
    ub[j] = u;
  }
  for (int p = lane; p < D; p += 32) {
    xa[p] = Xa[p];
    uacc[p] = 0.0;
  }
  for (int e = lane; e < 3 * D; e += 32) ga[e] = Ga[e];
  __syncwarp();
  for (int q = 0; q < S; ++q) {
    const int* pi = pis + (int64_t)q * D;
    const int* pv = pinv + (int64_t)q * D;
    for (int p = lane; p < D; p += 32) dq[p] = xa[p] - Xb[pi[p]];
    __syncwarp();
    double sd = 0.0;
    for (int j = lane; j < N; j += 32)
      if (j != i) sd = fma(ub[j], dq[pv[pair_idx(i, j)]], sd);
    for (int o = 16; o > 0; o >>= 1) sd += __shfl_xor_sync(0xffffffffu, sd, o);
    const double Sq = Stab[a * MB + b * S + q], Aq = Atab[a * ldA + b * S + q];
    const double coef = -c2 * Sq * sd;
    for (int p = lane; p < D; p += 32) uacc[p] = fma(coef, dq[p], uacc[p]);
    __syncwarp();
    for (int j = lane; j < N; j += 32)
      if (j != i) {
        const int p = pv[pair_idx(i, j)];
        uacc[p] = fma(Aq, ub[j], uacc[p]);
      }
    __syncwarp();
  }
  for (int l2 = lane; l2 < B; l2 += 32) {
    const int i2 = l2 / 3, q2 = l2 - 3 * i2;
    double s = 0.0;
    for (int j = 0; j < N; ++j) {
      if (j == i2) continue;
      const int p = pair_idx(i2, j);
      const double gj = ga[3 * p + q2] * uacc[p];
      s += (i2 > j) ? -gj : gj;
    }
    out[c * ldo + a * B + l2] = s;
  }
}

bool launch_kcol_sym(const int64_t* cols, int64_t ncols, const double* X, const double* G, const double* Stab,
                     const double* Atab, int64_t ldA, int64_t M, int64_t MB, int N, int D, const int* pis,
                     const int* pinv, int S, double c, double* out, int64_t ldo, const int* stop_flag,
                     cudaStream_t st) {
  const size_t per_warp = ((size_t)N + 6 * (size_t)D) * sizeof(double);
  const int W = (int)std::min<size_t>(8, (200 * 1024) / per_warp);
  if (W < 1 || ncols < 1 || ncols > 65535) return false;
  const size_t smem = W * per_warp;
  if (!allow_smem(kcol_sym_kernel, smem)) return false;
  dim3 g((unsigned)cdiv(M, W), (unsigned)ncols);
  { kcol_sym_kernel<<<g, 32 * W, smem, st>>>(cols, X, G, Stab, Atab, ldA, M, MB, N, D, pis, pinv, S, c * c, out, ldo, stop_flag); count_launch(); }
  return true;
}

}  // namespace gdml
