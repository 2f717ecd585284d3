// Dense FP64 linear algebra for the Nystrom / Woodbury preconditioner (Eqs. 4-5):
//  - blocked Cholesky of a k x k SPD matrix (K_kk and C = lambda I + L^T L)
//  - forward substitution with many right-hand sides (L_k = K_nk L_kk^-T)
//  - the explicit inverse C^-1 = L_C^-T L_C^-1 used by the Woodbury apply
// A non-positive or non-finite pivot is reported through a device status word
// (index of the failing column + 1), never by trapping.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace gdml {

// Two levels of blocking: steps of NB = 32 columns factorise a block of NO = 128, whose update of the
// rest is one product.  An SM's FP64 pipe does under two multiply-adds per cycle, so the work of the
// serial kernels (the diagonal block on one SM, ~NB^3 / 3; a panel's rows at NB^2 / 2 each) decides:
// with steps of 64 the diagonal block took 105 us and a panel 150-190 us.  32 rows per CTA
// spread a panel over all SMs.  The four factorisations and four triangular inverses of a leverage-score build
// at k = 1500: 62 ms with one level of 64, 22 ms so.
constexpr int NB = 32;
constexpr int NO = 128;

// A warp's FP64 operation takes 64 cycles on its quarter of an SM, so all three kernels below use four
// warps per 32 rows: one warp each took 53, 31 and 24 us (22, 18 and 20 us so; 2 us of the two solves are the
// quotients' corrections, see solve_row).
constexpr int kGroup = 4;  // lanes (potrf: warps) that share a row: every fourth column each
constexpr int kOwn = NB / kGroup;

// Unblocked Cholesky of the nb x nb diagonal block at (j0, j0), in place (lower): lane r of every warp
// holds row r, warp w its columns w, w + 4, ...; the column of each step goes through shared memory.
__global__ void __launch_bounds__(32 * kGroup) potrf_diag_kernel(double* __restrict__ A, int64_t lda, int64_t j0,
                                                                 int nb, int* __restrict__ status) {
  __shared__ double colv[2][NB];
  // of even and odd steps, as colv: what is tested after a step's barrier is next written after the next one's
  __shared__ int s_bad[2];
  if (*status) return;
  const int r = threadIdx.x & 31, w = threadIdx.x >> 5;
  double* row = A + (j0 + r) * lda + j0;
  double a[kOwn];
#pragma unroll
  for (int q = 0; q < kOwn; ++q) {
    const int c = kGroup * q + w;
    a[q] = (r < nb && c <= r) ? row[c] : (c == r ? 1.0 : 0.0);
  }
  if (threadIdx.x < 2) s_bad[threadIdx.x] = 0;
  __syncthreads();
  int bad = 0;
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    double* v = colv[c & 1];
    if (w == c % kGroup) {
      const double d = __shfl_sync(0xffffffffu, a[c / kGroup], c);
      const bool ok = d > 0.0 && isfinite(d);
      if (!ok && r == 0) s_bad[c & 1] = c + 1;
      // 1 / l and l = d / l by a correction of each other (one square root, no division)
      const double inv = rsqrt(ok ? d : 1.0), l0 = d * inv;
      const double l = fma(fma(-l0, l0, d), 0.5 * inv, l0);
      a[c / kGroup] = r == c ? l : a[c / kGroup] * inv;
      v[r] = a[c / kGroup];
    }
    __syncthreads();
    bad = s_bad[c & 1];
    if (bad) break;
    const double x = v[r];
#pragma unroll
    for (int q = c / kGroup; q < kOwn; ++q) {
      const int cc = kGroup * q + w;
      if (cc > c) a[q] = fma(-x, v[cc], a[q]);
    }
  }
  if (bad) {
    if (threadIdx.x == 0) *status = (int)(j0 + bad);
    return;
  }
  if (r < nb)
#pragma unroll
    for (int q = 0; q < kOwn; ++q) {
      const int c = kGroup * q + w;
      if (c < nb) row[c] = c <= r ? a[q] : 0.0;
    }
}

// x <- x L^-T for the row x spread over four neighbouring lanes (lane g: entries g, g + 4, ...); inv: the
// reciprocals of L's diagonal, whose product with x is corrected to the rounded quotient (a division takes
// ten times the operations)
__device__ __forceinline__ void solve_row(double (&x)[kOwn], const double (&L)[NB][NB + 1], const double* inv) {
  const int g = threadIdx.x & (kGroup - 1), first = (threadIdx.x & 31) & ~(kGroup - 1);
#pragma unroll
  for (int c = 0; c < NB; ++c) {  // column by column: the updates of the later ones are independent
    if (g == c % kGroup) {
      const double q = x[c / kGroup] * inv[c];
      x[c / kGroup] = fma(fma(-q, L[c][c], x[c / kGroup]), inv[c], q);
    }
    const double xc = __shfl_sync(0xffffffffu, x[c / kGroup], first + c % kGroup);
#pragma unroll
    for (int q = c / kGroup; q < kOwn; ++q) {
      const int cc = kGroup * q + g;
      if (cc > c) x[q] = fma(-xc, L[cc][c], x[q]);
    }
  }
}

// Rows r in [r0, rend): solve x L_jj^T = A[r, j0:j0+nb]  (four lanes per row, 32 rows per CTA).
__global__ void __launch_bounds__(32 * kGroup) trsm_right_kernel(double* __restrict__ A, int64_t lda, int64_t j0,
                                                                 int nb, int64_t r0, int64_t rend,
                                                                 const int* __restrict__ status) {
  __shared__ double L[NB][NB + 1];
  __shared__ double inv[NB];
  if (*status) return;
  const int t = threadIdx.x;
  for (int r = t >> 5; r < NB; r += kGroup) {
    const int c = t & 31;
    const double l = r < nb && c < nb ? A[(j0 + r) * lda + j0 + c] : (r == c ? 1.0 : 0.0);
    L[r][c] = l;
    if (r == c) inv[r] = 1.0 / l;
  }
  const int64_t row = r0 + blockIdx.x * (int64_t)NB + t / kGroup;
  const int g = t & (kGroup - 1);
  double* a = A + row * lda + j0;
  double x[kOwn];
#pragma unroll
  for (int q = 0; q < kOwn; ++q) x[q] = row < rend && kGroup * q + g < nb ? a[kGroup * q + g] : 0.0;
  __syncthreads();
  solve_row(x, L, inv);
  if (row < rend)
#pragma unroll
    for (int q = 0; q < kOwn; ++q)
      if (kGroup * q + g < nb) a[kGroup * q + g] = x[q];
}

// Left forward substitution on a block of rows of B (k x nrhs, row-major, ld):
// B[j0:j0+nb, col] <- L_jj^-1 B[j0:j0+nb, col]; four lanes per column, 32 columns per CTA.
__global__ void __launch_bounds__(32 * kGroup) trsm_left_diag_kernel(const double* __restrict__ Lkk, int64_t ldl,
                                                                     int64_t j0, int nb, double* __restrict__ Bm,
                                                                     int64_t ldb, int64_t nrhs) {
  __shared__ double L[NB][NB + 1];
  __shared__ double B[NB][NB + 1];
  __shared__ double inv[NB];
  const int t = threadIdx.x;
  const int64_t c0 = blockIdx.x * (int64_t)NB;
  for (int r = t >> 5; r < NB; r += kGroup) {
    const int c = t & 31;
    const double l = r < nb && c < nb ? Lkk[(j0 + r) * ldl + j0 + c] : (r == c ? 1.0 : 0.0);
    L[r][c] = l;
    if (r == c) inv[r] = 1.0 / l;
    B[r][c] = r < nb && c0 + c < nrhs ? Bm[(j0 + r) * ldb + c0 + c] : 0.0;
  }
  __syncthreads();
  const int g = t & (kGroup - 1), col = t / kGroup;
  double x[kOwn];
#pragma unroll
  for (int q = 0; q < kOwn; ++q) x[q] = B[kGroup * q + g][col];
  solve_row(x, L, inv);
#pragma unroll
  for (int q = 0; q < kOwn; ++q) B[kGroup * q + g][col] = x[q];
  __syncthreads();
  for (int r = t >> 5; r < nb; r += kGroup) {
    const int c = t & 31;
    if (c0 + c < nrhs) Bm[(j0 + r) * ldb + c0 + c] = B[r][c];
  }
}

__global__ void add_diag_kernel(double* A, int64_t lda, int64_t k, double eps) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < k) A[i * lda + i] += eps;
}

// ---------------------------------------------------------------- host drivers
// In-place lower Cholesky of the k x k row-major matrix A.  status (device int)
// receives 0 on success or (failing column + 1).
void cholesky_inplace(double* A, int64_t k, int* status, cudaStream_t st) {
  for (int64_t o0 = 0; o0 < k; o0 += NO) {
    const int64_t o1 = std::min<int64_t>(k, o0 + NO);
    for (int64_t j0 = o0; j0 < o1; j0 += NB) {
      const int nb = (int)std::min<int64_t>(NB, o1 - j0);
      { potrf_diag_kernel<<<1, 32 * kGroup, 0, st>>>(A, k, j0, nb, status); count_launch(); }
      const int64_t r0 = j0 + nb;
      if (r0 >= k) break;
      { trsm_right_kernel<<<(unsigned)cdiv(k - r0, NB), 32 * kGroup, 0, st>>>(A, k, j0, nb, r0, k, status); count_launch(); }
      // the block's remaining columns: A[r0:, r0:o1] -= L[r0:, j0:r0] L[r0:o1, j0:r0]^T
      if (r0 < o1)
        launch_dgemm<double, double>(true, k - r0, o1 - r0, nb, -1.0, A + r0 * k + j0, k, A + r0 * k + j0, k, 1.0,
                                     A + r0 * k + r0, k, true, st);
    }
    // A22 -= L21 L21^T (lower tiles only)
    if (o1 < k)
      launch_dgemm<double, double>(true, k - o1, k - o1, o1 - o0, -1.0, A + o1 * k + o0, k, A + o1 * k + o0, k, 1.0,
                                   A + o1 * k + o1, k, true, st);
  }
}

// B (k x nrhs row-major) <- Lkk^-1 B  (blocked forward substitution).  lower_rhs: B is lower
// triangular (the identity, for Lkk^-1 itself), so row block j0 and everything it updates
// have no nonzeros past column j0 + nb and only those columns are touched (a third of the
// flops).
void trsm_left_lower(const double* Lkk, int64_t k, double* Bm, int64_t nrhs, cudaStream_t st, bool lower_rhs) {
  for (int64_t o0 = 0; o0 < k; o0 += NO) {
    const int64_t o1 = std::min<int64_t>(k, o0 + NO);
    auto cols = [&](int64_t end) { return lower_rhs ? std::min<int64_t>(nrhs, end) : nrhs; };
    // B[rows b0..b1, :] -= L[b0:b1, c0:c1] B[c0:c1, :]
    auto update = [&](int64_t b0, int64_t b1, int64_t c0, int64_t c1) {
      launch_dgemm<double, double>(false, b1 - b0, cols(c1), c1 - c0, -1.0, Lkk + b0 * k + c0, k, Bm + c0 * nrhs, nrhs,
                                   1.0, Bm + b0 * nrhs, nrhs, false, st);
    };
    for (int64_t j0 = o0; j0 < o1; j0 += NB) {
      const int nb = (int)std::min<int64_t>(NB, o1 - j0);
      const int64_t ncols = cols(j0 + nb);
      { trsm_left_diag_kernel<<<(unsigned)cdiv(ncols, NB), 32 * kGroup, 0, st>>>(Lkk, k, j0, nb, Bm, nrhs, ncols); count_launch(); }
      if (j0 + nb < o1) update(j0 + nb, o1, j0, j0 + nb);
    }
    if (o1 < k) update(o1, k, o0, o1);
  }
}

__global__ void transpose_square_kernel(const double* __restrict__ A, int64_t k, double* __restrict__ At) {
  __shared__ double tile[32][33];
  const int64_t bx = blockIdx.x * 32, by = blockIdx.y * 32;
  for (int yy = threadIdx.y; yy < 32; yy += 8) {
    const int64_t r = by + yy, c = bx + threadIdx.x;
    tile[yy][threadIdx.x] = (r < k && c < k) ? A[r * k + c] : 0.0;
  }
  __syncthreads();
  for (int yy = threadIdx.y; yy < 32; yy += 8) {
    const int64_t r = bx + yy, c = by + threadIdx.x;
    if (r < k && c < k) At[r * k + c] = tile[threadIdx.x][yy];
  }
}

__global__ void set_identity_kernel(double* A, int64_t k) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e < k * k) A[e] = (e / k == e % k) ? 1.0 : 0.0;
}

void transpose_square(const double* A, int64_t k, double* At, cudaStream_t st) {
  dim3 grid((unsigned)cdiv(k, 32), (unsigned)cdiv(k, 32));
  { transpose_square_kernel<<<grid, dim3(32, 8), 0, st>>>(A, k, At); count_launch(); }
}

// A[c][r] = A[r][c] for r > c (copy the lower triangle onto the upper one)
__global__ void mirror_lower_kernel(double* A, int64_t k) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= k * k) return;
  const int64_t r = e / k, c = e % k;
  if (r > c) A[c * k + r] = A[e];
}

void mirror_lower(double* A, int64_t k, cudaStream_t st) {
  { mirror_lower_kernel<<<(unsigned)cdiv(k * k, 256), 256, 0, st>>>(A, k); count_launch(); }
}

void set_identity(double* A, int64_t k, cudaStream_t st) {
  { set_identity_kernel<<<(unsigned)cdiv(k * k, 256), 256, 0, st>>>(A, k); count_launch(); }
}

void add_diag(double* A, int64_t lda, int64_t k, double eps, cudaStream_t st) {
  { add_diag_kernel<<<(unsigned)cdiv(k, 256), 256, 0, st>>>(A, lda, k, eps); count_launch(); }
}

}  // namespace gdml
