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
// with steps of 64 the diagonal block took 105 us and a panel 150-190 us.  A warp of 32 rows per CTA
// spreads a panel over all SMs.  Two factorisations and two triangular inverses at k = 1500: 62 ms
// with one level of 64, 31 ms so.
constexpr int NB = 32;
constexpr int NO = 128;

// Unblocked Cholesky of the nb x nb diagonal block at (j0, j0), in place (lower): one warp, lane r
// holds row r.
__global__ void __launch_bounds__(32) potrf_diag_kernel(double* __restrict__ A, int64_t lda, int64_t j0, int nb,
                                                        int* __restrict__ status) {
  if (*status) return;
  const int r = threadIdx.x;
  double* row = A + (j0 + r) * lda + j0;
  double a[NB];
#pragma unroll
  for (int c = 0; c < NB; ++c) a[c] = (r < nb && c <= r) ? row[c] : (c == r ? 1.0 : 0.0);
  int bad = 0;
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    const double d = __shfl_sync(0xffffffffu, a[c], c);
    if (!(d > 0.0) || !isfinite(d)) {  // (warp-uniform)
      bad = c + 1;
      break;
    }
    const double l = sqrt(d), inv = 1.0 / l;
    a[c] = r == c ? l : a[c] * inv;
#pragma unroll
    for (int cc = c + 1; cc < NB; ++cc) a[cc] = fma(-a[c], __shfl_sync(0xffffffffu, a[c], cc), a[cc]);
  }
  if (bad) {
    if (r == 0) *status = (int)(j0 + bad);
    return;
  }
  if (r < nb)
#pragma unroll
    for (int c = 0; c < NB; ++c)
      if (c < nb) row[c] = c <= r ? a[c] : 0.0;
}

// Rows r in [r0, rend): solve x L_jj^T = A[r, j0:j0+nb]  (one thread per row, one warp per CTA).
__global__ void __launch_bounds__(32) trsm_right_kernel(double* __restrict__ A, int64_t lda, int64_t j0, int nb,
                                                        int64_t r0, int64_t rend, const int* __restrict__ status) {
  __shared__ double L[NB][NB + 1];
  __shared__ double rows[NB][NB + 1];
  if (*status) return;
  const int t = threadIdx.x;
  const int64_t base = r0 + blockIdx.x * (int64_t)NB;
  for (int r = 0; r < NB; ++r) {
    const bool in = r < nb && t < nb;
    L[r][t] = in ? A[(j0 + r) * lda + j0 + t] : (r == t ? 1.0 : 0.0);
    rows[r][t] = base + r < rend && t < nb ? A[(base + r) * lda + j0 + t] : 0.0;
  }
  __syncwarp();
  const double inv = 1.0 / L[t][t];
  double x[NB];
#pragma unroll
  for (int c = 0; c < NB; ++c) x[c] = rows[t][c];
#pragma unroll
  for (int c = 0; c < NB; ++c) {  // column by column: the updates of the later ones are independent
    x[c] *= __shfl_sync(0xffffffffu, inv, c);
#pragma unroll
    for (int cc = c + 1; cc < NB; ++cc) x[cc] = fma(-x[c], L[cc][c], x[cc]);
  }
#pragma unroll
  for (int c = 0; c < NB; ++c) rows[t][c] = x[c];
  __syncwarp();
  for (int r = 0; r < NB; ++r)
    if (base + r < rend && t < nb) A[(base + r) * lda + j0 + t] = rows[r][t];
}

// Left forward substitution on a block of rows of B (k x nrhs, row-major, ld):
// B[j0:j0+nb, col] <- L_jj^-1 B[j0:j0+nb, col]; one thread per column, one warp per CTA.
__global__ void __launch_bounds__(32) trsm_left_diag_kernel(const double* __restrict__ Lkk, int64_t ldl, int64_t j0,
                                                            int nb, double* __restrict__ Bm, int64_t ldb,
                                                            int64_t nrhs) {
  __shared__ double L[NB][NB + 1];
  const int t = threadIdx.x;
  for (int r = 0; r < NB; ++r)
    L[r][t] = r < nb && t < nb ? Lkk[(j0 + r) * ldl + j0 + t] : (r == t ? 1.0 : 0.0);
  __syncwarp();
  const double inv = 1.0 / L[t][t];
  const int64_t col = blockIdx.x * (int64_t)NB + t;
  const bool in = col < nrhs;
  double x[NB];
#pragma unroll
  for (int r = 0; r < NB; ++r) x[r] = in && r < nb ? Bm[(j0 + r) * ldb + col] : 0.0;
#pragma unroll
  for (int r = 0; r < NB; ++r) {
    x[r] *= __shfl_sync(0xffffffffu, inv, r);
#pragma unroll
    for (int rr = r + 1; rr < NB; ++rr) x[rr] = fma(-L[rr][r], x[r], x[rr]);
  }
  if (in)
#pragma unroll
    for (int r = 0; r < NB; ++r)
      if (r < nb) Bm[(j0 + r) * ldb + col] = x[r];
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
      { potrf_diag_kernel<<<1, 32, 0, st>>>(A, k, j0, nb, status); count_launch(); }
      const int64_t r0 = j0 + nb;
      if (r0 >= k) break;
      { trsm_right_kernel<<<(unsigned)cdiv(k - r0, NB), NB, 0, st>>>(A, k, j0, nb, r0, k, status); count_launch(); }
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
      { trsm_left_diag_kernel<<<(unsigned)cdiv(ncols, NB), NB, 0, st>>>(Lkk, k, j0, nb, Bm, nrhs, ncols); count_launch(); }
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
