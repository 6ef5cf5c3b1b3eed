// Factorisations and Lanczos steps of the FP64 solves (pw_chebfi_solve, pw_batch_chebfi_solve), in one
// fixed order of operations.
//
// The phase of a Ritz vector is a product of the phases of all the elements that the Jacobi rounds
// met, the last of them at rounding level: another order of sums anywhere before it, however exact,
// turns the vectors by phases of order one.  A program that keeps vectors of FP64 solves (or compares
// them) sees the same ones only with the same operations, so these calls run the FP64 transforms, these
// kernels and the plain Jacobi (pw_ctx::keep64), and a k-point has the same vectors alone and in a
// batch.  Every other call returns the faster kernels' results:
// the densities, energies, residuals and gradients that are made from Ritz vectors do not depend on
// the phases.  The order covers what an FP64 solve does itself: the Woodbury matrices of Q are made with
// the context, by the faster factorisations, and blocks of 2 to 4 bands take matrix-vector products whose
// sums have four parts.
#include <math.h>

#include <algorithm>

#include "la.cuh"
#include "pw_internal.cuh"

namespace pw {

// ---- blocked Cholesky A = L L^dagger (lower, in place; strict upper part zeroed) ---
constexpr int NB = 32;

static __global__ void k_keep_chol_diag(double2* A, int64_t lda, int k0, int kb, int* flag) {
  __shared__ double2 S[NB][NB + 1];
  const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 32
  if (tx < kb && ty < kb) S[ty][tx] = A[(k0 + ty) + (int64_t)(k0 + tx) * lda];  // S[row][col]
  __syncthreads();
  for (int j = 0; j < kb; ++j) {
    if (tx == 0 && ty == 0) {
      double d = S[j][j].x;
      if (!(d > 0.0) || !isfinite(d)) { atomicExch(flag, 1); d = 1.0; }
      S[j][j] = make_double2(sqrt(d), 0.0);
    }
    __syncthreads();
    const double dj = S[j][j].x;
    if (tx == 0 && ty > j && ty < kb) S[ty][j] = cscale(S[ty][j], 1.0 / dj);
    __syncthreads();
    // trailing: S[i][k] -= S[i][j] conj(S[k][j]) for j < k <= i
    if (ty > j && ty < kb && tx > j && tx <= ty) S[ty][tx] = csub(S[ty][tx], cmul(S[ty][j], cconj(S[tx][j])));
    __syncthreads();
  }
  if (tx < kb && ty < kb) {
    const double2 v = (tx <= ty) ? S[ty][tx] : make_double2(0.0, 0.0);
    A[(k0 + ty) + (int64_t)(k0 + tx) * lda] = v;
  }
}

// rows i >= k0+kb: L21[i,:] = A21[i,:] L11^{-dagger}
static __global__ void k_keep_chol_panel(double2* A, int64_t lda, int n, int k0, int kb) {
  __shared__ double2 Ls[NB][NB + 1];
  const int t = threadIdx.x;
  for (int e = t; e < kb * kb; e += blockDim.x) {
    const int r = e % kb, c = e / kb;
    Ls[r][c] = A[(k0 + r) + (int64_t)(k0 + c) * lda];
  }
  __syncthreads();
  const int i = k0 + kb + blockIdx.x * blockDim.x + t;
  if (i >= n) return;
  double2 x[NB];
  for (int j = 0; j < kb; ++j) {
    double2 s = A[i + (int64_t)(k0 + j) * lda];
    for (int tt = 0; tt < j; ++tt) s = csub(s, cmul(x[tt], cconj(Ls[j][tt])));
    x[j] = cscale(s, 1.0 / Ls[j][j].x);
  }
  for (int j = 0; j < kb; ++j) A[i + (int64_t)(k0 + j) * lda] = x[j];
}

// trailing update of the lower triangle: A[i][j] -= sum_t L[i][t] conj(L[j][t])
static __global__ void k_keep_chol_update(double2* A, int64_t lda, int n, int k0, int kb) {
  const int bi = blockIdx.x, bj = blockIdx.y;
  if (bj > bi) return;
  __shared__ double2 Li[32][NB + 1], Lj[32][NB + 1];
  const int s0 = k0 + kb;
  const int i0 = s0 + bi * 32, j0 = s0 + bj * 32;
  const int t = threadIdx.x;  // 256
  for (int e = t; e < 32 * kb; e += 256) {
    const int r = e % 32, c = e / 32;
    Li[r][c] = (i0 + r < n) ? A[(i0 + r) + (int64_t)(k0 + c) * lda] : make_double2(0, 0);
    Lj[r][c] = (j0 + r < n) ? A[(j0 + r) + (int64_t)(k0 + c) * lda] : make_double2(0, 0);
  }
  __syncthreads();
  for (int e = t; e < 32 * 32; e += 256) {
    const int r = e % 32, c = e / 32;
    const int i = i0 + r, j = j0 + c;
    if (i >= n || j >= n || j > i) continue;
    double2 s = make_double2(0, 0);
    for (int tt = 0; tt < kb; ++tt) {
      const double2 a = Li[r][tt], b = Lj[c][tt];
      s.x += a.x * b.x + a.y * b.y;
      s.y += a.y * b.x - a.x * b.y;
    }
    A[i + (int64_t)j * lda] = csub(A[i + (int64_t)j * lda], s);
  }
}

static __global__ void k_keep_zero_upper(double2* A, int64_t lda, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i < n && j < n && j > i) A[i + (int64_t)j * lda] = make_double2(0, 0);
}

cudaError_t la_cholesky_keep(double2* A, int64_t lda, int n, int* flag, cudaStream_t st) {
  for (int k0 = 0; k0 < n; k0 += NB) {
    const int kb = min(NB, n - k0);
    k_keep_chol_diag<<<1, dim3(32, 32), 0, st>>>(A, lda, k0, kb, flag); count_launch();
    const int rest = n - k0 - kb;
    if (rest > 0) {
      k_keep_chol_panel<<<(rest + 127) / 128, 128, 0, st>>>(A, lda, n, k0, kb); count_launch();
      const int nt = (rest + 31) / 32;
      k_keep_chol_update<<<dim3(nt, nt), 256, 0, st>>>(A, lda, n, k0, kb); count_launch();
    }
  }
  // zero the strict upper triangle
  dim3 zb(16, 16), zg((n + 15) / 16, (n + 15) / 16);
  k_keep_zero_upper<<<zg, zb, 0, st>>>(A, lda, n); count_launch();
  return cudaGetLastError();
}

// ---- triangular inverse X = L^{-1} (lower) -------------------------------------------
static __global__ void k_keep_transpose(const double2* A, int64_t lda, int n, double2* At) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i < n && j < n) At[j + (int64_t)i * n] = A[i + (int64_t)j * lda];
}

// one warp per column j of X; Lt holds L row-major (Lt[t + i n] = L[i][t])
static __global__ void k_keep_trinv(const double2* __restrict__ Lt, int n, double2* __restrict__ X, int64_t ldx) {
  extern __shared__ double2 xs[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j = blockIdx.x * (blockDim.x >> 5) + warp;
  if (j >= n) return;
  double2* x = xs + (int64_t)warp * n;
  for (int i = lane; i < j; i += 32) X[i + (int64_t)j * ldx] = make_double2(0, 0);
  if (lane == 0) {
    const double d = Lt[j + (int64_t)j * n].x;
    x[j] = make_double2(1.0 / d, 0.0);
    X[j + (int64_t)j * ldx] = x[j];
  }
  __syncwarp();
  for (int i = j + 1; i < n; ++i) {
    const double2* row = Lt + (int64_t)i * n;
    double sr = 0, si = 0;
    for (int t = j + lane; t < i; t += 32) {
      const double2 a = row[t], b = x[t];
      sr += a.x * b.x - a.y * b.y;
      si += a.x * b.y + a.y * b.x;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sr += __shfl_down_sync(0xffffffffu, sr, o);
      si += __shfl_down_sync(0xffffffffu, si, o);
    }
    if (lane == 0) {
      const double d = row[i].x;
      x[i] = make_double2(-sr / d, -si / d);
      X[i + (int64_t)j * ldx] = x[i];
    }
    __syncwarp();
  }
}

cudaError_t la_trinv_lower_keep(const double2* L, int64_t lda, int n, double2* X, int64_t ldx, double2* tmp,
                           cudaStream_t st) {
  dim3 b(16, 16), g((n + 15) / 16, (n + 15) / 16);
  k_keep_transpose<<<g, b, 0, st>>>(L, lda, n, tmp); count_launch();
  const int wpb = 4;
  const size_t sm = sizeof(double2) * (size_t)n * wpb;
  cudaError_t e = smem_limit(k_keep_trinv, sm);
  if (e) return e;
  k_keep_trinv<<<(n + wpb - 1) / wpb, 32 * wpb, sm, st>>>(tmp, n, X, ldx); count_launch();
  return cudaGetLastError();
}

// ---- Lanczos helpers (one vector) ---------------------------------------------------
// ab: device array, alpha at ab[2k], beta at ab[2k+1]
static __global__ void k_keep_lz_dot(const double2* v, const double2* w, int n, double* alpha_out) {
  __shared__ double sh[1024];
  double s = 0;
  for (int g = threadIdx.x; g < n; g += blockDim.x) s += v[g].x * w[g].x + v[g].y * w[g].y;
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int k = blockDim.x / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) sh[threadIdx.x] += sh[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) *alpha_out = sh[0];
}

// w <- w - alpha v - beta vprev ; beta_out = ||w|| ; vprev <- v ; v <- w / beta_out
static __global__ void k_keep_lz_update(double2* w, double2* v, double2* vprev, int n, const double* alpha,
                            const double* beta_prev, double* beta_out) {
  __shared__ double sh[1024];
  const double a = *alpha, b = beta_prev ? *beta_prev : 0.0;
  double s = 0;
  for (int g = threadIdx.x; g < n; g += blockDim.x) {
    double2 x = w[g];
    const double2 vv = v[g], vp = vprev[g];
    x.x -= a * vv.x + b * vp.x;
    x.y -= a * vv.y + b * vp.y;
    w[g] = x;
    s += x.x * x.x + x.y * x.y;
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int k = blockDim.x / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) sh[threadIdx.x] += sh[threadIdx.x + k];
    __syncthreads();
  }
  const double nb = sqrt(sh[0]);
  const double inv = nb > 0 ? 1.0 / nb : 0.0;
  for (int g = threadIdx.x; g < n; g += blockDim.x) {
    vprev[g] = v[g];
    v[g] = cscale(w[g], inv);
  }
  if (threadIdx.x == 0) *beta_out = nb;
}

static __global__ void k_keep_lz_normalize(const double2* v0, double2* v, double2* vprev, int n) {
  __shared__ double sh[1024];
  double s = 0;
  for (int g = threadIdx.x; g < n; g += blockDim.x) s += v0[g].x * v0[g].x + v0[g].y * v0[g].y;
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int k = blockDim.x / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) sh[threadIdx.x] += sh[threadIdx.x + k];
    __syncthreads();
  }
  const double inv = 1.0 / sqrt(sh[0]);
  for (int g = threadIdx.x; g < n; g += blockDim.x) {
    v[g] = cscale(v0[g], inv);
    vprev[g] = make_double2(0, 0);
  }
}

// largest eigenvalue of the k x k symmetric tridiagonal (alpha, beta) by Sturm bisection;
// out[0] = theta_max + |beta_k|, out[1] = theta_max
static __global__ void k_keep_lz_bound(const double* ab, int k, double* out) {
  if (threadIdx.x != 0) return;
  double lo = INFINITY, hi = -INFINITY;
  for (int i = 0; i < k; ++i) {
    const double a = ab[2 * i];
    const double r = (i > 0 ? fabs(ab[2 * i - 1]) : 0.0) + (i < k - 1 ? fabs(ab[2 * i + 1]) : 0.0);
    lo = fmin(lo, a - r);
    hi = fmax(hi, a + r);
  }
  // count of eigenvalues < x
  for (int it = 0; it < 200; ++it) {
    const double x = 0.5 * (lo + hi);
    if (x == lo || x == hi) break;
    int cnt = 0;
    double d = 1.0;
    for (int i = 0; i < k; ++i) {
      const double b2 = (i > 0) ? ab[2 * i - 1] * ab[2 * i - 1] : 0.0;
      d = (ab[2 * i] - x) - (i > 0 ? b2 / d : 0.0);
      if (d == 0.0) d = -1e-300;
      if (d < 0) ++cnt;
    }
    if (cnt == k) hi = x; else lo = x;
  }
  out[1] = hi;
  out[0] = hi + fabs(ab[2 * k - 1]);
}

cudaError_t la_lanczos_keep(const double2* v0, int n, int steps, double2* v, double2* vprev, double2* w, double* ab,
                       double* bound, ApplyFn apply, void* ctx, cudaStream_t st) {
  k_keep_lz_normalize<<<1, 1024, 0, st>>>(v0, v, vprev, n); count_launch();
  for (int k = 0; k < steps; ++k) {
    int s = apply(ctx, v, w);
    if (s != PW_OK) return cudaErrorUnknown;
    k_keep_lz_dot<<<1, 1024, 0, st>>>(v, w, n, ab + 2 * k); count_launch();
    k_keep_lz_update<<<1, 1024, 0, st>>>(w, v, vprev, n, ab + 2 * k, k > 0 ? ab + 2 * k - 1 : nullptr, ab + 2 * k + 1); count_launch();
  }
  k_keep_lz_bound<<<1, 32, 0, st>>>(ab, steps, bound); count_launch();
  return cudaGetLastError();
}

}  // namespace pw
