// complex64 FFT passes for any two-stage plan: lengths and radices are run-time values.
//
// The specialised kernels of fft_local.cu exist for a few boxes; for every other box of lengths up
// to 256 these run: batches of one-dimensional transforms of 32 lines per CTA (lane = line, the
// CTA's warps split a stage's butterflies, a switch on the radix around the stage), z, y, x, y, z.
// The rows between the z- and y-lines lie in the half-box plane at their own y, so no pass needs a
// buffer of its own.  The block-wide stages that ran here before index every element with a
// division by the line length and keep a whole row set per CTA.  8-step PAW filter of 37 bands on
// 45 x 50 x 54, per step: x-lines 71 -> 18 us, pass 1 37 -> 23 us, pass 3 45 -> 25 us, the filter
// 1.87 -> 1.18 ms.  24^3 keeps its line-group planes (32 bands, 6 steps: 0.39 ms, 0.48 ms here).
#include <cuda_bf16.h>

#include <algorithm>

#include "fft_lines.cuh"
#include "fft_radix.cuh"

namespace pw {
namespace fl {

typedef float2 C;
constexpr int kWarps = 4, kThreads = 32 * kWarps;
constexpr int PT = 33;  // pitch of an element's 32 lines: lane-wise and line-wise accesses are conflict-free

struct Dim {
  int n, r1, r2;
  const C* tw;  // [j][m - 1], j < r2, 1 <= m < r1
};

#define FL_SWITCH(R, F)    \
  switch (R) {             \
    case 16: F(16); break; \
    case 15: F(15); break; \
    case 12: F(12); break; \
    case 10: F(10); break; \
    case 9: F(9); break;   \
    case 8: F(8); break;   \
    case 6: F(6); break;   \
    case 5: F(5); break;   \
    case 4: F(4); break;   \
    case 3: F(3); break;   \
    default: F(2); break;  \
  }

// inverse stage 1: elements J + r2 a (zero where !valid) -> DFT, twiddle, in place
template <int R, typename V> __device__ __forceinline__ void inv1(C* col, int J, const Dim& d, V valid) {
  C x[R];
#pragma unroll
  for (int a = 0; a < R; ++a) {
    const int e = J + d.r2 * a;
    x[a] = valid(e) ? col[e * PT] : make_float2(0.f, 0.f);
  }
  dftR<C, +1, R>(x);
  if (J) {
    const C* w = d.tw + J * (R - 1);
#pragma unroll
    for (int m = 1; m < R; ++m) x[m] = cmul(x[m], cconj(w[m - 1]));
  }
#pragma unroll
  for (int m = 0; m < R; ++m) col[(J + d.r2 * m) * PT] = x[m];
}
// block blk of R adjacent elements: DFT in place
template <int S, int R> __device__ __forceinline__ void block_dft(C* col, int blk) {
  C y[R];
  C* c = col + blk * R * PT;
#pragma unroll
  for (int m = 0; m < R; ++m) y[m] = c[m * PT];
  dftR<C, S, R>(y);
#pragma unroll
  for (int m = 0; m < R; ++m) c[m * PT] = y[m];
}
// elements J + r2 m times the twiddles, forward DFT
template <int R> __device__ __forceinline__ void fwd2(const C* col, int J, const Dim& d, C (&x)[R]) {
#pragma unroll
  for (int m = 0; m < R; ++m) x[m] = col[(J + d.r2 * m) * PT];
  if (J) {
    const C* w = d.tw + J * (R - 1);
#pragma unroll
    for (int m = 1; m < R; ++m) x[m] = cmul(x[m], w[m - 1]);
  }
  dftR<C, -1, R>(x);
}

__device__ __forceinline__ int posmod(int a, int n) {
  const int r = a % n;
  return r < 0 ? r + n : r;
}
__device__ __forceinline__ int plane_of(const SphereDev& sp, int r) {
  int lo = 0, hi = sp.nplane;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (sp.plane_row0[mid] <= r) lo = mid;
    else hi = mid;
  }
  return lo;
}

// ---- z: 32 sphere rows per CTA, rows read and written by warps along z ---------------------------
__global__ void __launch_bounds__(kThreads) k_fl_zinv(const C* __restrict__ psi, int64_t ldpsi, C* __restrict__ hb,
                                                      int64_t hb_bs, SphereDev sp, Dim d, int n2) {
  extern __shared__ __align__(16) unsigned char smem[];
  C* buf = reinterpret_cast<C*>(smem);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int row0 = blockIdx.x * 32, n = d.n;
  const C* src = psi + (int64_t)blockIdx.y * ldpsi;
#pragma unroll 4
  for (int rr = w; rr < 32; rr += kWarps) {
    const int r = row0 + rr;
    if (r < sp.nrow) {
      const int g0 = sp.row_g0[r], cnt = sp.row_cnt[r], l0 = posmod(sp.row_l0[r], n);
      for (int i = lane; i < cnt; i += 32) {
        const int e = l0 + i;
        buf[(e >= n ? e - n : e) * PT + rr] = src[g0 + i];
      }
    }
  }
  C* col = buf + lane;
  int cnt = 0, l0 = 0;
  if (row0 + lane < sp.nrow) {
    cnt = sp.row_cnt[row0 + lane];
    l0 = posmod(sp.row_l0[row0 + lane], n);
  }
  __syncthreads();
#define FL_F(R)                                              \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) \
      inv1<R>(col, J, d, [&](int e) { return (e < l0 ? e - l0 + n : e - l0) < cnt; })
  FL_SWITCH(d.r1, FL_F)
#undef FL_F
  __syncthreads();
#define FL_F(R) _Pragma("unroll 1") for (int blk = w; blk < d.r1; blk += kWarps) block_dft<+1, R>(col, blk)
  FL_SWITCH(d.r2, FL_F)
#undef FL_F
  __syncthreads();
  for (int rr = w; rr < 32; rr += kWarps) {
    const int r = row0 + rr;
    if (r >= sp.nrow) break;
    C* dst = hb + (int64_t)blockIdx.y * hb_bs + ((int64_t)plane_of(sp, r) * n2 + posmod(sp.row_k[r], n2)) * n;
    for (int z = lane; z < n; z += 32) dst[z] = buf[z * PT + rr];
  }
}

// REC: 0 the kinetic term, 1 the recurrence, 2 the recurrence without P Z
template <int REC>
__global__ void __launch_bounds__(kThreads) k_fl_zfwd(const C* __restrict__ hb, int64_t hb_bs, SphereDev sp, Dim d,
                                                      int n2, const float* __restrict__ kin,
                                                      const C* __restrict__ psi, int64_t ldpsi, C* __restrict__ out,
                                                      int64_t ldout, Pass3Rec rec) {
  extern __shared__ __align__(16) unsigned char smem[];
  C* buf = reinterpret_cast<C*>(smem);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int row0 = blockIdx.x * 32, n = d.n;
#pragma unroll 4
  for (int rr = w; rr < 32; rr += kWarps) {
    const int r = row0 + rr;
    if (r < sp.nrow) {
      const C* src = hb + (int64_t)blockIdx.y * hb_bs + ((int64_t)plane_of(sp, r) * n2 + posmod(sp.row_k[r], n2)) * n;
      for (int z = lane; z < n; z += 32) buf[z * PT + rr] = src[z];
    } else {
      for (int z = lane; z < n; z += 32) buf[z * PT + rr] = make_float2(0.f, 0.f);
    }
  }
  C* col = buf + lane;
  __syncthreads();
#define FL_F(R) _Pragma("unroll 1") for (int blk = w; blk < d.r1; blk += kWarps) block_dft<-1, R>(col, blk)
  FL_SWITCH(d.r2, FL_F)
#undef FL_F
  __syncthreads();
#define FL_F(R)                                                                                    \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) {                                     \
    C x[R];                                                                                        \
    fwd2<R>(col, J, d, x);                                                                         \
    _Pragma("unroll") for (int a = 0; a < R; ++a) col[(J + d.r2 * a) * PT] = x[a];                 \
  }
  FL_SWITCH(d.r1, FL_F)
#undef FL_F
  __syncthreads();
  const int b = blockIdx.y;
  const C* yv = psi + (int64_t)b * ldpsi;
  C* o = out + (int64_t)b * ldout;
  float ra = 0, rs = 0;  // recurrence alpha and shift
  if constexpr (REC) {
    ra = rec.alpha;
    rs = rec.shift;
    if (rec.dev_ce) {
      rs = (float)rec.dev_ce[0];
      ra = (float)((rec.first ? 1.0 : 2.0) / rec.dev_ce[1]);
    }
  }
  for (int rr = w; rr < 32; rr += kWarps) {
    const int r = row0 + rr;
    if (r >= sp.nrow) break;
    const int g0 = sp.row_g0[r], cnt = sp.row_cnt[r], l0 = posmod(sp.row_l0[r], n);
    for (int i = lane; i < cnt; i += 32) {
      const int e = l0 + i, gg = g0 + i;
      const C v = buf[(e >= n ? e - n : e) * PT + rr];
      const C yy = yv[gg];
      const float k = kin[gg];
      if constexpr (!REC) {
        o[gg] = make_float2(k * yy.x + v.x, k * yy.y + v.y);
      } else {
        const C pz = REC == 1 ? rec.pz[(int64_t)b * rec.ldpz + gg] : make_float2(0.f, 0.f);
        C t = make_float2(ra * (k * yy.x + v.x + pz.x - rs * yy.x), ra * (k * yy.y + v.y + pz.y - rs * yy.y));
        if (rec.ykm1) {
          const C ym = rec.ykm1[(int64_t)b * rec.ldykm1 + gg];
          t.x -= rec.beta * ym.x;
          t.y -= rec.beta * ym.y;
        }
        o[gg] = t;
        if (rec.split) {
          __nv_bfloat16* sb = (__nv_bfloat16*)rec.split + (int64_t)b * rec.split_ld + 2 * (int64_t)gg;
          for (int pc = 0; pc < rec.pieces; ++pc) {
            const __nv_bfloat162 two = __floats2bfloat162_rn(t.x, t.y);
            *reinterpret_cast<__nv_bfloat162*>(sb + (int64_t)pc * rec.split_piece_stride) = two;
            t.x -= __bfloat162float(two.x);
            t.y -= __bfloat162float(two.y);
          }
        }
      }
    }
  }
}

// ---- y: 32 columns of one plane per CTA, in place ---------------------------------------------
__global__ void __launch_bounds__(kThreads) k_fl_yinv(C* __restrict__ hb, int64_t hb_bs, SphereDev sp, Dim d, int n3,
                                                      int nc) {
  extern __shared__ __align__(16) unsigned char smem[];
  C* buf = reinterpret_cast<C*>(smem);
  int* ymap = reinterpret_cast<int*>(buf + d.n * PT);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int p = blockIdx.x / nc, c = (blockIdx.x % nc) * 32 + lane, n = d.n;
  const bool live = c < n3;
  const int r0 = sp.plane_row0[p], nr = sp.plane_row0[p + 1] - r0;
  for (int i = threadIdx.x; i < n; i += kThreads) ymap[i] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < nr; i += kThreads) ymap[posmod(sp.row_k[r0 + i], n)] = 1;
  C* pl = hb + (int64_t)blockIdx.y * hb_bs + (int64_t)p * n * n3 + (live ? c : 0);
#pragma unroll 4
  for (int i = w; i < nr; i += kWarps) {
    const int k = posmod(sp.row_k[r0 + i], n);
    buf[k * PT + lane] = live ? pl[(int64_t)k * n3] : make_float2(0.f, 0.f);
  }
  C* col = buf + lane;
  __syncthreads();
#define FL_F(R)                                              \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) \
      inv1<R>(col, J, d, [&](int e) { return ymap[e] != 0; })
  FL_SWITCH(d.r1, FL_F)
#undef FL_F
  __syncthreads();
#define FL_F(R)                                                                            \
  _Pragma("unroll 1") for (int blk = w; blk < d.r1; blk += kWarps) {                       \
    C y[R];                                                                                \
    _Pragma("unroll") for (int m = 0; m < R; ++m) y[m] = col[(blk * R + m) * PT];          \
    dftR<C, +1, R>(y);                                                                     \
    if (live) {                                                                            \
      _Pragma("unroll") for (int m = 0; m < R; ++m) pl[(int64_t)(blk * R + m) * n3] = y[m]; \
    }                                                                                      \
  }
  FL_SWITCH(d.r2, FL_F)
#undef FL_F
}

__global__ void __launch_bounds__(kThreads) k_fl_yfwd(C* __restrict__ hb, int64_t hb_bs, SphereDev sp, Dim d, int n3,
                                                      int nc) {
  extern __shared__ __align__(16) unsigned char smem[];
  C* buf = reinterpret_cast<C*>(smem);
  int* ymap = reinterpret_cast<int*>(buf + d.n * PT);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int p = blockIdx.x / nc, c = (blockIdx.x % nc) * 32 + lane, n = d.n;
  const bool live = c < n3;
  const int r0 = sp.plane_row0[p], nr = sp.plane_row0[p + 1] - r0;
  for (int i = threadIdx.x; i < n; i += kThreads) ymap[i] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < nr; i += kThreads) ymap[posmod(sp.row_k[r0 + i], n)] = 1;
  C* pl = hb + (int64_t)blockIdx.y * hb_bs + (int64_t)p * n * n3 + (live ? c : 0);
  C* col = buf + lane;
  // first stage straight from the plane: the block's elements are rows of 32 columns
#define FL_F(R)                                                                                          \
  _Pragma("unroll 1") for (int blk = w; blk < d.r1; blk += kWarps) {                                     \
    C y[R];                                                                                              \
    _Pragma("unroll") for (int m = 0; m < R; ++m)                                                        \
        y[m] = live ? pl[(int64_t)(blk * R + m) * n3] : make_float2(0.f, 0.f);                           \
    dftR<C, -1, R>(y);                                                                                   \
    _Pragma("unroll") for (int m = 0; m < R; ++m) col[(blk * R + m) * PT] = y[m];                        \
  }
  FL_SWITCH(d.r2, FL_F)
#undef FL_F
  __syncthreads();
#define FL_F(R)                                                              \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) {               \
    C x[R];                                                                  \
    fwd2<R>(col, J, d, x);                                                   \
    _Pragma("unroll") for (int a = 0; a < R; ++a) {                          \
      const int e = J + d.r2 * a;                                            \
      if (live && ymap[e]) pl[(int64_t)e * n3] = x[a];                       \
    }                                                                        \
  }
  FL_SWITCH(d.r1, FL_F)
#undef FL_F
}

// ---- x: 32 (y,z) lines of one band per CTA --------------------------------------------------------
__global__ void __launch_bounds__(kThreads) k_fl_x(C* __restrict__ hb, int64_t hb_bs,
                                                   const float* __restrict__ vperm, int np, int nyz, Dim d) {
  extern __shared__ __align__(16) unsigned char smem[];
  C* col = reinterpret_cast<C*>(smem) + (threadIdx.x & 31);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int yz = blockIdx.x * 32 + lane;
  const bool live = yz < nyz;
  C* pl = hb + (int64_t)blockIdx.y * hb_bs + (live ? yz : 0);
  const float* vb = vperm + (live ? yz : 0);
  // first stage straight from the planes (plane p at x-frequency p: a shift of the line's
  // frequencies multiplies by a phase that the two transforms cancel)
#define FL_F(R)                                                                                     \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) {                                      \
    C x[R];                                                                                         \
    _Pragma("unroll") for (int a = 0; a < R; ++a) {                                                 \
      const int e = J + d.r2 * a;                                                                   \
      x[a] = (live && e < np) ? pl[(int64_t)e * nyz] : make_float2(0.f, 0.f);                       \
    }                                                                                               \
    dftR<C, +1, R>(x);                                                                              \
    if (J) {                                                                                        \
      const C* tw = d.tw + J * (R - 1);                                                             \
      _Pragma("unroll") for (int m = 1; m < R; ++m) x[m] = cmul(x[m], cconj(tw[m - 1]));            \
    }                                                                                               \
    _Pragma("unroll") for (int m = 0; m < R; ++m) col[(J + d.r2 * m) * PT] = x[m];                  \
  }
  FL_SWITCH(d.r1, FL_F)
#undef FL_F
  __syncthreads();
#define FL_F(R)                                                                       \
  _Pragma("unroll 1") for (int blk = w; blk < d.r1; blk += kWarps) {                  \
    C y[R];                                                                           \
    float v[R];                                                                       \
    C* c = col + blk * R * PT;                                                        \
    const float* vl = vb + (int64_t)blk * R * nyz;                                    \
    _Pragma("unroll") for (int m = 0; m < R; ++m) v[m] = vl[(int64_t)m * nyz];        \
    _Pragma("unroll") for (int m = 0; m < R; ++m) y[m] = c[m * PT];                   \
    dftR<C, +1, R>(y);                                                                \
    _Pragma("unroll") for (int m = 0; m < R; ++m) y[m] = cscale(y[m], v[m]);          \
    dftR<C, -1, R>(y);                                                                \
    _Pragma("unroll") for (int m = 0; m < R; ++m) c[m * PT] = y[m];                   \
  }
  FL_SWITCH(d.r2, FL_F)
#undef FL_F
  __syncthreads();
#define FL_F(R)                                                      \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) {       \
    C x[R];                                                          \
    fwd2<R>(col, J, d, x);                                           \
    _Pragma("unroll") for (int a = 0; a < R; ++a) {                  \
      const int e = J + d.r2 * a;                                    \
      if (live && e < np) pl[(int64_t)e * nyz] = x[a];               \
    }                                                                \
  }
  FL_SWITCH(d.r1, FL_F)
#undef FL_F
}

// ---- host -------------------------------------------------------------------------------
bool covers(const FftPlan& plan) {
  for (int i = 0; i < 3; ++i)
    if (plan.d[i].nst != 2 || plan.n[i] > 256) return false;
  return true;
}
static Dim dim_of(const FftPlan& plan, const C* tw, int i) {
  const FftDim& f = plan.d[i];
  return {f.n, f.radix[0], f.radix[1], tw + f.tw_off[0]};
}
static size_t line_bytes(const Dim& d) { return sizeof(C) * PT * d.n; }

cudaError_t inverse_planes(const FftPlan& plan, const C* tw, const SphereDev& sp, const C* psi, int64_t ldpsi, C* hb,
                           int64_t hb_bs, int nb, cudaStream_t st) {
  const Dim dy = dim_of(plan, tw, 1), dz = dim_of(plan, tw, 2);
  const int nc = (dz.n + 31) / 32;
  const size_t smz = line_bytes(dz), smy = line_bytes(dy) + sizeof(int) * dy.n;
  cudaError_t e;
  if ((e = smem_limit(k_fl_zinv, smz)) || (e = smem_limit(k_fl_yinv, smy))) return e;
  k_fl_zinv<<<dim3((sp.nrow + 31) / 32, nb), kThreads, smz, st>>>(psi, ldpsi, hb, hb_bs, sp, dz, dy.n); count_launch();
  k_fl_yinv<<<dim3(sp.nplane * nc, nb), kThreads, smy, st>>>(hb, hb_bs, sp, dy, dz.n, nc); count_launch();
  return cudaGetLastError();
}

cudaError_t xlines(const FftPlan& plan, const C* tw, const SphereDev& sp, const float* vperm, C* hb, int64_t hb_bs,
                   int nb, cudaStream_t st) {
  const Dim dx = dim_of(plan, tw, 0);
  const int nyz = plan.n[1] * plan.n[2];
  const size_t sm = line_bytes(dx);
  cudaError_t e;
  if ((e = smem_limit(k_fl_x, sm))) return e;
  k_fl_x<<<dim3((nyz + 31) / 32, nb), kThreads, sm, st>>>(hb, hb_bs, vperm, sp.nplane, nyz, dx); count_launch();
  return cudaGetLastError();
}

cudaError_t forward_planes(const FftPlan& plan, const C* tw, const SphereDev& sp, const float* kin, C* hb,
                           int64_t hb_bs, const C* psi, int64_t ldpsi, C* out, int64_t ldout, int nb, cudaStream_t st,
                           const Pass3Rec* rec) {
  const Dim dy = dim_of(plan, tw, 1), dz = dim_of(plan, tw, 2);
  const int nc = (dz.n + 31) / 32;
  const size_t smz = line_bytes(dz), smy = line_bytes(dy) + sizeof(int) * dy.n;
  cudaError_t e;
  if ((e = smem_limit(k_fl_yfwd, smy)) || (e = smem_limit(k_fl_zfwd<0>, smz)) || (e = smem_limit(k_fl_zfwd<1>, smz)) ||
      (e = smem_limit(k_fl_zfwd<2>, smz)))
    return e;
  k_fl_yfwd<<<dim3(sp.nplane * nc, nb), kThreads, smy, st>>>(hb, hb_bs, sp, dy, dz.n, nc); count_launch();
  const dim3 g((sp.nrow + 31) / 32, nb);
  if (rec && !rec->pz)
    k_fl_zfwd<2><<<g, kThreads, smz, st>>>(hb, hb_bs, sp, dz, dy.n, kin, psi, ldpsi, out, ldout, *rec);
  else if (rec)
    k_fl_zfwd<1><<<g, kThreads, smz, st>>>(hb, hb_bs, sp, dz, dy.n, kin, psi, ldpsi, out, ldout, *rec);
  else
    k_fl_zfwd<0><<<g, kThreads, smz, st>>>(hb, hb_bs, sp, dz, dy.n, kin, psi, ldpsi, out, ldout, Pass3Rec{});
  count_launch();
  return cudaGetLastError();
}

}  // namespace fl
}  // namespace pw
