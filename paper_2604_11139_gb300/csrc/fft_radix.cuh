// Butterflies of the complex64 and complex128 FFT passes: DFTs of the in-register radices.
#pragma once
#include "pw_internal.cuh"

namespace pw {

// ---- butterfly arithmetic ---------------------------------------------------------
// complex64 sums, differences and real scalings use the paired FP32 instructions of
// sm_100-class SMs (one add, multiply or fused multiply-add for both halves of a float2,
// each half rounded to nearest as the scalar instruction would); complex128 keeps the
// scalar forms.  The products by +-i swap the halves of an operand, which a paired
// instruction cannot do in place, so they stay two scalar instructions (measured on the
// 120^3 plane passes: 6% faster than paired with the swap; all-scalar butterflies are
// slower still).  Every form rounds each result identically.
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 bf_add(double2 a, double2 b) { return cadd(a, b); }
__device__ __forceinline__ float2 bf_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 bf_sub(double2 a, double2 b) { return csub(a, b); }
__device__ __forceinline__ float2 bf_sub(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f, -1.f), a); }
__device__ __forceinline__ double2 bf_scale(double2 a, double s) { return cscale(a, s); }
__device__ __forceinline__ float2 bf_scale(float2 a, float s) { return __fmul2_rn(a, f2(s, s)); }
// a + s b
__device__ __forceinline__ double2 bf_axpy(double2 a, double s, double2 b) {
  return make_double2(fma(s, b.x, a.x), fma(s, b.y, a.y));
}
__device__ __forceinline__ float2 bf_axpy(float2 a, float s, float2 b) { return __ffma2_rn(b, f2(s, s), a); }
// a + (S i) s b  and  a - (S i) s b
template <int S> __device__ __forceinline__ double2 bf_add_muli(double2 a, double2 b, double s = 1.0) {
  return make_double2(fma(-S * s, b.y, a.x), fma(S * s, b.x, a.y));
}
template <int S> __device__ __forceinline__ float2 bf_add_muli(float2 a, float2 b, float s = 1.f) {
  return f2(__fmaf_rn(-S * s, b.y, a.x), __fmaf_rn(S * s, b.x, a.y));
}
template <int S> __device__ __forceinline__ double2 bf_sub_muli(double2 a, double2 b, double s = 1.0) {
  return make_double2(fma(S * s, b.y, a.x), fma(-S * s, b.x, a.y));
}
template <int S> __device__ __forceinline__ float2 bf_sub_muli(float2 a, float2 b, float s = 1.f) {
  return f2(__fmaf_rn(S * s, b.y, a.x), __fmaf_rn(-S * s, b.x, a.y));
}

// ---- small DFTs: y_m = sum_k x_k exp(S 2 pi i k m / R) -------------------------
template <typename C, int S> __device__ __forceinline__ void dft2(C& a, C& b) {
  C t = a; a = bf_add(t, b); b = bf_sub(t, b);
}
template <typename C, int S> __device__ __forceinline__ void dft4(C* x) {
  C s02 = bf_add(x[0], x[2]), d02 = bf_sub(x[0], x[2]);
  C s13 = bf_add(x[1], x[3]), d13 = bf_sub(x[1], x[3]);
  x[0] = bf_add(s02, s13); x[2] = bf_sub(s02, s13);
  x[1] = bf_add_muli<S>(d02, d13); x[3] = bf_sub_muli<S>(d02, d13);
}
template <typename C, int S> __device__ __forceinline__ void dft8(C* x) {
  using R = decltype(C{}.x);
  const R h = (R)0.70710678118654752440084436210485;  // cos(pi/4)
  C e[4] = {x[0], x[2], x[4], x[6]};
  C o[4] = {x[1], x[3], x[5], x[7]};
  dft4<C, S>(e); dft4<C, S>(o);
  // o[m] *= w8^m, w8 = exp(S i pi/4): w8 = h (1 + S i), w8^3 = h (-1 + S i)
  const C o1 = bf_scale(bf_add_muli<S>(o[1], o[1]), h);
  const C o3 = bf_scale(bf_sub_muli<S>(o[3], o[3]), -h);
  x[0] = bf_add(e[0], o[0]); x[4] = bf_sub(e[0], o[0]);
  x[1] = bf_add(e[1], o1); x[5] = bf_sub(e[1], o1);
  x[2] = bf_add_muli<S>(e[2], o[2]); x[6] = bf_sub_muli<S>(e[2], o[2]);
  x[3] = bf_add(e[3], o3); x[7] = bf_sub(e[3], o3);
}
template <typename C, int S> __device__ __forceinline__ void dft3(C* x) {
  using R = decltype(C{}.x);
  const R s3 = (R)0.86602540378443864676372317075294;  // sin(pi/3)
  C t = bf_add(x[1], x[2]);
  C d = bf_sub(x[1], x[2]);
  C m = bf_axpy(x[0], (R)-0.5, t);
  x[0] = bf_add(x[0], t);
  x[1] = bf_add_muli<S>(m, d, s3);
  x[2] = bf_sub_muli<S>(m, d, s3);
}
template <typename C, int S> __device__ __forceinline__ void dft5(C* x) {
  using R = decltype(C{}.x);
  const R c1 = (R)0.30901699437494742410229341718282;   // cos(2pi/5)
  const R c2 = (R)-0.80901699437494742410229341718282;  // cos(4pi/5)
  const R s1 = (R)0.95105651629515357211643933337938;   // sin(2pi/5)
  const R s2 = (R)0.58778525229247312916870595463907;   // sin(4pi/5)
  C t1 = bf_add(x[1], x[4]), t2 = bf_add(x[2], x[3]);
  C d1 = bf_sub(x[1], x[4]), d2 = bf_sub(x[2], x[3]);
  C a1 = bf_add(x[0], bf_axpy(bf_scale(t1, c1), c2, t2));
  C a2 = bf_add(x[0], bf_axpy(bf_scale(t1, c2), c1, t2));
  C u1 = bf_axpy(bf_scale(d1, s1), s2, d2);    // b1 = (S i) u1
  C u2 = bf_axpy(bf_scale(d1, s2), -s1, d2);   // b2 = (S i) u2
  x[0] = bf_add(x[0], bf_add(t1, t2));
  x[1] = bf_add_muli<S>(a1, u1); x[4] = bf_sub_muli<S>(a1, u1);
  x[2] = bf_add_muli<S>(a2, u2); x[3] = bf_sub_muli<S>(a2, u2);
}
// exp(-2 pi i m / R) for the composite in-register radices: cos and sin of the FP64 angle.
// Offsets: R=6: 0, 9: 6, 10: 15, 12: 25, 15: 37, 16: 52.
static __constant__ double2 c_wtab64[68] = {
    {1.0, -0.0}, {0.5000000000000001, -0.8660254037844386}, {-0.4999999999999998, -0.8660254037844387},
    {-1.0, -1.2246467991473532e-16}, {-0.5000000000000004, 0.8660254037844384},
    {0.5000000000000001, 0.8660254037844386}, {1.0, -0.0}, {0.766044443118978, -0.6427876096865393},
    {0.17364817766693041, -0.984807753012208}, {-0.4999999999999998, -0.8660254037844387},
    {-0.9396926207859083, -0.3420201433256689}, {-0.9396926207859084, 0.34202014332566866},
    {-0.5000000000000004, 0.8660254037844384}, {0.17364817766692997, 0.9848077530122081},
    {0.7660444431189778, 0.6427876096865396}, {1.0, -0.0}, {0.8090169943749475, -0.5877852522924731},
    {0.30901699437494745, -0.9510565162951535}, {-0.30901699437494734, -0.9510565162951536},
    {-0.8090169943749473, -0.5877852522924732}, {-1.0, -1.2246467991473532e-16},
    {-0.8090169943749476, 0.587785252292473}, {-0.30901699437494756, 0.9510565162951535},
    {0.30901699437494723, 0.9510565162951536}, {0.8090169943749473, 0.5877852522924734}, {1.0, -0.0},
    {0.8660254037844387, -0.49999999999999994}, {0.5000000000000001, -0.8660254037844386},
    {6.123233995736766e-17, -1.0}, {-0.4999999999999998, -0.8660254037844387},
    {-0.8660254037844387, -0.49999999999999994}, {-1.0, -1.2246467991473532e-16},
    {-0.8660254037844388, 0.4999999999999997}, {-0.5000000000000004, 0.8660254037844384},
    {-1.8369701987210297e-16, 1.0}, {0.5000000000000001, 0.8660254037844386},
    {0.8660254037844384, 0.5000000000000004}, {1.0, -0.0}, {0.9135454576426009, -0.40673664307580015},
    {0.6691306063588582, -0.7431448254773941}, {0.30901699437494745, -0.9510565162951535},
    {-0.10452846326765333, -0.9945218953682734}, {-0.4999999999999998, -0.8660254037844387},
    {-0.8090169943749473, -0.5877852522924732}, {-0.9781476007338057, -0.20791169081775931},
    {-0.9781476007338057, 0.20791169081775907}, {-0.8090169943749476, 0.587785252292473},
    {-0.5000000000000004, 0.8660254037844384}, {-0.10452846326765423, 0.9945218953682733},
    {0.30901699437494723, 0.9510565162951536}, {0.6691306063588585, 0.743144825477394},
    {0.913545457642601, 0.40673664307580015}, {1.0, -0.0}, {0.9238795325112867, -0.3826834323650898},
    {0.7071067811865476, -0.7071067811865475}, {0.38268343236508984, -0.9238795325112867},
    {6.123233995736766e-17, -1.0}, {-0.3826834323650897, -0.9238795325112867},
    {-0.7071067811865475, -0.7071067811865476}, {-0.9238795325112867, -0.3826834323650899},
    {-1.0, -1.2246467991473532e-16}, {-0.9238795325112868, 0.38268343236508967},
    {-0.7071067811865477, 0.7071067811865475}, {-0.38268343236509034, 0.9238795325112865},
    {-1.8369701987210297e-16, 1.0}, {0.38268343236509, 0.9238795325112866},
    {0.7071067811865474, 0.7071067811865477}, {0.9238795325112865, 0.3826834323650904},
};
static __constant__ float2 c_wtab32[68] = {
    {1.f, -0.f}, {0.5f, -0.866025388f}, {-0.5f, -0.866025388f}, {-1.f, -1.22464685e-16f}, {-0.5f, 0.866025388f},
    {0.5f, 0.866025388f}, {1.f, -0.f}, {0.766044438f, -0.642787635f}, {0.173648179f, -0.98480773f},
    {-0.5f, -0.866025388f}, {-0.939692616f, -0.342020154f}, {-0.939692616f, 0.342020154f}, {-0.5f, 0.866025388f},
    {0.173648179f, 0.98480773f}, {0.766044438f, 0.642787635f}, {1.f, -0.f}, {0.809017003f, -0.587785244f},
    {0.309017003f, -0.95105654f}, {-0.309017003f, -0.95105654f}, {-0.809017003f, -0.587785244f},
    {-1.f, -1.22464685e-16f}, {-0.809017003f, 0.587785244f}, {-0.309017003f, 0.95105654f},
    {0.309017003f, 0.95105654f}, {0.809017003f, 0.587785244f}, {1.f, -0.f}, {0.866025388f, -0.5f},
    {0.5f, -0.866025388f}, {6.12323426e-17f, -1.f}, {-0.5f, -0.866025388f}, {-0.866025388f, -0.5f},
    {-1.f, -1.22464685e-16f}, {-0.866025388f, 0.5f}, {-0.5f, 0.866025388f}, {-1.83697015e-16f, 1.f},
    {0.5f, 0.866025388f}, {0.866025388f, 0.5f}, {1.f, -0.f}, {0.91354543f, -0.406736642f},
    {0.669130623f, -0.74314481f}, {0.309017003f, -0.95105654f}, {-0.104528464f, -0.994521916f},
    {-0.5f, -0.866025388f}, {-0.809017003f, -0.587785244f}, {-0.978147626f, -0.207911685f},
    {-0.978147626f, 0.207911685f}, {-0.809017003f, 0.587785244f}, {-0.5f, 0.866025388f},
    {-0.104528464f, 0.994521916f}, {0.309017003f, 0.95105654f}, {0.669130623f, 0.74314481f},
    {0.91354543f, 0.406736642f}, {1.f, -0.f}, {0.923879504f, -0.382683426f}, {0.707106769f, -0.707106769f},
    {0.382683426f, -0.923879504f}, {6.12323426e-17f, -1.f}, {-0.382683426f, -0.923879504f},
    {-0.707106769f, -0.707106769f}, {-0.923879504f, -0.382683426f}, {-1.f, -1.22464685e-16f},
    {-0.923879504f, 0.382683426f}, {-0.707106769f, 0.707106769f}, {-0.382683426f, 0.923879504f},
    {-1.83697015e-16f, 1.f}, {0.382683426f, 0.923879504f}, {0.707106769f, 0.707106769f},
    {0.923879504f, 0.382683426f},
};
template <int R> struct WOff;
template <> struct WOff<6> { static constexpr int v = 0; };
template <> struct WOff<9> { static constexpr int v = 6; };
template <> struct WOff<10> { static constexpr int v = 15; };
template <> struct WOff<12> { static constexpr int v = 25; };
template <> struct WOff<15> { static constexpr int v = 37; };
template <> struct WOff<16> { static constexpr int v = 52; };

template <typename C, int S, int R> __device__ __forceinline__ C wconst(int m) {
  C w;
  if constexpr (sizeof(C) == 16) { const double2 t = c_wtab64[WOff<R>::v + m]; w.x = t.x; w.y = t.y; }
  else { const float2 t = c_wtab32[WOff<R>::v + m]; w.x = t.x; w.y = t.y; }
  if (S > 0) w.y = -w.y;
  return w;
}

template <typename C, int S, int R> __device__ __forceinline__ void dftR(C* x);

// R = R1 R2 in registers: R2 DFTs of length R1 (stride R2), constant twiddles w_R^{b k1},
// R1 DFTs of length R2; natural-order output X[k1 + R1 k2].
template <typename C, int S, int R, int R1, int R2> __device__ __forceinline__ void dft_comp(C* x) {
  C t[R];
#pragma unroll
  for (int b = 0; b < R2; ++b) {
    C u[R1];
#pragma unroll
    for (int a = 0; a < R1; ++a) u[a] = x[b + R2 * a];
    dftR<C, S, R1>(u);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) t[b + R2 * k1] = (b * k1 == 0) ? u[k1] : cmul(u[k1], wconst<C, S, R>(b * k1));
  }
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) {
    C v[R2];
#pragma unroll
    for (int b = 0; b < R2; ++b) v[b] = t[b + R2 * k1];
    dftR<C, S, R2>(v);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) x[k1 + R1 * k2] = v[k2];
  }
}

template <typename C, int S, int R> __device__ __forceinline__ void dftR(C* x) {
  if constexpr (R == 2) dft2<C, S>(x[0], x[1]);
  else if constexpr (R == 3) dft3<C, S>(x);
  else if constexpr (R == 4) dft4<C, S>(x);
  else if constexpr (R == 5) dft5<C, S>(x);
  else if constexpr (R == 8) dft8<C, S>(x);
  else if constexpr (R == 6) dft_comp<C, S, 6, 3, 2>(x);
  else if constexpr (R == 9) dft_comp<C, S, 9, 3, 3>(x);
  else if constexpr (R == 10) dft_comp<C, S, 10, 5, 2>(x);
  else if constexpr (R == 12) dft_comp<C, S, 12, 4, 3>(x);
  else if constexpr (R == 15) dft_comp<C, S, 15, 5, 3>(x);
  else dft_comp<C, S, 16, 4, 4>(x);
}

}  // namespace pw
