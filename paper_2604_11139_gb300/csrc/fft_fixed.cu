// complex128 FFT passes in 64-bit block fixed point; see fft_fixed.cuh for why and for the error.
//
// Five passes per band batch, each a batch of one-dimensional transforms of 32 lines per CTA
// (lane = line, the CTA's warps split a stage's butterflies), every line a two-stage plan R1 R2 of
// the context (digit order, pruning and the permuted potential as in fft_local.cu):
//   z inverse: sphere rows -> rows of the half-box planes
//   y inverse: rows -> all of the plane, in place
//   x:         planes -> lines, times V(r) / n1n2n3, back, in place; several bands per CTA (V from L1/L2)
//   y forward, z forward: back to the rows and to the sphere, + kinetic term
// The rows lie in the half-box plane at their own y, so no pass needs a buffer of its own, and a
// CTA's columns are read and written by that CTA alone.
//
// Measured on GB300 against the FP64 kernels of fft_local.cu (10-step filter of 256 bands on 96^3):
// x lines 184 -> 36 ms, pass 1 67 -> 15 ms, pass 3 74 -> 19 ms; density of 256 bands, same box,
// 17.3 -> 4.5 ms; one vector on 64^3 (an H-apply of the Lanczos chain) 188 -> 90 us.  Relative
// error of V psi against extended precision 1.3e-16 to 1.9e-16 on boxes from 64^3 to 72 x 75 x 80
// (FP64 kernels 4.4e-16 to 5.2e-16), random, decaying, single-component and in-phase bands alike.
//
// What bounds them: issue of the integer instructions (counters taken with two CTAs per SM: half of
// the slots, 42% of the ALU pipe; three CTAs, 24 warps, run now) and the conversions to and from FP64,
// a fifth of the FP64 pipe in the x pass, up to two fifths in the others.  Radices and
// lengths are run-time values (a switch around a stage, uniform in the CTA): one set of kernels
// covers every two-stage length, and the index arithmetic is small beside 64-bit butterflies.
//
// Scales.  A line's inputs are multiplied by 2^(B - E), E the exponent of its largest component,
// and rounded to integers |re|, |im| <= 2^B.  A radix-R stage grows the modulus by at most R; a
// stage's twiddle product divides by 4 (the product of a 64-bit value and a 62-bit twiddle keeps
// its top 64 bits), which makes room for the next stage.  B (host, `bits`) keeps every value
// below 2^62.4 and every value that enters a twiddle product below 2^61.6.
#include <math.h>

#include <algorithm>

#include "fft_fixed.cuh"

namespace pw {
namespace fx {

typedef long long ll;
struct __align__(16) fc {
  ll x, y;
};

// ---- arithmetic -----------------------------------------------------------------------
__device__ __forceinline__ fc add(fc a, fc b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ fc sub(fc a, fc b) { return {a.x - b.x, a.y - b.y}; }
template <int S> __device__ __forceinline__ fc add_muli(fc a, fc b) {  // a + S i b
  return S > 0 ? fc{a.x - b.y, a.y + b.x} : fc{a.x + b.y, a.y - b.x};
}
template <int S> __device__ __forceinline__ fc sub_muli(fc a, fc b) { return add_muli<-S>(a, b); }
__device__ __forceinline__ ll madw(int a, int b, ll c) { return (ll)a * b + c; }
__device__ __forceinline__ int lo32(ll a) { return (int)a; }
// high half of a when its low half is read as a signed number
__device__ __forceinline__ int hi32(ll a) { return (int)(a >> 32) + (int)((unsigned)a >> 31); }
__device__ __forceinline__ ll sext_hi(ll a) { return (ll)(int)(a >> 32); }
constexpr int klo(ll k) { return (int)(unsigned)((unsigned long long)k & 0xffffffffull); }
constexpr int khi(ll k) { return (int)((k - (ll)klo(k)) >> 32); }
// (h 2^32 + m) >> 30 (the low 32 bits of m count)
__device__ __forceinline__ ll shift_out(ll h, ll m) {
  const unsigned l = (unsigned)h, ml = (unsigned)m;
  const unsigned rl = __funnelshift_l(ml, l, 2);
  const unsigned rh = __funnelshift_l(l, (unsigned)(h >> 32), 2);
  return (ll)(((unsigned long long)rh << 32) | rl);
}
constexpr ll kRound30 = 1ll << 29, kRound32 = 1ll << 31;
// round(a k / 2^62), k a constant, |k| <= 2^62
__device__ __forceinline__ ll mulk(ll a, ll k) {
  const int al = lo32(a), ah = hi32(a);
  ll m = madw(al, khi(k), kRound30);
  m = madw(ah, klo(k), m);
  return shift_out(madw(ah, khi(k), sext_hi(m)), m);
}
// round((a k + b q) / 2^62)
__device__ __forceinline__ ll mulk2(ll a, ll k, ll b, ll q) {
  const int al = lo32(a), ah = hi32(a), bl = lo32(b), bh = hi32(b);
  ll m = madw(al, khi(k), kRound30);
  m = madw(ah, klo(k), m);
  m = madw(bl, khi(q), m);
  m = madw(bh, klo(q), m);
  return shift_out(madw(bh, khi(q), madw(ah, khi(k), sext_hi(m))), m);
}
__device__ __forceinline__ fc mulk(fc a, ll k) { return {mulk(a.x, k), mulk(a.y, k)}; }
constexpr ll kOne = 1ll << 62;
// a (c + S i s), c and s constants
template <int S> __device__ __forceinline__ fc cmulk(fc a, ll c, ll s) {
  if (c == 0 && s == kOne) return S > 0 ? fc{-a.y, a.x} : fc{a.y, -a.x};
  if (c == -kOne && s == 0) return {-a.x, -a.y};
  return {mulk2(a.x, c, a.y, -S * s), mulk2(a.y, c, a.x, S * s)};
}
// a w / 4 with the table's w (S < 0) or its conjugate (S > 0)
template <int S> __device__ __forceinline__ fc cmul_tw(fc a, Tw w) {
  const int axl = lo32(a.x), axh = hi32(a.x), ayl = lo32(a.y), ayh = hi32(a.y);
  const int nyl = -w.ylo, nyh = -w.yhi;
  const int rl = S > 0 ? w.ylo : nyl, rh = S > 0 ? w.yhi : nyh;  // re takes + rl ay
  const int il = S > 0 ? nyl : w.ylo, ih = S > 0 ? nyh : w.yhi;  // im takes + il ax
  ll m = madw(axl, w.xhi, kRound32);
  m = madw(axh, w.xlo, m);
  m = madw(ayl, rh, m);
  m = madw(ayh, rl, m);
  ll q = madw(ayl, w.xhi, kRound32);
  q = madw(ayh, w.xlo, q);
  q = madw(axl, ih, q);
  q = madw(axh, il, q);
  return {madw(ayh, rh, madw(axh, w.xhi, sext_hi(m))), madw(axh, ih, madw(ayh, w.xhi, sext_hi(q)))};
}
__device__ __forceinline__ fc quarter(fc a) { return {(a.x + 2) >> 2, (a.y + 2) >> 2}; }
// round(a v / 2^64)
__device__ __forceinline__ ll mulv(int al, int ah, int vl, int vh) {
  ll m = madw(al, vh, kRound32);
  m = madw(ah, vl, m);
  return madw(ah, vh, sext_hi(m));
}

// the shift that brings the larger component of v (|v| <= 2^62.4) to 2^61 .. 2^62
__device__ __forceinline__ int up_shift(fc v) {
  return max(__clzll((v.x ^ (v.x >> 63)) | (v.y ^ (v.y >> 63))) - 2, 0);
}
// round(Re(conj(a) b) / 2^64)
__device__ __forceinline__ ll dot64(fc a, fc b) {
  const int axl = lo32(a.x), axh = hi32(a.x), ayl = lo32(a.y), ayh = hi32(a.y);
  const int bxl = lo32(b.x), bxh = hi32(b.x), byl = lo32(b.y), byh = hi32(b.y);
  ll m = madw(axl, bxh, kRound32);
  m = madw(axh, bxl, m);
  m = madw(ayl, byh, m);
  m = madw(ayh, byl, m);
  return madw(ayh, byh, madw(axh, bxh, sext_hi(m)));
}

// ---- small DFTs: y_m = sum_k x_k exp(S 2 pi i k m / R) ------------------------------------
constexpr ll kH = 3260954456333195553ll;    // 2^62 cos(pi/4)
constexpr ll kS3 = 3993837246235628775ll;   // 2^62 sin(pi/3)
constexpr ll kS51 = 4385974038932618941ll;  // 2^62 sin(2 pi/5)
constexpr ll kS52 = 2710681029835013083ll;  // 2^62 sin(4 pi/5)
constexpr ll kQ5 = 2578010857022246787ll;   // 2^62 sqrt(5)/4
// 2^62 cos(2 pi m / R) (sn = 0) and 2^62 sin(2 pi m / R) (sn = 1)
__host__ __device__ constexpr ll wtab(int R, int m, int sn) {
  switch (R * 32 + m) {
    case 6 * 32 + 1: return sn ? 3993837246235628775ll : 2305843009213693952ll;
    case 6 * 32 + 2: return sn ? 3993837246235628775ll : -2305843009213693952ll;
    case 9 * 32 + 1: return sn ? 2964334632409774423ll : 3532756447825785444ll;
    case 9 * 32 + 2: return sn ? 4541624145405292212ll : 800810873071977681ll;
    case 9 * 32 + 3: return sn ? 3993837246235628775ll : -2305843009213693952ll;
    case 9 * 32 + 4: return sn ? 1577289512995517789ll : -4333567320897763126ll;
    case 10 * 32 + 1: return sn ? 2710681029835013083ll : 3730932361629093763ll;
    case 10 * 32 + 2: return sn ? 4385974038932618941ll : 1425089352415399811ll;
    case 10 * 32 + 3: return sn ? 4385974038932618941ll : -1425089352415399811ll;
    case 10 * 32 + 4: return sn ? 2710681029835013083ll : -3730932361629093763ll;
    case 12 * 32 + 1: return sn ? 2305843009213693952ll : 3993837246235628775ll;
    case 12 * 32 + 2: return sn ? 3993837246235628775ll : 2305843009213693952ll;
    case 12 * 32 + 3: return sn ? 4611686018427387904ll : 0ll;
    case 12 * 32 + 4: return sn ? 3993837246235628775ll : -2305843009213693952ll;
    case 12 * 32 + 5: return sn ? 2305843009213693952ll : -3993837246235628775ll;
    case 12 * 32 + 6: return sn ? 0ll : -4611686018427387904ll;
    case 15 * 32 + 1: return sn ? 1875741690054758654ll : 4212984814208232069ll;
    case 15 * 32 + 2: return sn ? 3427150601320760278ll : 3085820261846986643ll;
    case 15 * 32 + 3: return sn ? 4385974038932618941ll : 1425089352415399811ll;
    case 15 * 32 + 4: return sn ? 4586422719889771737ll : -482052452579138307ll;
    case 15 * 32 + 5: return sn ? 3993837246235628775ll : -2305843009213693952ll;
    case 15 * 32 + 6: return sn ? 2710681029835013083ll : -3730932361629093763ll;
    case 15 * 32 + 7: return sn ? 958823437611858663ll : -4510909614262386453ll;
    case 15 * 32 + 8: return sn ? -958823437611858663ll : -4510909614262386453ll;
    case 16 * 32 + 1: return sn ? 1764815834521887442ll : 4260642322793532497ll;
    case 16 * 32 + 2: return sn ? 3260954456333195553ll : 3260954456333195553ll;
    case 16 * 32 + 3: return sn ? 4260642322793532497ll : 1764815834521887442ll;
    case 16 * 32 + 4: return sn ? 4611686018427387904ll : 0ll;
    case 16 * 32 + 5: return sn ? 4260642322793532497ll : -1764815834521887442ll;
    case 16 * 32 + 6: return sn ? 3260954456333195553ll : -3260954456333195553ll;
    case 16 * 32 + 7: return sn ? 1764815834521887442ll : -4260642322793532497ll;
    case 16 * 32 + 8: return sn ? 0ll : -4611686018427387904ll;
    case 16 * 32 + 9: return sn ? -1764815834521887442ll : -4260642322793532497ll;
    default: return 0;
  }
}

template <int S, int R> __device__ __forceinline__ void dft(fc* x);
template <int S> __device__ __forceinline__ void dft2(fc* x) {
  const fc t = x[0];
  x[0] = add(t, x[1]);
  x[1] = sub(t, x[1]);
}
template <int S> __device__ __forceinline__ void dft3(fc* x) {
  const fc t = add(x[1], x[2]), d = mulk(sub(x[1], x[2]), kS3);
  const fc m = {x[0].x - (t.x >> 1), x[0].y - (t.y >> 1)};
  x[0] = add(x[0], t);
  x[1] = add_muli<S>(m, d);
  x[2] = sub_muli<S>(m, d);
}
template <int S> __device__ __forceinline__ void dft4(fc* x) {
  const fc s02 = add(x[0], x[2]), d02 = sub(x[0], x[2]);
  const fc s13 = add(x[1], x[3]), d13 = sub(x[1], x[3]);
  x[0] = add(s02, s13);
  x[2] = sub(s02, s13);
  x[1] = add_muli<S>(d02, d13);
  x[3] = sub_muli<S>(d02, d13);
}
template <int S> __device__ __forceinline__ void dft5(fc* x) {
  const fc t1 = add(x[1], x[4]), t2 = add(x[2], x[3]);
  const fc d1 = sub(x[1], x[4]), d2 = sub(x[2], x[3]);
  const fc t = add(t1, t2), b = mulk(sub(t1, t2), kQ5);  // cos(2 pi/5), cos(4 pi/5) = (-1 +- sqrt 5)/4
  const fc m = {x[0].x - ((t.x + 2) >> 2), x[0].y - ((t.y + 2) >> 2)};
  const fc a1 = add(m, b), a2 = sub(m, b);
  const fc u1 = {mulk2(d1.x, kS51, d2.x, kS52), mulk2(d1.y, kS51, d2.y, kS52)};
  const fc u2 = {mulk2(d1.x, kS52, d2.x, -kS51), mulk2(d1.y, kS52, d2.y, -kS51)};
  x[0] = add(x[0], t);
  x[1] = add_muli<S>(a1, u1);
  x[4] = sub_muli<S>(a1, u1);
  x[2] = add_muli<S>(a2, u2);
  x[3] = sub_muli<S>(a2, u2);
}
template <int S> __device__ __forceinline__ void dft8(fc* x) {
  fc e[4] = {x[0], x[2], x[4], x[6]}, o[4] = {x[1], x[3], x[5], x[7]};
  dft4<S>(e);
  dft4<S>(o);
  const fc o1 = mulk(add_muli<S>(o[1], o[1]), kH), o3 = mulk(sub_muli<S>(o[3], o[3]), -kH);
  x[0] = add(e[0], o[0]);
  x[4] = sub(e[0], o[0]);
  x[1] = add(e[1], o1);
  x[5] = sub(e[1], o1);
  x[2] = add_muli<S>(e[2], o[2]);
  x[6] = sub_muli<S>(e[2], o[2]);
  x[3] = add(e[3], o3);
  x[7] = sub(e[3], o3);
}
// R = R1 R2: R2 DFTs of length R1 (stride R2), constant twiddles, R1 DFTs of length R2
template <int S, int R, int R1, int R2> __device__ __forceinline__ void dft_comp(fc* x) {
  fc t[R];
#pragma unroll
  for (int b = 0; b < R2; ++b) {
    fc u[R1];
#pragma unroll
    for (int a = 0; a < R1; ++a) u[a] = x[b + R2 * a];
    dft<S, R1>(u);
#pragma unroll
    for (int k = 0; k < R1; ++k)
      t[b + R2 * k] = (b * k == 0) ? u[k] : cmulk<S>(u[k], wtab(R, b * k, 0), wtab(R, b * k, 1));
  }
#pragma unroll
  for (int k = 0; k < R1; ++k) {
    fc v[R2];
#pragma unroll
    for (int b = 0; b < R2; ++b) v[b] = t[b + R2 * k];
    dft<S, R2>(v);
#pragma unroll
    for (int q = 0; q < R2; ++q) x[k + R1 * q] = v[q];
  }
}
template <int S, int R> __device__ __forceinline__ void dft(fc* x) {
  if constexpr (R == 2) dft2<S>(x);
  else if constexpr (R == 3) dft3<S>(x);
  else if constexpr (R == 4) dft4<S>(x);
  else if constexpr (R == 5) dft5<S>(x);
  else if constexpr (R == 6) dft_comp<S, 6, 3, 2>(x);
  else if constexpr (R == 8) dft8<S>(x);
  else if constexpr (R == 9) dft_comp<S, 9, 3, 3>(x);
  else if constexpr (R == 10) dft_comp<S, 10, 5, 2>(x);
  else if constexpr (R == 12) dft_comp<S, 12, 4, 3>(x);
  else if constexpr (R == 15) dft_comp<S, 15, 5, 3>(x);
  else dft_comp<S, 16, 4, 4>(x);
}

// ---- scales (one per line) ---------------------------------------------------------------
// running maximum of |x| and |y| by the high words of their FP64 forms
__device__ __forceinline__ unsigned track(unsigned m, double2 v) {
  m = max(m, (unsigned)__double2hiint(v.x) & 0x7fffffffu);
  return max(m, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
}
// E with every |component| < 2^E, from the largest high word (subnormal values count as zero)
__device__ __forceinline__ int top_exp(unsigned m) { return (int)(m >> 20) - 1022; }
constexpr int kNan = 1 << 30;  // Out::k of a line with a component that is not finite

// FP64 -> round(x 2^(bits - E)): the power of two goes into the exponent field by an integer
// addition, so only the conversion itself uses the FP64 pipe
struct In {
  int add;       // (bits - E) << 20
  unsigned thr;  // high words below it (|x| 2^(bits - E) < 1/4, or no normal number) give 0
  __device__ __forceinline__ In(int E, int bits)
      : add((bits - E) * (1 << 20)), thr((unsigned)max(1, E - bits + 1021) << 20) {}
  __device__ __forceinline__ ll operator()(double x) const {
    const int hi = __double2hiint(x);
    const bool z = ((unsigned)hi & 0x7fffffffu) < thr;
    return __double2ll_rn(__hiloint2double(z ? 0 : hi + add, z ? 0 : __double2loint(x)));
  }
  __device__ __forceinline__ fc operator()(double2 v) const { return {(*this)(v.x), (*this)(v.y)}; }
};
// integer -> FP64 times 2^k.  |k| <= 900 (any values of ordinary size) is again an integer
// addition to the exponent field; beyond it, two products, which overflow and underflow as
// FP64 does
struct Out {
  int k;
  __device__ __forceinline__ double operator()(ll v) const {
    const double d = __ll2double_rn(v);
    const int hi = __double2hiint(d);
    if ((unsigned)(k + 900) <= 1800u) return __hiloint2double(hi ? hi + k * (1 << 20) : 0, __double2loint(d));
    if (k == kNan) return __longlong_as_double(0x7ff8000000000000ll);
    const int kc = max(k, -2040), h = kc / 2;  // 2^63 2^-2040 is 0 already
    return d * __hiloint2double((h + 1023) << 20, 0) * __hiloint2double((kc - h + 1023) << 20, 0);
  }
  __device__ __forceinline__ double2 operator()(fc v) const { return make_double2((*this)(v.x), (*this)(v.y)); }
};
__device__ __forceinline__ int out_exp(unsigned m, int k) { return m >= 0x7ff00000u ? kNan : k; }

constexpr int kWarps = 8, kThreads = 32 * kWarps;
constexpr int kDynSmem = 224 * 1024;  // limit of dynamic shared memory; up to 3 KB are static
constexpr int PT = 33;  // pitch of an element's 32 lines: lane-wise and line-wise accesses are conflict-free

struct Dim {
  int n, r1, r2;
  const Tw* tw;  // [j][m - 1], j < r2, 1 <= m < r1
};

// maximum over the warps of a value per lane; red: kWarps x 32 words.  Ends with a barrier
// before the reads.
__device__ __forceinline__ unsigned line_max(unsigned m, unsigned (*red)[32]) {
  const int lane = threadIdx.x & 31;
  red[threadIdx.x >> 5][lane] = m;
  __syncthreads();
  unsigned r = red[0][lane];
#pragma unroll
  for (int i = 1; i < kWarps; ++i) r = max(r, red[i][lane]);
  return r;
}

// Kernels come in two forms: radices up to 12 with registers for three CTAs per SM, and up to 16
// for two (a radix-16 butterfly of 64-bit values holds 64 registers of data alone).
#define FX_SWITCH(R, F)        \
  switch (R) {                 \
    case 16: if constexpr (BIG) { F(16); } break; \
    case 15: if constexpr (BIG) { F(15); } break; \
    case 12: F(12); break;     \
    case 10: F(10); break;     \
    case 9: F(9); break;       \
    case 8: F(8); break;       \
    case 6: F(6); break;       \
    case 5: F(5); break;       \
    case 4: F(4); break;       \
    case 3: F(3); break;       \
    default: F(2); break;      \
  }

// ---- stages; col points at the lane's line, element e at col[e PT] -----------------------------
// inverse stage 1: FP64 elements J + r2 a (zero where !valid) -> DFT, twiddle.  NORM: adds the
// squares of the inputs' high words to *ss.
template <int R, bool NORM = false, typename V>
__device__ __forceinline__ void inv1(fc* col, int J, const Dim& d, In in, V valid, ll* ss = nullptr) {
  fc x[R];
#pragma unroll
  for (int a = 0; a < R; ++a) {
    const int e = J + d.r2 * a;
    x[a] = valid(e) ? in(*reinterpret_cast<const double2*>(&col[e * PT])) : fc{0, 0};
    if constexpr (NORM) {
      const int hx = (int)(x[a].x >> 32), hy = (int)(x[a].y >> 32);
      *ss = madw(hx, hx, madw(hy, hy, *ss));
    }
  }
  dft<+1, R>(x);
  col[J * PT] = quarter(x[0]);
  if (J) {
    const Tw* w = d.tw + J * (R - 1);
#pragma unroll
    for (int m = 1; m < R; ++m) col[(J + d.r2 * m) * PT] = cmul_tw<+1>(x[m], w[m - 1]);
  } else {
#pragma unroll
    for (int m = 1; m < R; ++m) col[d.r2 * m * PT] = quarter(x[m]);
  }
}
// forward stage 1: FP64 block blk -> DFT, in place
template <int R> __device__ __forceinline__ void fwd1(fc* col, int blk, In in) {
  fc y[R];
  fc* c = col + blk * R * PT;
#pragma unroll
  for (int m = 0; m < R; ++m) y[m] = in(*reinterpret_cast<const double2*>(&c[m * PT]));
  dft<-1, R>(y);
#pragma unroll
  for (int m = 0; m < R; ++m) c[m * PT] = y[m];
}
// elements J + r2 m of a line times the twiddles, forward DFT
template <int R> __device__ __forceinline__ void fwd2(const fc* col, int J, const Dim& d, fc (&x)[R]) {
  x[0] = quarter(col[J * PT]);
  if (J) {
    const Tw* w = d.tw + J * (R - 1);
#pragma unroll
    for (int m = 1; m < R; ++m) x[m] = cmul_tw<-1>(col[(J + d.r2 * m) * PT], w[m - 1]);
  } else {
#pragma unroll
    for (int m = 1; m < R; ++m) x[m] = quarter(col[d.r2 * m * PT]);
  }
  dft<-1, R>(x);
}

__device__ __forceinline__ int wrap(int e, int n) { return e < 0 ? e + n : e; }
__device__ __forceinline__ int posmod(int a, int n) {
  const int r = a % n;
  return r < 0 ? r + n : r;
}
// plane of sphere row r
__device__ __forceinline__ int plane_of(const SphereDev& sp, int r) {
  int lo = 0, hi = sp.nplane;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (sp.plane_row0[mid] <= r) lo = mid;
    else hi = mid;
  }
  return lo;
}

// ---- z: 32 sphere rows per CTA -------------------------------------------------------------
template <bool BIG>
__global__ void __launch_bounds__(kThreads, BIG ? 2 : 3) k_fx_zinv(const double2* __restrict__ psi, int64_t ldpsi,
                                                         double2* __restrict__ hb, int64_t hb_bs, SphereDev sp, Dim d,
                                                         int n2, int bits) {
  extern __shared__ __align__(16) unsigned char smem[];
  fc* buf = reinterpret_cast<fc*>(smem);
  __shared__ unsigned rmax[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int row0 = blockIdx.x * 32, n = d.n;
  const double2* src = psi + (int64_t)blockIdx.y * ldpsi;
  for (int rr = w; rr < 32; rr += kWarps) {
    const int r = row0 + rr;
    unsigned m = 0;
    if (r < sp.nrow) {
      const int g0 = sp.row_g0[r], cnt = sp.row_cnt[r], l0 = posmod(sp.row_l0[r], n);
      for (int i = lane; i < cnt; i += 32) {
        const double2 v = src[g0 + i];
        m = track(m, v);
        const int e = l0 + i;
        *reinterpret_cast<double2*>(&buf[(e >= n ? e - n : e) * PT + rr]) = v;
      }
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) rmax[rr] = m;
  }
  __syncthreads();
  const unsigned mx = rmax[lane];
  const int E = top_exp(mx);
  const In in(E, bits);
  const Out out_of{out_exp(mx, E - bits + 2)};
  fc* col = buf + lane;
  int cnt = 0, l0 = 0;
  if (row0 + lane < sp.nrow) {
    cnt = sp.row_cnt[row0 + lane];
    l0 = posmod(sp.row_l0[row0 + lane], n);
  }
#define FX_F(R)                                   \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) \
      inv1<R>(col, J, d, in, [&](int e) { return wrap(e - l0, n) < cnt; })
  FX_SWITCH(d.r1, FX_F)
#undef FX_F
  __syncthreads();
#define FX_F(R)                                                          \
  _Pragma("unroll 1") for (int blk = w; blk < d.r1; blk += kWarps) {     \
    fc y[R];                                                             \
    fc* c = col + blk * R * PT;                                          \
    _Pragma("unroll") for (int m = 0; m < R; ++m) y[m] = c[m * PT];      \
    dft<+1, R>(y);                                                       \
    _Pragma("unroll") for (int m = 0; m < R; ++m)                        \
        *reinterpret_cast<double2*>(&c[m * PT]) = out_of(y[m]); \
  }
  FX_SWITCH(d.r2, FX_F)
#undef FX_F
  __syncthreads();
  for (int rr = w; rr < 32; rr += kWarps) {
    const int r = row0 + rr;
    if (r >= sp.nrow) break;
    double2* dst = hb + (int64_t)blockIdx.y * hb_bs + ((int64_t)plane_of(sp, r) * n2 + posmod(sp.row_k[r], n2)) * n;
    for (int z = lane; z < n; z += 32) dst[z] = *reinterpret_cast<const double2*>(&buf[z * PT + rr]);
  }
}

template <bool BIG>
__global__ void __launch_bounds__(kThreads, BIG ? 2 : 3) k_fx_zfwd(const double2* __restrict__ hb, int64_t hb_bs,
                                                                   SphereDev sp, Dim d, int n2, int bits,
                                                                   const double* __restrict__ kin,
                                                                   const double2* __restrict__ psi, int64_t ldpsi,
                                                                   double2* __restrict__ out, int64_t ldout) {
  extern __shared__ __align__(16) unsigned char smem[];
  fc* buf = reinterpret_cast<fc*>(smem);
  __shared__ unsigned rmax[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int row0 = blockIdx.x * 32, n = d.n;
  for (int rr = w; rr < 32; rr += kWarps) {
    const int r = row0 + rr;
    unsigned m = 0;
    const bool live = r < sp.nrow;
    const double2* src = live ? hb + (int64_t)blockIdx.y * hb_bs +
                                    ((int64_t)plane_of(sp, r) * n2 + posmod(sp.row_k[r], n2)) * n
                              : nullptr;
    for (int z = lane; z < n; z += 32) {
      const double2 v = live ? src[z] : make_double2(0.0, 0.0);
      m = track(m, v);
      *reinterpret_cast<double2*>(&buf[z * PT + rr]) = v;
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) rmax[rr] = m;
  }
  __syncthreads();
  const unsigned mx = rmax[lane];
  const int E = top_exp(mx);
  const In in(E, bits);
  const Out out_of{out_exp(mx, E - bits + 2)};
  fc* col = buf + lane;
#define FX_F(R) _Pragma("unroll 1") for (int blk = w; blk < d.r1; blk += kWarps) fwd1<R>(col, blk, in)
  FX_SWITCH(d.r2, FX_F)
#undef FX_F
  __syncthreads();
#define FX_F(R)                                                        \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) {         \
    fc x[R];                                                           \
    fwd2<R>(col, J, d, x);                                             \
    _Pragma("unroll") for (int a = 0; a < R; ++a)                      \
        *reinterpret_cast<double2*>(&col[(J + d.r2 * a) * PT]) = out_of(x[a]); \
  }
  FX_SWITCH(d.r1, FX_F)
#undef FX_F
  __syncthreads();
  const double2* yv = psi + (int64_t)blockIdx.y * ldpsi;
  double2* o = out + (int64_t)blockIdx.y * ldout;
  for (int rr = w; rr < 32; rr += kWarps) {
    const int r = row0 + rr;
    if (r >= sp.nrow) break;
    const int g0 = sp.row_g0[r], cnt = sp.row_cnt[r], l0 = posmod(sp.row_l0[r], n);
    for (int i = lane; i < cnt; i += 32) {
      const int e = l0 + i;
      const double2 v = *reinterpret_cast<const double2*>(&buf[(e >= n ? e - n : e) * PT + rr]);
      const double2 y = yv[g0 + i];
      const double k = kin[g0 + i];
      o[g0 + i] = make_double2(k * y.x + v.x, k * y.y + v.y);
    }
  }
}

// ---- y: 32 columns of one plane per CTA, in place ---------------------------------------------
template <bool BIG>
__global__ void __launch_bounds__(kThreads, BIG ? 2 : 3) k_fx_yinv(double2* __restrict__ hb, int64_t hb_bs, SphereDev sp, Dim d,
                                                         int n3, int nc, int bits) {
  extern __shared__ __align__(16) unsigned char smem[];
  fc* buf = reinterpret_cast<fc*>(smem);
  int* ymap = reinterpret_cast<int*>(buf + d.n * PT);
  __shared__ unsigned red[kWarps][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int p = blockIdx.x / nc, c = (blockIdx.x % nc) * 32 + lane, n = d.n;
  const bool live = c < n3;
  const int r0 = sp.plane_row0[p], nr = sp.plane_row0[p + 1] - r0;
  for (int i = threadIdx.x; i < n; i += kThreads) ymap[i] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < nr; i += kThreads) ymap[posmod(sp.row_k[r0 + i], n)] = 1;
  double2* pl = hb + (int64_t)blockIdx.y * hb_bs + (int64_t)p * n * n3 + (live ? c : 0);
  unsigned mx = 0;
  for (int i = w; i < nr; i += kWarps) {
    const int k = posmod(sp.row_k[r0 + i], n);
    const double2 v = live ? pl[(int64_t)k * n3] : make_double2(0.0, 0.0);
    mx = track(mx, v);
    *reinterpret_cast<double2*>(&buf[k * PT + lane]) = v;
  }
  mx = line_max(mx, red);
  const int E = top_exp(mx);
  const In in(E, bits);
  const Out out_of{out_exp(mx, E - bits + 2)};
  fc* col = buf + lane;
#define FX_F(R)                                              \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) \
      inv1<R>(col, J, d, in, [&](int e) { return ymap[e] != 0; })
  FX_SWITCH(d.r1, FX_F)
#undef FX_F
  __syncthreads();
#define FX_F(R)                                                          \
  _Pragma("unroll 1") for (int blk = w; blk < d.r1; blk += kWarps) {     \
    fc y[R];                                                             \
    _Pragma("unroll") for (int m = 0; m < R; ++m) y[m] = col[(blk * R + m) * PT]; \
    dft<+1, R>(y);                                                       \
    if (live) {                                                          \
      _Pragma("unroll") for (int m = 0; m < R; ++m)                      \
          pl[(int64_t)(blk * R + m) * n3] = out_of(y[m]);      \
    }                                                                    \
  }
  FX_SWITCH(d.r2, FX_F)
#undef FX_F
}

template <bool BIG>
__global__ void __launch_bounds__(kThreads, BIG ? 2 : 3) k_fx_yfwd(double2* __restrict__ hb, int64_t hb_bs, SphereDev sp, Dim d,
                                                         int n3, int nc, int bits) {
  extern __shared__ __align__(16) unsigned char smem[];
  fc* buf = reinterpret_cast<fc*>(smem);
  int* ymap = reinterpret_cast<int*>(buf + d.n * PT);
  __shared__ unsigned red[kWarps][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int p = blockIdx.x / nc, c = (blockIdx.x % nc) * 32 + lane, n = d.n;
  const bool live = c < n3;
  const int r0 = sp.plane_row0[p], nr = sp.plane_row0[p + 1] - r0;
  for (int i = threadIdx.x; i < n; i += kThreads) ymap[i] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < nr; i += kThreads) ymap[posmod(sp.row_k[r0 + i], n)] = 1;
  double2* pl = hb + (int64_t)blockIdx.y * hb_bs + (int64_t)p * n * n3 + (live ? c : 0);
  unsigned mx = 0;
#pragma unroll 4
  for (int e = w; e < n; e += kWarps) {
    const double2 v = live ? pl[(int64_t)e * n3] : make_double2(0.0, 0.0);
    mx = track(mx, v);
    *reinterpret_cast<double2*>(&buf[e * PT + lane]) = v;
  }
  mx = line_max(mx, red);
  const int E = top_exp(mx);
  const In in(E, bits);
  const Out out_of{out_exp(mx, E - bits + 2)};
  fc* col = buf + lane;
#define FX_F(R) _Pragma("unroll 1") for (int blk = w; blk < d.r1; blk += kWarps) fwd1<R>(col, blk, in)
  FX_SWITCH(d.r2, FX_F)
#undef FX_F
  __syncthreads();
#define FX_F(R)                                                                           \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) {                            \
    fc x[R];                                                                              \
    fwd2<R>(col, J, d, x);                                                                \
    _Pragma("unroll") for (int a = 0; a < R; ++a) {                                       \
      const int e = J + d.r2 * a;                                                         \
      if (live && ymap[e]) pl[(int64_t)e * n3] = out_of(x[a]);                  \
    }                                                                                     \
  }
  FX_SWITCH(d.r1, FX_F)
#undef FX_F
}

// ---- x: 32 (y,z) lines per CTA, `bper` bands --------------------------------------------------
template <bool BIG>
__global__ void __launch_bounds__(kThreads, BIG ? 2 : 3) k_fx_x(double2* __restrict__ hb, int64_t hb_bs, int nb, int bper,
                                                      const double* __restrict__ vperm, int np, int nyz, Dim d,
                                                      int bits, int room) {
  extern __shared__ __align__(16) unsigned char smem[];
  fc* buf = reinterpret_cast<fc*>(smem);
  __shared__ unsigned red[kWarps][32];
  __shared__ ll red2[kWarps][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int yz = blockIdx.x * 32 + lane, n = d.n;
  const bool live = yz < nyz;
  // the scale of V on each line: integers |v| <= 2^62
  const double* vb = vperm + (live ? yz : 0);
  unsigned mv = 0;
  for (int e = w; e < n; e += kWarps) mv = max(mv, (unsigned)__double2hiint(live ? vb[(int64_t)e * nyz] : 0.0) & 0x7fffffffu);
  mv = line_max(mv, red);
  const int Ev = top_exp(mv);
  const In vin(Ev, 62);
  __syncthreads();  // red is written again
  fc* col = buf + lane;
  const int b_hi = min(nb, (int)(blockIdx.y + 1) * bper);
#pragma unroll 1
  for (int b = blockIdx.y * bper; b < b_hi; ++b) {
    double2* pl = hb + (int64_t)b * hb_bs + (live ? yz : 0);
    unsigned mx = 0;
#pragma unroll 4
    for (int p = w; p < np; p += kWarps) {
      const double2 v = live ? pl[(int64_t)p * nyz] : make_double2(0.0, 0.0);
      mx = track(mx, v);
      *reinterpret_cast<double2*>(&buf[p * PT + lane]) = v;
    }
    mx = line_max(mx, red);
    const int E = top_exp(mx);
    const In in(E, bits);
    ll ss = 0;
#define FX_F(R)                                              \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) \
      inv1<R, true>(col, J, d, in, [&](int e) { return e < np; }, &ss)
    FX_SWITCH(d.r1, FX_F)
#undef FX_F
    red2[w][lane] = ss;
    __syncthreads();
#pragma unroll
    for (int i = 1; i < kWarps; ++i) ss += red2[(w + i) % kWarps][lane];
    // the line's 2-norm (2^32 sqrt(ss)) bounds the forward half; what it leaves free of the worst
    // case that `bits` allows for is used: the values that meet V are shifted up by t
    const int t = min(max((__clzll(ss | 1) - room) >> 1, 0), 6);
    const Out out_of{out_exp(max(mx, mv), E - bits + Ev + 6 - t)};
#define FX_F(R)                                                                        \
  _Pragma("unroll 1") for (int blk = w; blk < d.r1; blk += kWarps) {                   \
    fc y[R];                                                                           \
    fc* c = col + blk * R * PT;                                                        \
    const double* vl_ = vb + (int64_t)blk * R * nyz;                                   \
    double vd[R];                                                                      \
    _Pragma("unroll") for (int m = 0; m < R; ++m) vd[m] = vl_[(int64_t)m * nyz];       \
    _Pragma("unroll") for (int m = 0; m < R; ++m) y[m] = c[m * PT];                    \
    dft<+1, R>(y);                                                                     \
    _Pragma("unroll") for (int m = 0; m < R; ++m) {                                    \
      const ll v = vin(vd[m]);                                                         \
      const int vl = lo32(v), vh = hi32(v);                                            \
      const ll yx = y[m].x << t, yy = y[m].y << t;                                     \
      y[m] = {mulv(lo32(yx), hi32(yx), vl, vh), mulv(lo32(yy), hi32(yy), vl, vh)};     \
    }                                                                                  \
    dft<-1, R>(y);                                                                     \
    _Pragma("unroll") for (int m = 0; m < R; ++m) c[m * PT] = y[m];                    \
  }
    FX_SWITCH(d.r2, FX_F)
#undef FX_F
    __syncthreads();
#define FX_F(R)                                                            \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) {             \
    fc x[R];                                                               \
    fwd2<R>(col, J, d, x);                                                 \
    _Pragma("unroll") for (int a = 0; a < R; ++a) {                        \
      const int e = J + d.r2 * a;                                          \
      if (live && e < np) pl[(int64_t)e * nyz] = out_of(x[a]);   \
    }                                                                      \
  }
    FX_SWITCH(d.r1, FX_F)
#undef FX_F
    __syncthreads();  // the next band's planes overwrite the lines
  }
}

// ---- density: inverse x of a (and b), out[r] += sum_b w_b Re[conj(a) b] --------------------------
// 32 lines per CTA and a share of the bands (blockIdx.y); the sums stay in shared memory until the
// end and are added to the permuted grid atomically.  The products are integers too: one conversion
// and one FMA per point are left to the FP64 pipe, which was the bound with FP64 products.  Each
// value is shifted up to 2^62 by its own leading zeros first, so that a product keeps 2^-58 of
// itself: where a band has died away the density is as close as the transform left the band, not
// one unit of the line's largest product.
template <bool BIG>
__global__ void __launch_bounds__(kThreads, BIG ? 2 : 3) k_fx_dens(const double2* __restrict__ hba,
                                                         const double2* __restrict__ hbb, int64_t hb_bs, int nb,
                                                         int bper, const double* __restrict__ wgt, int np, int nyz,
                                                         Dim d, int bits, double* __restrict__ out_perm) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, n = d.n;
  fc* bufa = reinterpret_cast<fc*>(smem);
  fc* bufb = bufa + (hbb ? n * PT : 0);
  double* acc = reinterpret_cast<double*>(bufb + n * PT) + lane;  // [n][32]
  __shared__ unsigned red[2][kWarps][32];
  const int yz = blockIdx.x * 32 + lane;
  const bool live = yz < nyz;
  for (int e = w; e < n; e += kWarps) acc[e * 32] = 0.0;
  const int b_lo = blockIdx.y * bper, b_hi = min(nb, b_lo + bper);
#pragma unroll 1
  for (int b = b_lo; b < b_hi; ++b) {
    int ka = 0, kb = 0;  // exponents of a and b; kNan
#pragma unroll 1
    for (int which = 0; which < (hbb ? 2 : 1); ++which) {
      const double2* pl = (which ? hbb : hba) + (int64_t)b * hb_bs + (live ? yz : 0);
      fc* col = (which ? bufb : bufa) + lane;
      unsigned mx = 0;
#pragma unroll 4
      for (int p = w; p < np; p += kWarps) {
        const double2 v = live ? pl[(int64_t)p * nyz] : make_double2(0.0, 0.0);
        mx = track(mx, v);
        *reinterpret_cast<double2*>(&col[p * PT]) = v;
      }
      mx = line_max(mx, red[which]);
      const int E = top_exp(mx);
      const In in(E, bits);
      (which ? kb : ka) = out_exp(mx, E - bits + 2);
#define FX_F(R)                                              \
  _Pragma("unroll 1") for (int J = w; J < d.r2; J += kWarps) \
      inv1<R>(col, J, d, in, [&](int e) { return e < np; })
      FX_SWITCH(d.r1, FX_F)
#undef FX_F
    }
    __syncthreads();
    if (!hbb) kb = ka;
    const bool bad = ka == kNan || kb == kNan;
    const int kab = bad ? 0 : ka + kb + 64;
    const double wb = bad ? __longlong_as_double(0x7ff8000000000000ll) : wgt[b];
    // the last stage of a (and b); with b, a's values go back to its line
#define FX_F(R)                                                                   \
  _Pragma("unroll 1") for (int blk = w; blk < d.r1; blk += kWarps) {              \
    fc y[R];                                                                      \
    if (hbb) {                                                                    \
      fc* ca = bufa + lane + blk * R * PT;                                        \
      _Pragma("unroll") for (int m = 0; m < R; ++m) y[m] = ca[m * PT];            \
      dft<+1, R>(y);                                                              \
      _Pragma("unroll") for (int m = 0; m < R; ++m) ca[m * PT] = y[m];                  \
    }                                                                             \
    const fc* cb = bufb + lane + blk * R * PT;                                    \
    _Pragma("unroll") for (int m = 0; m < R; ++m) y[m] = cb[m * PT];              \
    dft<+1, R>(y);                                                                \
    _Pragma("unroll") for (int m = 0; m < R; ++m) {                               \
      const int tb = up_shift(y[m]);                                              \
      const fc vb = {y[m].x << tb, y[m].y << tb};                                 \
      int ta = tb;                                                                \
      fc va = vb;                                                                 \
      if (hbb) {                                                                  \
        va = bufa[lane + (blk * R + m) * PT];                                     \
        ta = up_shift(va);                                                        \
        va = {va.x << ta, va.y << ta};                                            \
      }                                                                           \
      double* s = &acc[(blk * R + m) * 32];                                       \
      *s = fma(wb, Out{kab - ta - tb}(dot64(va, vb)), *s);                        \
    }                                                                             \
  }
    FX_SWITCH(d.r2, FX_F)
#undef FX_F
    __syncthreads();  // the next band's planes overwrite the lines
  }
  if (live && b_hi > b_lo)
    for (int r = w; r < d.r1; r += kWarps)
      for (int e = r * d.r2; e < (r + 1) * d.r2; ++e) atomicAdd(&out_perm[(int64_t)e * nyz + yz], acc[e * 32]);
}

// ---- host -------------------------------------------------------------------------------
std::vector<Tw> twiddles(int L) {
  // angle 2 pi k / L: octant 8 k / L, remainder r / L of pi / 4 (mirrored in odd octants), so the
  // long double functions (software on some hosts) run once per remainder and below pi / 4 only
  const long long one = 1ll << 62;
  std::vector<long long> c(L + 1), s(L + 1);
  std::vector<char> have(L + 1, 0);
  auto halves = [](long long v, int& lo, int& hi) {
    if ((int)(unsigned)(v & 0xffffffffll) == INT32_MIN) v += 1;  // keep -lo representable
    lo = (int)(unsigned)(v & 0xffffffffll);
    hi = (int)((v - lo) >> 32);
  };
  std::vector<Tw> t(L);
  for (int k = 0; k < L; ++k) {
    const int o = (int)(8ll * k / L), r0 = (int)(8ll * k - (long long)o * L), r = (o & 1) ? L - r0 : r0;
    if (!have[r]) {
      const long double a = 0.78539816339744830961566084581987572L * (long double)r / (long double)L;
      c[r] = llroundl(cosl(a) * (long double)one);
      s[r] = llroundl(sinl(a) * (long double)one);
      have[r] = 1;
    }
    // cos and sin of pi / 4 o' + a (o odd: pi / 4 (o + 1) - a)
    const long long C = c[r], Sn = s[r];
    long long x, y;
    switch (o) {
      case 0: x = C; y = Sn; break;
      case 1: x = Sn; y = C; break;
      case 2: x = -Sn; y = C; break;
      case 3: x = -C; y = Sn; break;
      case 4: x = -C; y = -Sn; break;
      case 5: x = -Sn; y = -C; break;
      case 6: x = Sn; y = -C; break;
      default: x = C; y = -Sn; break;
    }
    halves(x, t[k].xlo, t[k].xhi);
    halves(-y, t[k].ylo, t[k].yhi);  // exp(-i angle)
  }
  return t;
}

bool covers(const FftPlan& plan) {
  for (int i = 0; i < 3; ++i)
    if (plan.d[i].nst != 2 || plan.n[i] > 256) return false;
  return true;
}

static bool big(const Dim& d) { return std::max(d.r1, d.r2) > 12; }

static Dim dim_of(const FftPlan& plan, const double2* tw, int i) {
  const FftDim& f = plan.d[i];
  return {f.n, f.radix[0], f.radix[1], reinterpret_cast<const Tw*>(tw + plan.tw_total) + f.tw_off[0]};
}

// Largest B (see the top of the file).  log2 bounds of a value's modulus with inputs of 2^(B + 1/2):
// before the twiddles of an inverse (forward) transform R1 (R2) times that, after the whole
// transform n / 4 times that.
static int bits_line(const Dim& d) {
  double over = 0.0;
  over = std::max(over, 57.5 + log2((double)std::max(d.r1, d.r2)) - 61.6);
  over = std::max(over, 57.5 + log2((double)d.n) - 2.0 - 62.4);
  return 57 - (int)ceil(over);
}
// The x pass: `np` non-zero inputs.  Its forward half starts from the line times |v| <= 1, of
// 2-norm at most sqrt(n np) times an input, so a sum of R2 of its values is at most sqrt(R2 n np)
// and the whole transform n sqrt(np) times an input (divided by 4 in each twiddle product and
// in the product with V).
static int bits_x(const Dim& d, int np) {
  double over = 57.0 - bits_line(d);
  const double q = 0.5 * log2((double)np);
  over = std::max(over, 57.5 + 0.5 * log2((double)d.r2 * d.n) + q - 4.0 - 61.6);
  over = std::max(over, 57.5 + log2((double)d.n) + q - 6.0 - 62.4);
  return 57 - (int)ceil(over);
}

// Leading zeros of ss = (2-norm / 2^32)^2 below which the forward half has no room: with a 2-norm
// of 2^x, x = (64 - clz(ss)) / 2 + 32, and a shift by t, the line times V has at most
// sqrt(n) 2^(x - 4 + t), a sum of R2 of its values sqrt(R2) times that (<= 2^61.6), the transform
// sqrt(n) / 4 times that (<= 2^62.4); the shifted values themselves, at most sqrt(np) 2^(x - 2 + t),
// stay below 2^62.4.
static int room_x(const Dim& d, int np) {
  double x = 61.6 + 4.0 - 0.5 * log2((double)d.r2 * d.n);
  x = std::min(x, 62.4 + 6.0 - log2((double)d.n));
  x = std::min(x, 62.4 + 2.0 - 0.5 * log2((double)np));
  return (int)ceil(64.0 - 2.0 * (x - 32.0));
}

cudaError_t local_apply(const FftPlan& plan, const double2* tw, const SphereDev& sp, const double* vperm,
                        const double* kin, const double2* psi, int64_t ldpsi, int nband, double2* out, int64_t ldout,
                        double2* hb, int band_batch, cudaStream_t st, ::pw_ctx* prof) {
  if (nband <= 0) return cudaSuccess;
  const Dim dx = dim_of(plan, tw, 0), dy = dim_of(plan, tw, 1), dz = dim_of(plan, tw, 2);
  const int nyz = dy.n * dz.n, nc = (dz.n + 31) / 32, gz = (sp.nrow + 31) / 32, gx = (nyz + 31) / 32;
  const int64_t hb_bs = (int64_t)sp.nplane * nyz;
  const size_t line = sizeof(fc) * PT;
  const size_t smz = line * dz.n, smy = line * dy.n + sizeof(int) * dy.n, smx = line * dx.n;
  cudaError_t e;
  if ((e = smem_limit(big(dz) ? k_fx_zinv<true> : k_fx_zinv<false>, smz, kDynSmem)) || (e = smem_limit(big(dz) ? k_fx_zfwd<true> : k_fx_zfwd<false>, smz, kDynSmem)) ||
      (e = smem_limit(big(dy) ? k_fx_yinv<true> : k_fx_yinv<false>, smy, kDynSmem)) || (e = smem_limit(big(dy) ? k_fx_yfwd<true> : k_fx_yfwd<false>, smy, kDynSmem)) ||
      (e = smem_limit(big(dx) ? k_fx_x<true> : k_fx_x<false>, smx, kDynSmem)))
    return e;
  const int bz = bits_line(dz), by = bits_line(dy), bx = bits_x(dx, sp.nplane), rx = room_x(dx, sp.nplane);
  for (int b0 = 0; b0 < nband; b0 += band_batch) {
    const int nb = std::min(band_batch, nband - b0);
    prof_begin(prof, PW_PROF_PLANE_INV);
    (big(dz) ? k_fx_zinv<true> : k_fx_zinv<false>)<<<dim3(gz, nb), kThreads, smz, st>>>(psi + b0 * ldpsi, ldpsi, hb, hb_bs, sp, dz, dy.n, bz); count_launch();
    (big(dy) ? k_fx_yinv<true> : k_fx_yinv<false>)<<<dim3(sp.nplane * nc, nb), kThreads, smy, st>>>(hb, hb_bs, sp, dy, dz.n, nc, by); count_launch();
    prof_end(prof, PW_PROF_PLANE_INV);
    prof_begin(prof, PW_PROF_XLINE);
    // a few waves of CTAs; each finds the scale of V on its lines once for its bands
    int splits = std::max(1, std::min(nb, (152 * 2 * 4 + gx - 1) / gx));
    const int bper = (nb + splits - 1) / splits;
    splits = (nb + bper - 1) / bper;
    (big(dx) ? k_fx_x<true> : k_fx_x<false>)<<<dim3(gx, splits), kThreads, smx, st>>>(hb, hb_bs, nb, bper, vperm, sp.nplane, nyz, dx, bx, rx); count_launch();
    prof_end(prof, PW_PROF_XLINE);
    prof_begin(prof, PW_PROF_PLANE_FWD);
    (big(dy) ? k_fx_yfwd<true> : k_fx_yfwd<false>)<<<dim3(sp.nplane * nc, nb), kThreads, smy, st>>>(hb, hb_bs, sp, dy, dz.n, nc, by); count_launch();
    (big(dz) ? k_fx_zfwd<true> : k_fx_zfwd<false>)<<<dim3(gz, nb), kThreads, smz, st>>>(hb, hb_bs, sp, dz, dy.n, bz, kin, psi + b0 * ldpsi, ldpsi,
                                                  out + b0 * ldout, ldout); count_launch();
    prof_end(prof, PW_PROF_PLANE_FWD);
  }
  return cudaGetLastError();
}

cudaError_t density(const FftPlan& plan, const double2* tw, const SphereDev& sp, const double2* a, const double2* b,
                    int64_t ld, int nband, const double* w_dev, double* out_perm, double2* hb, int band_batch,
                    cudaStream_t st) {
  if (nband <= 0) return cudaSuccess;
  const Dim dx = dim_of(plan, tw, 0), dy = dim_of(plan, tw, 1), dz = dim_of(plan, tw, 2);
  const int nyz = dy.n * dz.n, nc = (dz.n + 31) / 32, gz = (sp.nrow + 31) / 32, gx = (nyz + 31) / 32;
  const int64_t hb_bs = (int64_t)sp.nplane * nyz;
  const size_t line = sizeof(fc) * PT;
  const size_t smz = line * dz.n, smy = line * dy.n + sizeof(int) * dy.n;
  const size_t smx = line * dx.n * (b ? 2 : 1) + sizeof(double) * 32 * dx.n;
  if (smx > 220 * 1024) return cudaErrorNotSupported;
  cudaError_t e;
  if ((e = smem_limit(big(dz) ? k_fx_zinv<true> : k_fx_zinv<false>, smz, kDynSmem)) || (e = smem_limit(big(dy) ? k_fx_yinv<true> : k_fx_yinv<false>, smy, kDynSmem)) ||
      (e = smem_limit(big(dx) ? k_fx_dens<true> : k_fx_dens<false>, smx, kDynSmem)))
    return e;
  const int bz = bits_line(dz), by = bits_line(dy), bx = bits_line(dx);
  double2* hbb = b ? hb + hb_bs * band_batch : nullptr;
  for (int b0 = 0; b0 < nband; b0 += band_batch) {
    const int nb = std::min(band_batch, nband - b0);
    for (int which = 0; which < (b ? 2 : 1); ++which) {
      double2* dst = which ? hbb : hb;
      (big(dz) ? k_fx_zinv<true> : k_fx_zinv<false>)<<<dim3(gz, nb), kThreads, smz, st>>>((which ? b : a) + b0 * ld, ld, dst, hb_bs, sp, dz, dy.n, bz); count_launch();
      (big(dy) ? k_fx_yinv<true> : k_fx_yinv<false>)<<<dim3(sp.nplane * nc, nb), kThreads, smy, st>>>(dst, hb_bs, sp, dy, dz.n, nc, by); count_launch();
    }
    // few splits of the bands: every split adds its lines to the grid once
    int splits = std::max(1, std::min(nb, (152 * 4 + gx - 1) / gx));
    const int bper = (nb + splits - 1) / splits;
    splits = (nb + bper - 1) / bper;
    (big(dx) ? k_fx_dens<true> : k_fx_dens<false>)<<<dim3(gx, splits), kThreads, smx, st>>>(hb, hbb, hb_bs, nb, bper, w_dev + b0, sp.nplane, nyz, dx, bx, out_perm); count_launch();
  }
  return cudaGetLastError();
}

}  // namespace fx
}  // namespace pw
