// Register FFT of the double path in 64-bit fixed point.
//
// GB300 issues about two FP64 operations per clock and SM, and integer ones at dozens of
// times that rate (measured: 1.7 double FMAs per clock and SM, so 0.43 complex products,
// against 1.8 fixed-point complex products; 64-bit additions 20 times faster).  A
// transform is additions and products with unit-modulus constants, so every value on
// the way is bounded by the sum of the inputs' moduli: with one power-of-two scale per
// transform, taken from that sum (block floating point), 64-bit integers hold it without
// overflow, with 62 bits below the bound where a double has 53 below each value.
//
// A value is v 2^(E - 62), v the integer, E the stage's exponent.  With S the sum of the
// moduli of the inputs and M their maximum, a value after s stages is at most min(S, G M),
// G the product of the stages' radices, and E is the smallest exponent of that bound
// (l1_exponent, stage_exponent): moduli are at most 2^62 all the way, inside the butterflies
// too (every intermediate is a sum of distinct inputs with unit weights), and a component
// of a value turned by pi/4 at most 2^62.5.  The scale that grows with the stages matters: with the final one
// throughout, the first stages round at 2^-62 S where a double rounds at 2^-53 of each
// value, and white input of L = 1024 came out with more error than in double (N = 512,
// 3.5e-16 against 3.1e-16; now 1.0e-16).
//
// Twiddles are 62-bit: w = W 2^-62, W split into balanced halves W = wh 2^32 + wl with wl
// signed, so that a product is three signed 32 x 32 + 64 multiply-adds per real product:
//   v W 2^-62 = (vh wh 2^64 + (vh wl + vl wh) 2^32 + vl wl) 2^-62,
// the last term (below one unit) dropped, the sum rounded once per complex component.
// The stages, exchanges and order are those of fft_reg.cuh.
#pragma once

#include "fft_reg.cuh"

namespace bem {
namespace fx {

typedef long long i64;
struct __align__(16) I2 { i64 x, y; };
// exponents of transforms that hold nothing, or a value that is not finite
constexpr int kZeroExp = -(1 << 28), kNanExp = 1 << 28;
__device__ __forceinline__ bool is_nan_exp(int e) { return e >= kNanExp / 2; }

__device__ __forceinline__ i64 madw(int a, int b, i64 c) { return (i64)a * b + c; }
// balanced halves of v: v = h 2^32 + l, l signed
__device__ __forceinline__ void halves(i64 v, int& h, int& l) {
  l = (int)v;
  h = (int)(v >> 32) + (int)((unsigned)l >> 31);
}
// (V 2^32 + low word of t) 2^-30, V = V0 + (t >> 32)
__device__ __forceinline__ i64 join(i64 V, i64 t) {
  const unsigned tl = (unsigned)t, vl = (unsigned)V, vh = (unsigned)((unsigned long long)V >> 32);
  const unsigned lo = __funnelshift_l(tl, vl, 2), hi = __funnelshift_l(vl, vh, 2);
  return (i64)(((unsigned long long)hi << 32) | lo);
}
// v 2^-n (n > 0), rounded to nearest with ties to even.  Ties are common at small n, and a
// tie rounded up is a bias of a quarter of the last place that all values share: it adds
// up in the zero wave number, the one that the compliance weights most (white input,
// N = 512: error 7.0e-16 with ties up).
__device__ __forceinline__ i64 rshift(i64 v, int n) { return (v + ((1ll << (n - 1)) - 1) + ((v >> n) & 1)) >> n; }
// (a + b) / 2, the same way, without the sum (which may need 65 bits)
__device__ __forceinline__ i64 mean(i64 a, i64 b) {
  const i64 m = (a >> 1) + (b >> 1) + (a & b & 1);
  return m + (m & (a ^ b) & 1);
}
// v 2^d, rounded
__device__ __forceinline__ i64 shift(i64 v, int d) {
  return d >= 0 ? (i64)((unsigned long long)v << min(d, 63)) : rshift(v, min(-d, 63));
}
constexpr i64 kHalf = 1ll << 29;   // rounds the 2^-30 of join

// v W 2^-62 for a real factor (wh, wl)
__device__ __forceinline__ i64 mulr(i64 v, int wh, int wl) {
  int h, l;
  halves(v, h, l);
  const i64 t = madw(l, wh, madw(h, wl, kHalf));
  return join(madw(h, wh, t >> 32), t);
}
// a w (forward) or a conj(w) (inverse), |a| <= 2^62: by the Cauchy-Schwarz inequality the
// middle products add up to at most 2 2^61.5 < 2^63; w = (re h, re l, im h, im l)
template <bool INV>
__device__ __forceinline__ I2 twmul(I2 a, int4 w) {
  int xh, xl, yh, yl;
  halves(a.x, xh, xl);
  halves(a.y, yh, yl);
  const int ih = INV ? -w.z : w.z, il = INV ? -w.w : w.w;      // imaginary part used
  const int nh = INV ? w.z : -w.z, nl = INV ? w.w : -w.w;      // its negative (no half is -2^31)
  const i64 t = madw(xl, w.x, madw(xh, w.y, madw(yl, nh, madw(yh, nl, kHalf))));
  const i64 u = madw(xl, ih, madw(xh, il, madw(yl, w.x, madw(yh, w.y, kHalf))));
  return I2{join(madw(xh, w.x, madw(yh, nh, t >> 32)), t), join(madw(xh, ih, madw(yh, w.x, u >> 32)), u)};
}

__device__ __forceinline__ I2 cadd(I2 a, I2 b) { return I2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ I2 csub(I2 a, I2 b) { return I2{a.x - b.x, a.y - b.y}; }
template <bool INV>
__device__ __forceinline__ I2 rot4(I2 a) {
  return INV ? I2{-a.y, a.x} : I2{a.y, -a.x};
}
// 2^62 cos(pi/4) in balanced halves
constexpr int kR2h = 0x2d413ccd, kR2l = (int)0xfe779921;
template <bool INV>
__device__ __forceinline__ I2 rot8(I2 a) {
  return INV ? I2{mulr(a.x - a.y, kR2h, kR2l), mulr(a.x + a.y, kR2h, kR2l)}
             : I2{mulr(a.x + a.y, kR2h, kR2l), mulr(a.y - a.x, kR2h, kR2l)};
}
template <bool INV>
__device__ __forceinline__ I2 rot8_3(I2 a) {
  return INV ? I2{-mulr(a.x + a.y, kR2h, kR2l), mulr(a.x - a.y, kR2h, kR2l)}
             : I2{mulr(a.y - a.x, kR2h, kR2l), -mulr(a.x + a.y, kR2h, kR2l)};
}

template <bool INV, bool Z2>
__device__ __forceinline__ void dft4z(I2& v0, I2& v1, I2& v2, I2& v3) {
  if (Z2) {
    const I2 a = v0, dm = rot4<INV>(v1);
    v0 = cadd(a, v1);
    v2 = csub(a, v1);
    v1 = cadd(a, dm);
    v3 = csub(a, dm);
  } else {
    const I2 a = cadd(v0, v2), b = csub(v0, v2), c = cadd(v1, v3), dm = rot4<INV>(csub(v1, v3));
    v0 = cadd(a, c);
    v2 = csub(a, c);
    v1 = cadd(b, dm);
    v3 = csub(b, dm);
  }
}
// 8-point DFT as in fft_reg.cuh; HALF: inputs 4..7 are zero
template <bool INV, bool HALF>
__device__ __forceinline__ void dft8(I2* v) {
  dft4z<INV, HALF>(v[0], v[2], v[4], v[6]);
  dft4z<INV, HALF>(v[1], v[3], v[5], v[7]);
  v[3] = rot8<INV>(v[3]);
  v[5] = rot4<INV>(v[5]);
  v[7] = rot8_3<INV>(v[7]);
  I2 o[8];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    o[q] = cadd(v[2 * q], v[2 * q + 1]);
    o[q + 4] = csub(v[2 * q], v[2 * q + 1]);
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = o[q];
}
template <int Q, bool INV, bool HALF>
__device__ __forceinline__ void dftq(I2* v) {
  if constexpr (Q == 2) {
    const I2 a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
  }
  if constexpr (Q == 4) dft4z<INV, HALF>(v[0], v[1], v[2], v[3]);
  if constexpr (Q == 8) dft8<INV, HALF>(v);
}

// x(r) *= w_r (conjugated for INV), r = 1 .. Q-1: plane r - 1 of the stage's table, ns
// records per plane
template <int Q, bool INV, typename X>
__device__ __forceinline__ void apply_twiddles_fix(const int4* tws, int ns, int k, X&& x) {
#pragma unroll
  for (int r = 1; r < Q; ++r) x(r) = twmul<INV>(x(r), tws[(r - 1) * ns + k]);
}
// offset (records) of the planes of stage s of a length-2^LOGL plan of radix 8
template <int LOGL>
__host__ __device__ constexpr int tw_offset(int s) {
  using P = Plan<LOGL, 3>;
  int off = 0, ns = 1;
  for (int i = 0; i < s; ++i) {
    if (i > 0) off += (P::radix(i) - 1) * ns;
    ns *= P::radix(i);
  }
  return off;
}

// Exponents of a transform's bounds: every input modulus below 2^max, their sum below 2^sum
struct Bound { int max, sum; };
// exponent of the values after stages 0 .. s (HALF: half of stage 0's inputs are zero)
template <int LOGL, bool HALF>
__device__ __forceinline__ int stage_exponent(Bound b, int s) {
  using P = Plan<LOGL, 3>;
  const int g = (s < P::SR ? 3 * (s + 1) : 3 * P::SR + P::LOGRL) - (HALF ? 1 : 0);
  return s + 1 < P::NSTAGES ? min(b.sum, b.max + g) : b.sum;
}

// Full transform on the thread's registers v[q] = x[t + T q] -> X[t + T q] (see reg_fft);
// x at the exponent of stage 0, X at b.sum.
template <int LOGL, bool INV, bool HALF, int PER_BLOCK>
__device__ __forceinline__ void fix_fft(I2* v, Bound b, I2* sh, const int4* __restrict__ tw, int t, int group) {
  using P = Plan<LOGL, 3>;
  constexpr int R = P::R, TT = P::T, RL = P::RL;
  int ns = 1;
#pragma unroll
  for (int s = 0; s < P::NSTAGES; ++s) {
    const bool small = (s == P::SR);
    if (s > 0) {
      // to this stage's exponent (later stages reach the final one: nothing to shift)
      const int d = stage_exponent<LOGL, HALF>(b, s) - stage_exponent<LOGL, HALF>(b, s - 1);
      if (d > 0) {
        const int n = min(d, 63);
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = I2{rshift(v[q].x, n), rshift(v[q].y, n)};
      }
      const int4* tws = opaque(tw + tw_offset<LOGL>(s));
      if (!small) {
        apply_twiddles_fix<R, INV>(tws, ns, t & (ns - 1), [&](int r) -> I2& { return v[r]; });
      } else {
#pragma unroll
        for (int c = 0; c < R / RL; ++c)
          apply_twiddles_fix<RL, INV>(tws, ns, (t + TT * c) & (ns - 1),
                                      [&](int r) -> I2& { return v[c + r * (R / RL)]; });
      }
    }
    if (!small) {
      if (s == 0 && HALF) dftq<R, INV, true>(v);
      else dftq<R, INV, false>(v);
    } else {
#pragma unroll
      for (int c = 0; c < R / RL; ++c) {
        I2 w[RL > 1 ? RL : 2];
#pragma unroll
        for (int r = 0; r < RL; ++r) w[r] = v[c + r * (R / RL)];
        dftq<RL, INV, false>(w);
#pragma unroll
        for (int r = 0; r < RL; ++r) v[c + r * (R / RL)] = w[r];
      }
    }
    if (s + 1 < P::NSTAGES) {
      const int base = (t / ns) * ns * R + (t & (ns - 1));
#pragma unroll
      for (int r = 0; r < R; ++r) sh[padi<3>(base + r * ns)] = v[r];
      GroupSync<TT, PER_BLOCK>::sync(group);
#pragma unroll
      for (int q = 0; q < R; ++q) v[q] = sh[padi<3>(t + TT * q)];
      GroupSync<TT, PER_BLOCK>::sync(group);
    }
    ns *= small ? RL : R;
  }
}

// --- scales -------------------------------------------------------------------
// the modulus of v in units of 2^32, rounded up
__device__ __forceinline__ unsigned mag(I2 v) {
  return (unsigned)(abs((int)(v.x >> 32)) + abs((int)(v.y >> 32)) + 2);
}
__device__ __forceinline__ bool nonzero(I2 v) { return (v.x | v.y) != 0; }

// Maximum and sum over the threads of one transform (TT of them, PER_BLOCK per block);
// sh: TT / 32 words of the group
template <int TT, int PER_BLOCK, typename F>
__device__ __forceinline__ int group_all(int v, int* sh, int t, int group, F&& f) {
  constexpr int W = TT < 32 ? TT : 32;
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) v = f(v, __shfl_xor_sync(0xffffffffu, v, o, W));
  if constexpr (TT > 32) {
    GroupSync<TT, PER_BLOCK>::sync(group);   // earlier readers are done
    if ((t & 31) == 0) sh[t >> 5] = v;
    GroupSync<TT, PER_BLOCK>::sync(group);
    v = sh[0];
#pragma unroll
    for (int w = 1; w < TT / 32; ++w) v = f(v, sh[w]);
  }
  return v;
}

// Exponents of the largest term a_i 2^(e_i) and of the sum over the transform's terms (NT
// per thread, at most 4096 in all, a_i < 2^31, terms with a_i = 0 absent).  The terms are
// rounded up to 2^-18 of the largest, so the sum's is at most one above the exact one.
template <int TT, int PER_BLOCK, int NT>
__device__ __forceinline__ Bound l1_exponent(const unsigned (&a)[NT], const int (&e)[NT], int* sh, int t, int group) {
  constexpr int Q = 18;
  int top = kZeroExp;
#pragma unroll
  for (int i = 0; i < NT; ++i)
    if (a[i] != 0u) top = max(top, e[i] + 32 - __clz((int)a[i]));
  top = group_all<TT, PER_BLOCK>(top, sh, t, group, [](int x, int y) { return max(x, y); });
  int s = 0;
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const int d = Q - (top - e[i]);
    if (a[i] != 0u) s += d >= 0 ? (int)(a[i] << min(d, 31)) : (int)(a[i] >> min(-d, 31)) + 1;
  }
  s = group_all<TT, PER_BLOCK>(s, sh, t, group, [](int x, int y) { return x + y; });
  if (top == kZeroExp) return Bound{kZeroExp, kZeroExp};
  return Bound{top, top - Q + 32 - __clz(s)};
}

// --- conversions --------------------------------------------------------------
// |x| as a term of l1_exponent: top 21 bits of the significand and its exponent
__device__ __forceinline__ void term_of(double x, unsigned& a, int& e) {
  const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu, lo = (unsigned)__double2loint(x);
  const int f = (int)(hi >> 20);
  a = (hi & 0xfffffu) | (f != 0 ? 0x100000u : 0u);
  if (lo != 0u) a += 1u;            // the bits below, rounded up
  e = (f != 0 ? f : 1) - 1043;      // x = a 2^e
  if (f == 2047) { a = 1u; e = kNanExp; }
}
// x 2^(62 - E) as an integer (|x| < 2^E)
__device__ __forceinline__ i64 to_fix(double x, int E) {
  const unsigned hi = (unsigned)__double2hiint(x);
  const int f = (int)((hi >> 20) & 0x7ffu);
  const i64 m = ((i64)((hi & 0xfffffu) | (f != 0 ? 0x100000u : 0u)) << 32) | (unsigned)__double2loint(x);
  const i64 v = shift(m, (f != 0 ? f : 1) - 1075 + 62 - E);
  return (int)hi < 0 ? -v : v;
}
__device__ __forceinline__ double pow2(int k) {   // k in [-1022, 1023]
  return __hiloint2double((k + 1023) << 20, 0);
}
// v 2^(E - 62) as a double, in two steps so that neither factor leaves the range
__device__ __forceinline__ double from_fix(i64 v, int E) {
  const int k = max(min(E - 62, 2044), -2044), a = k / 2;
  return (double)v * pow2(a) * pow2(k - a);
}

// e^{-2 pi i num / den} (den a power of two) as a twiddle record, from Taylor sums in
// double-double arithmetic over the first octant (106 bits; 62 are kept)
struct DD { double h, l; };
__device__ __forceinline__ DD dd_add(DD a, DD b) {
  const double s = a.h + b.h, v = s - a.h;
  const double e = (a.h - (s - v)) + (b.h - v) + a.l + b.l;
  const double h = s + e;
  return DD{h, e - (h - s)};
}
__device__ __forceinline__ DD dd_mul(DD a, DD b) {
  const double p = a.h * b.h;
  const double e = fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h);
  const double h = p + e;
  return DD{h, e - (h - p)};
}
// (-1)^k / (2k)! and (-1)^k / (2k + 1)!: the Taylor coefficients of cos and of sin(x)/x in x^2
static __constant__ double c_cos[12][2] = {
    {1.0, 0.0}, {-0.5, 0.0}, {0.041666666666666664, 2.3129646346357427e-18}, {-0.001388888888888889,
    5.300543954373577e-20}, {2.48015873015873e-05, 2.1511947866775882e-23}, {-2.755731922398589e-07,
    -2.3767714622250297e-23}, {2.08767569878681e-09, -1.20734505911326e-25}, {-1.1470745597729725e-11,
    -2.0655512752830745e-28}, {4.779477332387385e-14, 4.399205485834081e-31}, {-1.5619206968586225e-16,
    -1.1910679660273754e-32}, {4.110317623312165e-19, 1.4412973378659527e-36}, {-8.896791392450574e-22,
    7.911402614872376e-38}};
static __constant__ double c_sin[12][2] = {
    {1.0, 0.0}, {-0.16666666666666666, -9.25185853854297e-18}, {0.008333333333333333, 1.1564823173178714e-19},
    {-0.0001984126984126984, -1.7209558293420705e-22}, {2.7557319223985893e-06, -1.858393274046472e-22},
    {-2.505210838544172e-08, 1.448814070935912e-24}, {1.6059043836821613e-10, 1.2585294588752098e-26},
    {-7.647163731819816e-13, -7.03872877733453e-30}, {2.8114572543455206e-15, 1.6508842730861433e-31},
    {-8.22063524662433e-18, -2.2141894119604265e-34}, {1.9572941063391263e-20, -1.3643503830087908e-36},
    {-3.868170170630684e-23, 8.843177655482344e-40}};
__device__ __forceinline__ i64 dd_fix(DD v) {   // v 2^62, rounded
  const double s = 4611686018427387904.0;
  const i64 a = __double2ll_rn(v.h * s);
  return a + __double2ll_rn((v.h * s - (double)a) + v.l * s);
}
__device__ inline int4 fix_twiddle(int num, int den) {
  num &= den - 1;
  const int oct = (int)(((i64)num * 8) / den);
  // angle 2 pi (num / den) = oct pi/4 + r, r in [0, pi/4); odd octants are mirrored
  i64 rn = (i64)num * 8 - (i64)oct * den;           // r = rn / den * pi / 4
  if (oct & 1) rn = den - rn;
  const DD pi4 = DD{0.78539816339744830962, 3.0616169978683829431e-17};
  const DD x = dd_mul(DD{(double)rn / (double)den, 0.0}, pi4), x2 = dd_mul(x, x);
  // (the terms from x^12 / 12! on, 1e-10, in plain double)
  double ch = c_cos[11][0], sh = c_sin[11][0];
#pragma unroll
  for (int k = 10; k >= 6; --k) {
    ch = fma(ch, x2.h, c_cos[k][0]);
    sh = fma(sh, x2.h, c_sin[k][0]);
  }
  DD c = DD{ch, 0.0}, s = DD{sh, 0.0};
#pragma unroll 1
  for (int k = 5; k >= 0; --k) {
    c = dd_add(dd_mul(c, x2), DD{c_cos[k][0], c_cos[k][1]});
    s = dd_add(dd_mul(s, x2), DD{c_sin[k][0], c_sin[k][1]});
  }
  s = dd_mul(s, x);
  i64 C = dd_fix(c), S = dd_fix(s);
  const int q = (oct + 1) >> 1;                     // quarter turns added to +-r
  if (oct & 1) S = -S;
  // cos, sin of q pi/2 + (signed r)
  i64 re, im;
  switch (q & 3) {
    case 0: re = C; im = S; break;
    case 1: re = -S; im = C; break;
    case 2: re = -C; im = -S; break;
    default: re = S; im = -C; break;
  }
  im = -im;                                          // e^{-i angle}
  int4 w;
  w.y = (int)re;
  w.x = (int)((re - w.y) >> 32);
  w.w = (int)im;
  if (w.w == (int)0x80000000) { im += 1; w.w = (int)im; }   // its negative must exist
  w.z = (int)((im - w.w) >> 32);
  return w;
}

}  // namespace fx
}  // namespace bem
