// Block-floating-point arithmetic on 64-bit integers: the binary64-class FFT
// passes on the integer pipes.
//
// GB300 issues 2 binary64 operations per clock and SM, 1/64 of its 32-bit
// rate, so an FFT in binary64 is bound by that pipe (88-93% busy before this
// form).  Here a CTA's tile of line elements (in H each line) shares one exponent e and each
// real number is a 64-bit integer X with value X 2^e, |X| < 2^63: 58 to 62
// significant bits of the tile's largest element against binary64's 53.  An
// addition is two 32-bit instructions, a product with a twiddle three
// 32 x 32 -> 64 multiply-adds (64 a clock and SM), so a transform costs about
// 1/8 of its binary64 time.
//
// Rounding.  Products, the stages' scalings and every shift that brings a tile to
// a transform's 2^59 (d2i, cshift, shr_rnd) round to nearest, to one unit of 2^-59
// of the tile's largest component.  Between passes an element is first brought to
// the largest exponent among its tile's inputs; that shift cuts off (shr_clamp), at
// 2^-62 of the largest component of the tile that the exponent comes from, and so
// does the sum of H's three parts, three bits below its result's unit.  (Rounding
// there too left the errors as they are and cost H 2%, P and the potential 1%.)
// Against 80 bits (random states at 144x48x18): H 1.9e-16, P 2.1e-16 of the 2-norm,
// where binary64 transforms had 2.6e-16 and 3.8e-16.
//
// Bounds.  A transform takes components below 2^59 (modulus below 2^59.5).
// Its first stage, of radix R <= 8, grows the modulus by R, and every later
// stage multiplies by twiddles scaled by 1/8 (radix 5, 6, 8) or 1/4 (radix 2,
// 3, 4) first, so the modulus stays below 2^62.5 throughout; the exponent
// grows by the same 3 or 2.  The partial sums of a product then stay below
// 2^63 (see tmul).
#pragma once

#include <cuda_runtime.h>

namespace atkm {

struct __align__(16) c64 {
  long long x, y;
};

// Exponent of a tile that holds a NaN or an infinity.
constexpr int kExpNaN = 0x40000000;

__device__ __forceinline__ c64 cz() { return c64{0, 0}; }
__device__ __forceinline__ c64 cadd(c64 a, c64 b) { return c64{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ c64 csub(c64 a, c64 b) { return c64{a.x - b.x, a.y - b.y}; }
// S i a
template <int S> __device__ __forceinline__ c64 cmuli(c64 a) {
  return S > 0 ? c64{-a.y, a.x} : c64{a.y, -a.x};
}
template <int K> __device__ __forceinline__ long long rsh(long long v) { return (v + (1ll << (K - 1))) >> K; }
template <int K> __device__ __forceinline__ c64 crsh(c64 v) { return c64{rsh<K>(v.x), rsh<K>(v.y)}; }

// v = h 2^32 + l with both limbs signed.
struct Limbs {
  int h, l;
};
__device__ __forceinline__ Limbs limbs(long long v) {
  const int l = (int)v;
  return Limbs{(int)(v >> 32) + (int)((unsigned)l >> 31), l};
}
__device__ __forceinline__ long long mulw(int a, int b) { return (long long)a * (long long)b; }

// a b / 2^64, rounded, for |a| < 2^62.9, |b| <= 2^61: the low limbs' product
// (below one unit of the result) is left out.
__device__ __forceinline__ long long mul64(Limbs a, Limbs b) {
  const long long c = 0x80000000ll + mulw(a.h, b.l) + mulw(a.l, b.h);
  return (long long)(int)(c >> 32) + mulw(a.h, b.h);
}

// a W / 2^64 for a twiddle W = c + S i s given as 64-bit limbs (c.h, c.l,
// s.h, s.l).  With |a| < 2^62.5 and |W| = 2^61 the cross sums stay below
// 2^62.4, with |W| = 2^62 below 2^62.8.
template <int S> __device__ __forceinline__ c64 tmul(c64 a, int4 w) {
  const Limbs x = limbs(a.x), y = limbs(a.y);
  const int ph = S < 0 ? w.z : -w.z, pl = S < 0 ? w.w : -w.w;  // re = x c + y p, im = y c - x p
  const long long cr = 0x80000000ll + mulw(x.h, w.y) + mulw(x.l, w.x) + mulw(y.h, pl) + mulw(y.l, ph);
  const long long ci = 0x80000000ll + mulw(y.h, w.y) + mulw(y.l, w.x) + mulw(x.h, -pl) + mulw(x.l, -ph);
  c64 r;
  r.x = (long long)(int)(cr >> 32) + mulw(x.h, w.x) + mulw(y.h, ph);
  r.y = (long long)(int)(ci >> 32) + mulw(y.h, w.x) + mulw(x.h, -ph);
  return r;
}

// a times a constant c = C / 2^64, |c| < 1/2, rounded.
template <long long C> __device__ __forceinline__ long long mulc(long long a) {
  constexpr int cl = (int)(unsigned)(unsigned long long)C;
  constexpr int ch = (int)((C - (long long)cl) / 4294967296ll);
  const Limbs x = limbs(a);
  const long long c = 0x80000000ll + mulw(x.h, cl) + mulw(x.l, ch);
  return (long long)(int)(c >> 32) + mulw(x.h, ch);
}
// The irrational factors of the small DFTs, as 64-bit fractions (rounded from
// their closed forms): sqrt(1/2) - 1, sin 60 - 1, cos 72 = (sqrt5 - 1) / 4,
// cos 144 + 1, sin 72 - 1, sin 144 - 1.
constexpr long long kRt12m1 = -5402926248376769404ll;
constexpr long long kS60m1 = -2471395088767036514ll;
constexpr long long kC72 = 5700357409661599243ll;
constexpr long long kC144p1 = 3523014627193176565ll;
constexpr long long kS72m1 = -902847917979075853ll;
constexpr long long kS144m1 = -7604019954369499282ll;

// In-register R-point DFT, X_q = sum_r v_r e^{S 2 pi i r q / R}.  ZU: the
// inputs of the upper half are zero.  LO: only the lower half of the outputs
// is formed.
template <int RAD, int S> struct IDft;
template <int S> struct IDft<2, S> {
  template <bool ZU, bool LO> static __device__ __forceinline__ void go(c64* v) {
    const c64 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    if (!LO) v[1] = csub(a, b);
  }
};
template <int S> struct IDft<4, S> {
  template <bool ZU, bool LO> static __device__ __forceinline__ void go(c64* v) {
    const c64 a = ZU ? v[0] : cadd(v[0], v[2]), b = ZU ? v[0] : csub(v[0], v[2]);
    const c64 c = ZU ? v[1] : cadd(v[1], v[3]), d = cmuli<S>(ZU ? v[1] : csub(v[1], v[3]));
    v[0] = cadd(a, c);
    v[1] = cadd(b, d);
    if (!LO) {
      v[2] = csub(a, c);
      v[3] = csub(b, d);
    }
  }
};
template <int S> struct IDft<8, S> {
  template <bool ZU, bool LO> static __device__ __forceinline__ void go(c64* v) {
    c64 e[4] = {v[0], v[2], v[4], v[6]};
    c64 o[4] = {v[1], v[3], v[5], v[7]};
    IDft<4, S>::template go<ZU, false>(e);
    IDft<4, S>::template go<ZU, false>(o);
    // o_q *= e^{S i pi q / 4}
    const long long a1 = o[1].x - S * o[1].y, b1 = o[1].y + S * o[1].x;
    const long long a3 = -(o[3].x + S * o[3].y), b3 = S * o[3].x - o[3].y;
    const c64 o1 = {a1 + mulc<kRt12m1>(a1), b1 + mulc<kRt12m1>(b1)};
    const c64 o2 = cmuli<S>(o[2]);
    const c64 o3 = {a3 + mulc<kRt12m1>(a3), b3 + mulc<kRt12m1>(b3)};
    v[0] = cadd(e[0], o[0]);
    v[1] = cadd(e[1], o1);
    v[2] = cadd(e[2], o2);
    v[3] = cadd(e[3], o3);
    if (!LO) {
      v[4] = csub(e[0], o[0]);
      v[5] = csub(e[1], o1);
      v[6] = csub(e[2], o2);
      v[7] = csub(e[3], o3);
    }
  }
};
template <int S> struct IDft<3, S> {
  template <bool ZU, bool LO> static __device__ __forceinline__ void go(c64* v) {
    const c64 t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const c64 m = csub(v[0], crsh<1>(t));
    const c64 u = cmuli<S>(c64{d.x + mulc<kS60m1>(d.x), d.y + mulc<kS60m1>(d.y)});
    v[0] = cadd(v[0], t);
    v[1] = cadd(m, u);
    v[2] = csub(m, u);
  }
};
template <int S> struct IDft<5, S> {
  template <bool ZU, bool LO> static __device__ __forceinline__ void go(c64* v) {
    const c64 a1 = cadd(v[1], v[4]), b1 = csub(v[1], v[4]);
    const c64 a2 = cadd(v[2], v[3]), b2 = csub(v[2], v[3]);
    const c64 z = v[0];
    // cos 72 a1 + cos 144 a2 and the other way round
    const c64 m1 = {z.x + mulc<kC72>(a1.x) + mulc<kC144p1>(a2.x) - a2.x,
                    z.y + mulc<kC72>(a1.y) + mulc<kC144p1>(a2.y) - a2.y};
    const c64 m2 = {z.x + mulc<kC72>(a2.x) + mulc<kC144p1>(a1.x) - a1.x,
                    z.y + mulc<kC72>(a2.y) + mulc<kC144p1>(a1.y) - a1.y};
    const c64 n1 = cmuli<S>(c64{b1.x + mulc<kS72m1>(b1.x) + b2.x + mulc<kS144m1>(b2.x),
                                b1.y + mulc<kS72m1>(b1.y) + b2.y + mulc<kS144m1>(b2.y)});
    const c64 n2 = cmuli<S>(c64{b1.x + mulc<kS144m1>(b1.x) - b2.x - mulc<kS72m1>(b2.x),
                                b1.y + mulc<kS144m1>(b1.y) - b2.y - mulc<kS72m1>(b2.y)});
    v[0] = cadd(z, cadd(a1, a2));
    v[1] = cadd(m1, n1);
    v[4] = csub(m1, n1);
    v[2] = cadd(m2, n2);
    v[3] = csub(m2, n2);
  }
};
// 6 = 2 x 3 with coprime factors: n = 3 n1 + 2 n2 (mod 6), q = 3 q1 + 4 q2
// (mod 6), no twiddles between the two layers.
template <int S> struct IDft<6, S> {
  template <bool ZU, bool LO> static __device__ __forceinline__ void go(c64* v) {
    c64 a[3] = {v[0], v[2], v[4]}, b[3] = {v[3], v[5], v[1]};
    IDft<3, S>::template go<false, false>(a);
    IDft<3, S>::template go<false, false>(b);
    v[0] = cadd(a[0], b[0]);
    v[3] = csub(a[0], b[0]);
    v[4] = cadd(a[1], b[1]);
    v[1] = csub(a[1], b[1]);
    v[2] = cadd(a[2], b[2]);
    v[5] = csub(a[2], b[2]);
  }
};
// Scale (a power of two) that a stage of radix R applies with its twiddles.
__host__ __device__ constexpr int stage_shift(int rad) { return rad > 4 ? 3 : 2; }

// The lengths that the engine k_imix is built for, radices in ascending order;
// n = 0: none.
#define ATKM_IMIX_LENGTHS(F) \
  F(16) F(32) F(64) F(128) F(256) F(18) F(20) F(24) F(30) F(36) F(40) F(48) F(60) F(72) F(80) F(90) F(96) F(100) F(108) F(120) F(144) F(150) F(160) F(180) \
  F(192) F(200) F(216) F(240) F(288) F(320) F(384)
struct RadList {
  int n;
  int r[3];
};
__host__ __device__ constexpr RadList int_radices(int L) {
  switch (L) {
    case 16: return {2, {4, 4, 0}};
    case 32: return {2, {4, 8, 0}};
    case 64: return {3, {4, 4, 4}};
    case 128: return {3, {4, 4, 8}};
    case 256: return {3, {4, 8, 8}};
    case 18: return {2, {3, 6, 0}};
    case 20: return {2, {4, 5, 0}};
    case 24: return {2, {4, 6, 0}};
    case 30: return {2, {5, 6, 0}};
    case 36: return {2, {6, 6, 0}};
    case 40: return {2, {5, 8, 0}};
    case 48: return {2, {6, 8, 0}};
    case 60: return {3, {3, 4, 5}};
    case 72: return {3, {3, 4, 6}};
    case 80: return {3, {4, 4, 5}};
    case 90: return {3, {3, 5, 6}};
    case 96: return {3, {4, 4, 6}};
    case 100: return {3, {4, 5, 5}};
    case 108: return {3, {3, 6, 6}};
    case 120: return {3, {4, 5, 6}};
    case 144: return {3, {4, 6, 6}};
    case 150: return {3, {5, 5, 6}};
    case 160: return {3, {4, 5, 8}};
    case 180: return {3, {5, 6, 6}};
    case 192: return {3, {4, 6, 8}};
    case 200: return {3, {5, 5, 8}};
    case 216: return {3, {6, 6, 6}};
    case 240: return {3, {5, 6, 8}};
    case 288: return {3, {6, 6, 8}};
    case 320: return {3, {5, 8, 8}};
    case 384: return {3, {6, 8, 8}};
    default: return {0, {0, 0, 0}};
  }
}
// Lines of a k_imix tile: a power of two (the tile exponents are found by
// shifts), at least 8 (128-byte rows of a column tile), about 320 threads.
__host__ __device__ constexpr int imix_tile(int L) {
  const int M = L / int_radices(L).r[0];
  int T = 8;
  while (2 * T * M <= 320 && T < 64) T *= 2;
  return T;
}

// ------------------------------------------------------------ conversions
// |hi word| of a component: its largest over a tile gives the tile's size.
__device__ __forceinline__ unsigned mag(long long v) {
  const int h = (int)(v >> 32);
  return (unsigned)(h ^ (h >> 31));
}
__device__ __forceinline__ unsigned mag(c64 v) { return max(mag(v.x), mag(v.y)); }
// bits b with |X| < 2^b, from the largest mag of a tile (32 when it is 0)
__device__ __forceinline__ int mag_bits(unsigned m) { return 64 - __clz((int)m); }

// v / 2^s rounded down, s >= 0 of any size
__device__ __forceinline__ long long shr_clamp(long long v, int s) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
  return r;
}
// v / 2^s rounded, 0 <= s <= 62 (the caller cuts s off there: beyond, a |v| below
// 2^62.5 leaves one unit at most)
__device__ __forceinline__ long long shr_rnd(long long v, int s) { return (v + ((1ll << s) >> 1)) >> s; }
// v 2^s, rounded when s < 0
__device__ __forceinline__ c64 cshift(c64 v, int s) {
  if (s >= 0) return c64{(long long)((unsigned long long)v.x << s), (long long)((unsigned long long)v.y << s)};
  const long long h = 1ll << (-s - 1);
  return c64{(v.x + h) >> -s, (v.y + h) >> -s};
}

// A finite double to an integer: the 53-bit mantissa with its leading bit at
// bit 63, shifted right by base - (biased exponent) >= 1 and rounded.  base > 65,
// so that zeros and subnormals (no implicit bit) shift out.
__device__ __forceinline__ long long d2i(double d, int base) {
  const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
  const int s = base - 1 - (int)((h >> 20) & 0x7ffu);
  const unsigned mh = __funnelshift_l(l, h, 11) | 0x80000000u, ml = l << 11;
  unsigned long long m = ((unsigned long long)mh << 32) | ml;
  asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(s));
  const long long v = (long long)((m + 1) >> 1);
  return (int)h < 0 ? -v : v;
}

// X 2^e to binary64, rounded to nearest; c = e + 1085 with 64 <= c <= 2045.
__device__ __forceinline__ double i2d(long long v, int c) {
  const long long a = v < 0 ? -v : v;
  const unsigned h = (unsigned)(a >> 32), l = (unsigned)a;
  const int n = __clz((int)(h ? h : l)) + (h ? -1 : 31);  // leading bit to bit 62
  long long t = (long long)((unsigned long long)a << n);
  t = (t + 0x200) >> 10;
  const int hi = (int)(t >> 32) + ((c - 1 - n) << 20);
  const int sg = (int)(v >> 32) & (int)0x80000000;
  return a == 0 ? 0.0 : __hiloint2double(hi | sg, (int)t);
}
// The same, rounded alike, for any exponent (overflow to infinity, gradual underflow).
static __device__ __noinline__ double i2d_any(long long v, int e) {
  if (e >= kExpNaN / 2) return __longlong_as_double(0x7ff8000000000000ll);
  const long long a = v < 0 ? -v : v;
  const long long h = a >> 53 ? 1ll << (10 - __clzll(a)) : 0;  // half a unit in the last of 53 bits (a < 2^63)
  const long long r = (a + h) & -(h ? 2 * h : 1ll);
  return scalbn(__ll2double_rn(v < 0 ? -r : r), e);
}
__device__ __forceinline__ bool i2d_ok(int e) { return (unsigned)(e + 1085 - 64) <= 2045u - 64u; }

// 2^e as binary64 (0 or infinity outside its range)
__device__ __forceinline__ double pow2d(int e) {
  return e < -1022 ? 0.0 : (e > 1023 ? __longlong_as_double(0x7ff0000000000000ll) : __hiloint2double((e + 1023) << 20, 0));
}

}  // namespace atkm
