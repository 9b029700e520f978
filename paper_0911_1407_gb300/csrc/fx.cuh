// fx.cuh -- 64-bit block fixed point for the FP64 line transforms.
//
// GB300 issues 64-bit integer additions at 60 per SM and clock and 32 x 32 +
// 64 bit multiply-adds at 22, but FP64 additions and FMAs at 2 (measured with
// dependent-free loops on all SMs).  The line transforms of the FP64 passes
// (passesx.cuh) therefore run on integers: all values of a tile are q 2^E
// with a 64-bit q and one exponent E per tile, so a butterfly addition is
// exact and costs one 64-bit integer addition, and only the twiddle products
// and the changes of E round.
//
// E is chosen per tile from the data, by the L1 norm of its lines: every
// intermediate of a DFT of a line is a partial sum of its elements times unit
// factors, so |re|, |im| <= L1 throughout and L1 < 2^62 quanta rules out
// overflow.  The quantum is at most 2^-61 of the largest L1 norm among the
// tile's 16 lines.  For a line that reaches it, L1 <= sqrt(2) N rms makes the
// rounding error about 2^-54.5 of its rms at N = 256, below the 2^-53 relative
// rounding of each FP64 butterfly it replaces.  For the others the error is the
// same absolute one: a line 2^k times smaller has it 2^k times larger beside
// itself, where the butterflies' would shrink with the line; the transform
// across the lines then adds either to the larger ones.
#pragma once

#include "common.cuh"

namespace plc {

struct fx {
  long long v;
};
struct __align__(16) fxc {
  fx x, y;
};
template <> struct CplxOf<fx> { using type = fxc; };

// A factor |w| <= 1 as w 2^61 = h 2^32 + l with signed 32-bit halves, l never
// -2^31 (so that both halves can be negated).
constexpr int kFxOne = 61;
struct fxk {
  int h, l;
};
// A complex factor w = c + i d as c, d - c and c + d (up to sqrt(2)), for
// products with three real multiplications.
struct __align__(8) fxw {
  fxk c, m, p;
};
__host__ __device__ constexpr fxk fx_split(long long w) {
  const int l = (int)(unsigned)(unsigned long long)w;
  return l == (int)0x80000000 ? fx_split(w + 1) : fxk{(int)((w - l) >> 32), l};
}

__device__ __forceinline__ fx operator+(fx a, fx b) { return fx{a.v + b.v}; }
__device__ __forceinline__ fx operator-(fx a, fx b) { return fx{a.v - b.v}; }
__device__ __forceinline__ fx operator-(fx a) { return fx{-a.v}; }
__device__ __forceinline__ fx operator*(int s, fx a) { return s == 1 ? a : fx{-a.v}; }   // s = +-1
__device__ __forceinline__ fx halve(fx a) { return fx{(a.v + 1) >> 1}; }

__device__ __forceinline__ fx shfl_xor16(fx a) {
  return fx{__shfl_xor_sync(0xffffffffu, a.v, 16)};
}

// Signed halves of q: q = h 2^32 + l.
__device__ __forceinline__ int fx_lo(long long q) { return (int)(unsigned)(unsigned long long)q; }
__device__ __forceinline__ int fx_hi(long long q) {
  return (int)(q >> 32) + (int)((unsigned)fx_lo(q) >> 31);
}
__device__ __forceinline__ long long madw(int a, int b, long long c) { return (long long)a * b + c; }

// Products with factors: the partial products of the high halves and the two
// cross products, rounded to nearest in the cross sum; the product of the
// low halves is below 2 quanta and has zero mean, and is dropped.
constexpr long long kFxRound = 1ll << (kFxOne - 33);
__device__ __forceinline__ long long fx_join(long long hh, long long mid) {
  return (hh << (64 - kFxOne)) + (mid >> (kFxOne - 32));
}
__device__ __forceinline__ fx operator*(fx a, fxk w) {
  const int ah = fx_hi(a.v), al = fx_lo(a.v);
  return fx{fx_join(madw(ah, w.h, 0), madw(al, w.h, madw(ah, w.l, kFxRound)))};
}
__host__ __device__ constexpr fxw fx_factor(long long c, long long d) {
  return fxw{fx_split(c), fx_split(d - c), fx_split(c + d)};
}
// a w (SIGN < 0) or a conj(w) (SIGN > 0), w = c + i d, from c (x + y):
//   a w       = c (x + y) - y (c + d)  + i [c (x + y) + x (d - c)]
//   a conj(w) = c (x + y) + y (d - c)  + i [c (x + y) - x (c + d)]
// Nine wide multiply-adds in place of twelve (S^-1 at 256^3 486 -> 470 us, within
// 1% at 128^3 and 192^3).  |x|, |y| < 2^62 and |x + y| <
// 2^62.5 keep the cross sums below 2^63.
template <int SIGN> __device__ __forceinline__ fxc cmulx(fxc a, fxw w) {
  const long long s = a.x.v + a.y.v;
  const int sh = fx_hi(s), sl = fx_lo(s);
  int xh = fx_hi(a.x.v), xl = fx_lo(a.x.v), yh = fx_hi(a.y.v), yl = fx_lo(a.y.v);
  const long long km = madw(sl, w.c.h, madw(sh, w.c.l, kFxRound)), kh = madw(sh, w.c.h, 0);
  fxk fr = w.p, fi = w.m;       // factors of y in re, of x in im
  if (SIGN > 0) { fr = w.m; fi = w.p; }
  if (SIGN < 0) { fr.h = -fr.h; fr.l = -fr.l; }
  else { fi.h = -fi.h; fi.l = -fi.l; }
  return fxc{{fx_join(madw(yh, fr.h, kh), madw(yl, fr.h, madw(yh, fr.l, km)))},
             {fx_join(madw(xh, fi.h, kh), madw(xl, fi.h, madw(xh, fi.l, km)))}};
}

// cos(2 pi m / R) 2^61 for the radices of the register transforms.
constexpr long long kFxCos1 = 2130321161396766249ll;   // cos(pi / 8)
constexpr long long kFxSin1 = 882407917260943721ll;    // sin(pi / 8)
constexpr long long kFxH = 1630477228166597777ll;      // sqrt(1/2)
constexpr long long kFxT = 1996918623117814388ll;      // sqrt(3)/2
__host__ __device__ constexpr long long fx_cos(int R, int m) {
  if (R == 3 || R == 6) return fx_cos(12, m * (12 / R));
  if (R != 12) {
    constexpr long long c[16] = {1ll << kFxOne, kFxCos1, kFxH, kFxSin1, 0, -kFxSin1, -kFxH, -kFxCos1,
                                 -(1ll << kFxOne), -kFxCos1, -kFxH, -kFxSin1, 0, kFxSin1, kFxH, kFxCos1};
    return c[(m * (16 / R)) & 15];
  }
  constexpr long long c[12] = {1ll << kFxOne, kFxT, 1ll << 60, 0, -(1ll << 60), -kFxT,
                               -(1ll << kFxOne), -kFxT, -(1ll << 60), 0, 1ll << 60, kFxT};
  return c[m % 12];
}
__host__ __device__ constexpr long long fx_sin(int R, int m) {
  if (R == 3 || R == 6) return fx_sin(12, m * (12 / R));
  return R == 2 ? 0 : fx_cos(R, ((m - R / 4) % R + R) % R);
}

template <int SIGN> struct Rot<fx, SIGN> {
  static __device__ __forceinline__ fxc by(fxc a, int R, int m) {
    m %= R;
    if (m == 0) return a;
    if (4 * m == R) return cmul_si<SIGN>(a);
    if (2 * m == R) return fxc{-a.x, -a.y};
    if (4 * m == 3 * R) return cmul_si<-SIGN>(a);
    const long long c = fx_cos(R, m), s = SIGN * fx_sin(R, m);
    if ((8 * m) % R == 0) {   // c, s = +-sqrt(1/2): two products instead of four
      const fxk h = fx_split(kFxH);
      const int sc = c > 0 ? 1 : -1, ss = s > 0 ? 1 : -1;
      return fxc{(sc * a.x - ss * a.y) * h, (ss * a.x + sc * a.y) * h};
    }
    return cmulx<-1>(a, fx_factor(c, s));
  }
};

template <int SIGN> struct Dft<fx, SIGN> {
  using C = fxc;
  static __device__ __forceinline__ void r2(C* v) {
    C a = v[0], b = v[1];
    v[0] = cadd(a, b); v[1] = csub(a, b);
  }
  static __device__ __forceinline__ void r3(C* v) {
    const fxk h = fx_split(kFxT);
    C s = cadd(v[1], v[2]);
    C d = csub(v[1], v[2]);
    C m = C{v[0].x - halve(s.x), v[0].y - halve(s.y)};
    C t = cmul_si<SIGN>(C{d.x * h, d.y * h});
    v[0] = cadd(v[0], s);
    v[1] = cadd(m, t);
    v[2] = csub(m, t);
  }
  static __device__ __forceinline__ void r4(C* v) {
    C a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
    C c = cadd(v[1], v[3]), d = cmul_si<SIGN>(csub(v[1], v[3]));
    v[0] = cadd(a, c); v[2] = csub(a, c);
    v[1] = cadd(b, d); v[3] = csub(b, d);
  }
  static __device__ __forceinline__ void r8(C* v) {
    C e[4] = {v[0], v[2], v[4], v[6]};
    C o[4] = {v[1], v[3], v[5], v[7]};
    r4(e); r4(o);
#pragma unroll
    for (int k = 1; k < 4; ++k) o[k] = Rot<fx, SIGN>::by(o[k], 8, k);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = cadd(e[k], o[k]);
      v[k + 4] = csub(e[k], o[k]);
    }
  }
};

// ------------------------------ tile exponents ------------------------------
constexpr int kFxNaN = 1 << 20;      // tile holds a NaN or an infinity
constexpr int kFxNone = -(1 << 20);  // below the exponent of any tile
constexpr int kFxBits = 62;          // L1 of a line stays below 2^62 quanta

// Smallest b with l1 (1 + 2^-10) < 2^b (l1 > 0).
__device__ __forceinline__ int l1_bits(float l1) {
  return ((int)(__float_as_uint(l1 * 1.0009765625f) >> 23) - 127) + 1;
}
// 2^d as a float, d clamped to the normal range below 1.
__device__ __forceinline__ float exp2_le0(int d) {
  return __uint_as_float((unsigned)(127 + max(d, -120)) << 23);
}
// |q| in units of 2^32, low by less than one unit.
__device__ __forceinline__ float fx_mag(fx a) { return fabsf((float)(int)(a.v >> 32)); }
__device__ __forceinline__ float fx_mag(fxc a) { return fx_mag(a.x) + fx_mag(a.y); }

// q 2^-s rounded to nearest, s >= 0 (half = 2^(s-1), 0 for s = 0).  |q| <= 2^62,
// so every shift from 63 on gives 0.
struct FxShift {
  int s;
  long long half;
  __device__ __forceinline__ explicit FxShift(int d)
      : s(min(max(d, 0), 63)), half((long long)((1ull << s) >> 1)) {}
  __device__ __forceinline__ fx operator()(fx a) const { return fx{(a.v + half) >> s}; }
  __device__ __forceinline__ fxc operator()(fxc a) const { return fxc{(*this)(a.x), (*this)(a.y)}; }
};

// double -> quanta of 2^E, rounded to nearest, where |d| < 2^(E + 62) and, for
// subnormal d, E >= -1083.
__device__ __forceinline__ fx fx_from(double d, int E) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const int ex = (int)(b >> 52) & 0x7ff;   // 0 (zero, subnormal): no implicit bit
  const unsigned long long m = (((b & 0xFFFFFFFFFFFFFull) | (ex ? 1ull << 52 : 0ull)) << 10);
  const int sh = E - max(ex, 1) + 1085, s = min(max(sh, 1), 63);
  const long long q = sh > 63 ? 0ll : (long long)((m + (1ull << (s - 1))) >> s);
  const long long sg = (long long)b >> 63;
  return fx{(q ^ sg) - sg};
}

// q 2^E -> double, rounded to nearest, for |E| <= 900.
__device__ __forceinline__ double fx_to_double(fx a, int E) {
  const long long sg = a.v >> 63;
  const unsigned long long u = (unsigned long long)((a.v ^ sg) - sg);
  const int lz = __clzll((long long)u);
  const unsigned long long n = u << (lz & 63);
  const unsigned long long m = (n >> 11) + ((n >> 10) & 1);   // 53 bits, or 2^53
  const unsigned long long bits =
      ((unsigned long long)(unsigned)(1085 + E - lz) << 52) + m;
  return __longlong_as_double(
      (long long)(u ? (bits | ((unsigned long long)sg & 0x8000000000000000ull)) : 0ull));
}

// The same for any E: NaN tiles, all-zero grids and values near the ends of
// the double range (out of line: rare).
static __device__ __noinline__ double fx_to_double_far(long long q, int E) {
  if (E >= kFxNaN / 2) return __longlong_as_double(0x7ff8000000000000ll);
  return q == 0 ? 0.0 : ldexp((double)q, max(E, -4000));
}

}  // namespace plc
