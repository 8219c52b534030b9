// Fixed-point arithmetic for the FP64 QR: 64-bit integers on the integer
// multiply-add pipe.
//
// Why.  This GPU executes about 1.7 FP64 FMAs per clock and SM (a warp
// instruction every 77 cycles and scheduler) but 50 wide integer multiply-adds
// (32 x 32 + 64 bits; one every 2.5 cycles).  A Householder QR is unitary, so
// every column keeps its norm and needs no floating exponent: entries are held
// as integers at one power-of-two scale per column, |a| <= 2^58 for the
// column's norm, and a product of two such numbers costs three wide
// multiply-adds (the product of the two low limbs, below one unit, is
// dropped).  A real multiply-add costs 7.5 cycles instead of 77, at a rounding
// error of about 2^-58 of the column's norm against 2^-53 in FP64.
//
// A number x in [-2, 2] is the integer x 2^58 = h 2^29 + l with -2^28 <= l <
// 2^28 (|h| <= 2^30; signed low limbs, so that the dropped products average to
// zero and 0 stays exactly 0).  A sum of products is kept as two 64-bit accumulators,
// hh = sum h h' (units) and md = sum h l' + l h' (units 2^-29), by lane: a lane
// sums at most kFxEntries complex entries before it shifts md to units, and only
// units are added across lanes.  Bounds for u of norm sqrt(2) and a of norm 1
// (Cauchy-Schwarz, m entries): md of plain products is below 1.8 sqrt(m) 2^58, that
// of three-product complex ones (FxDot in qr.cu: sums of limbs, up to twice as large)
// 1.8 sqrt(m) 2^59, and their sum, as the imaginary part needs it, 3.6 sqrt(m) 2^59 <
// 2^63 up to m = 19.  Norms: md below sqrt(2 m) 2^57, ll (a square of the low limbs'
// each) m 2^57, added over up to 128 entries after the shift by 3: 2^61.
#pragma once

#include <stdint.h>

#include <cuda_runtime.h>

namespace mdx {

typedef long long i64;
typedef unsigned long long u64;

constexpr int kFxBits = 58;   // fraction bits
constexpr int kFxLimb = 29;   // bits of the low limb
constexpr int kFxEntries = 8;   // complex entries a lane sums at most
constexpr i64 kFxHalf = 1ll << (kFxLimb - 1);  // rounds md to the nearest unit

__device__ __forceinline__ int fx_lo(i64 a) { return (int)((unsigned)a << (32 - kFxLimb)) >> (32 - kFxLimb); }
__device__ __forceinline__ int fx_hi(i64 a) { return (int)(a >> kFxLimb) + (int)((unsigned)fx_lo(a) >> 31); }
// a b as one wide multiply.  (Written out: where the
// compiler can tell a limb's sign it may widen it with zeros and multiply in 64
// bits, three instructions for one.)
__device__ __forceinline__ i64 wide(int a, int b) {
  i64 r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
// c + a b: the multiply above and a plain addition fuse into one wide
// multiply-add (mad.wide itself becomes a multiply and an addition: 2 x the
// instructions, measured).
__device__ __forceinline__ i64 wide_add(int a, int b, i64 c) { return c + wide(a, b); }

// A complex number as limbs: {re high, re low, im high, im low}.
__device__ __forceinline__ int4 fx_split(i64 re, i64 im) {
  return make_int4(fx_hi(re), fx_lo(re), fx_hi(im), fx_lo(im));
}

// x 2^(58 - e) of a double |x| <= 2^e (e a power-of-two exponent), rounded to
// nearest (ties away); zero, subnormals and anything below half a unit give 0.
__device__ __forceinline__ i64 fx_from(u64 bits, int e) {
  const int ex = (int)((bits >> 52) & 0x7ff);
  const u64 m = (bits & 0xfffffffffffffull) | 0x10000000000000ull;
  const int s = ex - 1075 + kFxBits - e;  // m 2^s
  u64 v;
  if (s >= 0)
    v = m << (s & 63);
  else
    v = s < -54 ? 0ull : ((m >> ((-s - 1) & 63)) + 1ull) >> 1;
  if (ex == 0) v = 0;
  return (bits >> 63) ? -(i64)v : (i64)v;
}

// The double a 2^(e - 58), rounded to nearest even (the exponent must stay in
// the normal range).
__device__ __forceinline__ u64 fx_to_bits(i64 a, int e) {
  if (a == 0) return 0;
  const u64 sign = (u64)a & 0x8000000000000000ull;
  u64 m = a < 0 ? (u64)(-a) : (u64)a;
  const int lz = __clzll((i64)m);
  m <<= lz;
  const unsigned rem = (unsigned)m & 0x7ffu;
  u64 f = m >> 11;
  f += (rem > 0x400u || (rem == 0x400u && (f & 1))) ? 1 : 0;
  return sign | (((u64)(e + 63 - lz - kFxBits + 1022) << 52) + f);
}

// The float nearest the double `bits` (round to nearest even, as the
// conversion instruction), for zero or magnitudes in float's normal range.
__device__ __forceinline__ unsigned f32_bits_of(u64 bits) {
  if (bits == 0) return 0;
  const u64 m = bits & 0x7fffffffffffffffull;
  const unsigned rem = (unsigned)m & 0x1fffffffu;
  unsigned f = (unsigned)((m - (896ull << 52)) >> 29);
  f += (rem > 0x10000000u || (rem == 0x10000000u && (f & 1))) ? 1 : 0;
  return f | ((unsigned)(bits >> 32) & 0x80000000u);
}

__device__ __forceinline__ u64 fx_mulhi(u64 a, u64 b) {
  return __umul64hi(a, b);
}
__device__ __forceinline__ int fx_clz(u64 x) {
  return __clzll((i64)x);
}

// 2^59 / sqrt(X 2^-60) for X in [2^58, 2^60]: the single-precision estimate y
// (24 bits, exact square) refined by 1 / sqrt(1 - e) = 1 + e/2 + 3 e^2/8,
// e = 1 - x y^2 (|e| < 2^-20, so the next term is below 2^-61).
__device__ __forceinline__ u64 fx_rsqrt(u64 X) {
  const float xf = (float)(unsigned)(X >> 32) * 3.7252903e-9f;  // 2^-28
  const float yf = rsqrtf(xf);
  const unsigned Y = (unsigned)(yf * 8388608.0f);  // y 2^23
  const i64 e = (1ll << 61) - (i64)fx_mulhi(X << 4, ((u64)Y * Y) << 15);  // e 2^61
  const int es = (int)(e >> 21);
  const i64 t = (e >> 1) + ((wide(es, es) * 3) >> 22);  // (e/2 + 3 e^2/8) 2^61
  return ((u64)Y << 36) + (u64)(((i64)Y * (t >> 2)) >> 23);
}

// x y / 2^58 of |x|, |y| < 2^60, in units 2^-(58 + X): the full product's high
// part with X more bits.
template <int X>
__device__ __forceinline__ i64 fx_mul(i64 x, i64 y) {
  const int xh = fx_hi(x), xl = fx_lo(x), yh = fx_hi(y), yl = fx_lo(y);
  const i64 md = wide_add(xh, yl, wide_add(xl, yh, wide(xl, yl) >> kFxLimb));
  return (wide(xh, yh) << X) + ((md + (1ll << (kFxLimb - 1 - X))) >> (kFxLimb - X));
}

// S 2^-116 = x 4^h with x in [1/4, 1): returns x 2^60 and h (S > 0).
__device__ __forceinline__ u64 fx_norm4(unsigned __int128 S, int& h) {
  const u64 hi = (u64)(S >> 64), lo = (u64)S;
  const int p = hi ? 127 - fx_clz(hi) : 63 - fx_clz(lo);  // top bit
  h = (p - 114) >> 1;                                     // ceil((p - 115) / 2)
  const int sh = 56 + 2 * h;
  return sh >= 0 ? (u64)(S >> sh) : lo << -sh;
}

// Householder reflector of a column part with entries x (units 2^-58, norm
// sigma <= 1): H = I - u u^H, |u|^2 = 2, H x = -p sigma e_0 with p = x_0 / |x_0|
// (1 if x_0 = 0).  u_0 = p m and u_r = x_r g / 2^s.
struct FxReflector {
  i64 pr, pi;  // p, units 2^-58
  i64 ur, ui;  // u_0, units 2^-58
  i64 g;       // units 2^-58, at most 2
  int s;       // sigma in [2^(s-1), 2^s)
  u64 sigma;   // sigma 2^(62 - s)
  __device__ __forceinline__ i64 scale(i64 x) const {  // u_r of x_r
    return (fx_mul<4>(s > 0 ? x >> s : x << -s, g) + 8) >> 4;
  }
};
// hh = sum xh^2, md = sum xh xl, ll = sum xl^2 over the entries' limbs (ll / 8,
// so that the sum over 128 rows fits); x0 the first entry.  False (and nothing computed) if sigma < 2^-26.
__device__ __forceinline__ bool fx_reflector(i64 hh, i64 md, u64 ll, i64 x0r, i64 x0i, FxReflector& f) {
  typedef unsigned __int128 u128;
  const u128 S = ((u128)(u64)hh << 58) + ((u128)(__int128)md << 30) + ((u128)ll << 3);
  if ((i64)(S >> 64) <= 0) return false;
  const u64 X = fx_norm4(S, f.s);
  const u64 r1 = fx_rsqrt(X);
  f.sigma = fx_mulhi(X << 4, r1 << 3);  // sqrt(x) 2^62
  u64 ax = 0;
  f.pr = 1ll << kFxBits;
  f.pi = 0;
  const u64 ar = (u64)(x0r < 0 ? -x0r : x0r), ai = (u64)(x0i < 0 ? -x0i : x0i);
  if ((ar | ai) != 0) {
    int hq;
    const u64 Q = fx_norm4((u128)ar * ar + (u128)ai * ai, hq);
    const u64 r2 = fx_rsqrt(Q);
    const int d = f.s - hq;  // |x_0| <= sigma: d >= 0
    ax = d < 64 ? fx_mulhi(Q << 4, r2 << 3) >> d : 0;
    const i64 rr = (i64)(r2 >> 1);
    f.pr = fx_mul<0>(hq > 0 ? x0r >> hq : x0r << -hq, rr);
    f.pi = fx_mul<0>(hq > 0 ? x0i >> hq : x0i << -hq, rr);
  }
  const u64 sa = f.sigma + ax;             // (sigma + |x_0|) 2^(62 - s)
  const u64 A = fx_mulhi(f.sigma << 1, sa);  // sigma (sigma + |x_0|) 2^(61 - 2 s), below 2^62
  const bool big = A >= (1ull << 61);
  const u64 g59 = fx_rsqrt(big ? A >> 3 : A >> 1) >> (big ? 1 : 0);
  f.g = (i64)(g59 >> 1);
  const i64 m = (i64)(fx_mulhi(sa, g59 << 3) >> 2);  // (sigma + |x_0|) g, in [1, sqrt 2]
  f.ur = fx_mul<0>(f.pr, m);
  f.ui = fx_mul<0>(f.pi, m);
  return true;
}

}  // namespace mdx
