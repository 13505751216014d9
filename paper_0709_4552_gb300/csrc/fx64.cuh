// fx64.cuh -- the pair arithmetic of the FP64 force path in 64-bit fixed point.
//
// What bounds the FP64 path: GB300 issues one FP64 warp instruction per 19
// cycles and SM, 64 times less than FP32, and a pair needs 34 of them (646
// cycles; measured 1.6e10 pairs/s, 89% of that).  The 32-bit integer units are
// 15 to 75 times faster (measured, lanes per clock and SM: IMAD.WIDE 25,
// IMAD.HI 32, IMAD, shifts and logic 63, adds 128), so a pair is computed here
// with mantissas of 58 to 63 bits held in two 32-bit words.  40 IMAD.WIDE, 20
// IMAD.HI and about 275 cheaper instructions make a pair, 150 cycles per warp
// and SM (6.7e10 pairs/s at N = 65536, n = 4096); no pipe is busy for more than
// two thirds of them.  Measured, on another case (N = 40000, n = 4864): this
// form 2.92 ms; the products with their last bits and the velocities' fractions
// in every pair (FINE) 3.43; the upper 64 bits of each product only (an
// IMAD.WIDE and two IMAD.HI) with 96-bit sums 2.55, but the small components of
// a flat system and the forces of light particles then hold too few bits; 3
// CTAs of 128 threads per SM instead of 4 level.
//
// No result holds fewer bits than FP64 arithmetic gives it, component by
// component: the sums over j are exact and hold 32 bits below the unit of a
// product, and a tile that would need more is left to FP64 (fp64_view in
// force_common.cuh).  Against 113-bit sums, each component in units of the sum of
// its terms' sizes, the rms errors are 0.14 to 0.93 of those of FP64 arithmetic
// in Plummer spheres of 33 to 4000 (equal and Salpeter masses) and at most 0.98
// of them in discs of thickness 0.3 to 1e-4, needles, sheets, cold velocities,
// discs far from the origin or with a halo, a star's companions of 2^-4 to 2^-15
// of its mass and pairs of clusters; where nearly all pairs are left to FP64
// (flatter ones, far from the origin) they are FP64's.
//
// Formats.  2^g bounds the coordinates of the pair and eps, 2^gv the
// velocities, em is the exponent of the largest mass near by:
//   X = x 2^(60-g), V = v 2^(60-gv)         integers and 32 fraction bits
//   M in [2^62, 2^63), m = M 2^(em-k-63)    exact (k: this mass's own exponent)
// The pair is normalised by the even power 4^s that brings R = (r^2 + eps^2)
// into [2^58, 2^60) (units 2^(2(g-60)+64)); with sigma = sqrt(R 2^-60):
//   D = dX 2^s, W = dV, Y = 2^63 / (2 sigma), Z = 2^62 / (2 sigma)^2,
//   MY = M Y 2^-64, G = MY Z 2^-64, U = W - 3 (D.W) D / (D.D + eps^2),
// and the three kinds of terms are MY (potential), G D 2^-64 (acceleration)
// and G U 2^-64 (jerk), to be scaled by 2^(s-k), 2^(2s-k) and 2^(3s-k).  They
// are added up at one scale for all pairs, as integers of 96 bits (potential)
// and of 96 bits with 32 fraction bits, from which k may take up to 15: a light
// particle's terms keep their bits, as they are all there is on the heaviest one.
// 1/sigma: the hardware's FP32 rsqrt gives y0 to 2^-18 or better; e = 1 - R y0^2
// is formed to 2^-57 and y0 (1 + e/2 + 3 e^2 / 8) keeps that.
//
// Pairs this does not cover are left to FP64 arithmetic by the caller: those
// whose difference of position (velocity) is below 2^(g-8) (2^(gv-8)), and j
// whose mass is below 2^-kKMax of the largest, or negative.
#pragma once

#include <stdint.h>

namespace nbx {

constexpr int kKMax = 15;       // largest mass exponent below the tile's
constexpr int kFold = 512;      // pairs a sum takes (its headroom: 2^9 terms)
constexpr int kExpLo = -300, kExpHi = 300;  // exponents the formats take
// scales of the sums: potential 2^(em-g-78), acceleration 2^(em-2g-91),
// jerk 2^(em-3g+gv-91) times the integer
constexpr int kPotScale = -78, kAccScale = -91, kJerkScale = -91;
constexpr int32_t kWMin = 1 << 20;      // high word of the smallest velocity difference taken, 2^(gv-8)

struct Sum96 {
  uint32_t w0, w1, w2;
};
struct Sum128 {
  uint32_t w0, w1, w2, w3;
};
struct Sums {
  Sum128 f[6];  // acceleration, jerk
  Sum96 p;      // potential
};

// one j-particle on the tile's grid; xl, vl: 32 fraction bits below the unit
struct JFix {
  int64_t X[3], V[3];
  uint32_t xl[3], vl[3];
  uint64_t M;
  int k;
};

// one i-particle on the same grid; its softening, (eps / unit)^2 2^-64 as
// 32.32 bits above a 32-bit fraction and in FP32
struct IFix {
  int64_t X[3], V[3];
  uint32_t xl[3], vl[3];
  uint32_t e2[3];
  float e2f;
  float rmin;    // square of the smallest distance taken (high words): 2^(g-8), or eps / 16
  int kx, kv;    // the i-particle lies 2^kx (2^kv) outside the tile's grid: its own grid is that much coarser
  int32_t wmin;  // kWMin; 0 where every velocity is zero
};

// a = h 2^32 + l with both digits signed
__device__ __forceinline__ void digits(int64_t a, int32_t& h, int32_t& l) {
  l = (int32_t)(uint32_t)a;
  h = (int32_t)(a >> 32) + (int32_t)((uint32_t)a >> 31);
}

__device__ __forceinline__ int32_t mad_hi(int32_t a, int32_t b, int32_t c) {
  int32_t d;
  asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

__device__ __forceinline__ int32_t min_u32(int32_t a, int32_t b) {
  int32_t d;
  asm("min.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

__device__ __forceinline__ uint32_t sar(uint32_t a, int n) {  // n = 32 gives the sign
  uint32_t d;
  asm("shr.s32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(n));
  return d;
}

__device__ __forceinline__ void add2(uint32_t& a0, uint32_t& a1, uint32_t b0) {
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+&r"(a0), "+&r"(a1) : "r"(b0));
}
__device__ __forceinline__ void add3(uint32_t& a0, uint32_t& a1, uint32_t& a2, uint32_t b0, uint32_t b1, uint32_t b2) {
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
      : "+&r"(a0), "+&r"(a1), "+&r"(a2)
      : "r"(b0), "r"(b1), "r"(b2));
}
__device__ __forceinline__ void add4(Sum128& s, uint32_t b0, uint32_t b1, uint32_t b2, uint32_t b3) {
  asm("add.cc.u32 %0, %0, %4;\n\taddc.cc.u32 %1, %1, %5;\n\taddc.cc.u32 %2, %2, %6;\n\taddc.u32 %3, %3, %7;"
      : "+&r"(s.w0), "+&r"(s.w1), "+&r"(s.w2), "+&r"(s.w3)
      : "r"(b0), "r"(b1), "r"(b2), "r"(b3));
}
__device__ __forceinline__ void sub3(uint32_t& a0, uint32_t& a1, uint32_t& a2, uint32_t b0, uint32_t b1, uint32_t b2) {
  asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %4;\n\tsubc.u32 %2, %2, %5;"
      : "+&r"(a0), "+&r"(a1), "+&r"(a2)
      : "r"(b0), "r"(b1), "r"(b2));
}

// a b 2^-64 for a, b in signed digits, to a unit: the cross terms are rounded
// down and the mean of that, one unit, is put back (one = min_u32(ah, 1)), the
// low digits' product is left out.  Without bias, odd in a and b, zero where
// one of them is.
__device__ __forceinline__ int64_t mul_odd(int32_t ah, int32_t al, int32_t one, int32_t bh, int32_t bl) {
  return (int64_t)ah * bh + mad_hi(al, bh, mad_hi(ah, bl, min_u32(bh, one)));
}

// a b 2^-64 with 32 fraction bits.  Without FINE the low digits' product is
// left out, up to a quarter of a unit; with it all but a few units of the last
// bit are there, those of the fractions af and bf of a and b too.  Odd in a and
// b, but for what is left out, so a force and its reaction stay opposite.  The
// cross terms' sum must fit 63 bits.
template <bool FINE>
__device__ __forceinline__ int64_t mul(int32_t ah, int32_t al, uint32_t af, int32_t bh, int32_t bl, uint32_t bf,
                                       uint32_t& frac) {
  int64_t t = (int64_t)ah * bl;
  if (FINE) {
    t += (int64_t)__mulhi(al, bl);
    t += 2 * (int64_t)__mulhi(ah, (int32_t)(bf >> 1));
    t += 2 * (int64_t)__mulhi(bh, (int32_t)(af >> 1));
  }
  t = (int64_t)al * bh + t;
  frac = (uint32_t)t;
  return (int64_t)ah * bh + (int64_t)(int32_t)(t >> 32);
}

// a b 2^-64 for positive numbers below 2^63, rounded down to a unit
__device__ __forceinline__ uint64_t umul_fl(uint64_t a, uint64_t b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  const uint64_t t = (uint64_t)ah * bh;
  uint32_t lo = (uint32_t)t, hi = (uint32_t)(t >> 32);
  add2(lo, hi, __umulhi(ah, bl) + __umulhi(al, bh));
  return ((uint64_t)hi << 32) | lo;
}

// sum += t 2^L (0 <= L < 32)
__device__ __forceinline__ void add_shifted(Sum96& s, int64_t t, int L) {
  const uint32_t t0 = (uint32_t)t, t1 = (uint32_t)((uint64_t)t >> 32);
  add3(s.w0, s.w1, s.w2, __funnelshift_l(0u, t0, L), __funnelshift_l(t0, t1, L), sar(t1, 32 - L));
}

// sum += floor(t 2^-k) 2^L, t with 32 fraction bits f (0 <= k, L < 32)
__device__ __forceinline__ void add_shifted(Sum128& s, int64_t t, uint32_t f, int k, int L) {
  uint32_t t0 = f, t1 = (uint32_t)t, t2 = (uint32_t)((uint64_t)t >> 32);
  t0 = __funnelshift_r(t0, t1, k);
  t1 = __funnelshift_r(t1, t2, k);
  t2 = sar(t2, k);
  add4(s, __funnelshift_l(0u, t0, L), __funnelshift_l(t0, t1, L), __funnelshift_l(t1, t2, L), sar(t2, 32 - L));
}

// s 2^e, rounded once to nearest: a normal FP64 number built from the sum's
// bits.  About 50 integer instructions; by FP64 conversions, products and a
// TwoSum it was eleven FP64 ones, which a warp issues 64 cycles apart, 7 sums
// 2.4 us at the end of every item of a small system.
__device__ __forceinline__ double to_double(Sum128 s, int e) {
  const uint32_t neg = sar(s.w3, 31);
  Sum128 a = {s.w0 ^ neg, s.w1 ^ neg, s.w2 ^ neg, s.w3 ^ neg};
  add4(a, neg & 1u, 0u, 0u, 0u);
  // the leading bit to bit 127: whole words, then the rest
  int n = 0;
#pragma unroll
  for (int w = 0; w < 3; ++w)
    if (a.w3 == 0u) {
      n += 32;
      a.w3 = a.w2;
      a.w2 = a.w1;
      a.w1 = a.w0;
      a.w0 = 0u;
    }
  if (a.w3 == 0u) return 0.0;
  const int z = __clz((int)a.w3);
  const uint32_t m1 = __funnelshift_l(a.w2, a.w3, z), m0 = __funnelshift_l(a.w1, a.w2, z);
  const uint32_t rest = __funnelshift_l(a.w0, a.w1, z) | a.w0;
  const int E = 127 - n - z + e + 1023;
  const uint64_t m = ((uint64_t)m1 << 32) | m0;
  const uint32_t r = m0 & 0x7FFu;
  const uint32_t up = (r > 0x400u || (r == 0x400u && (rest != 0u || (m0 & 0x800u) != 0u))) ? 1u : 0u;
  const uint64_t f = (m >> 11) + up;  // [2^52, 2^53]
  const uint64_t sign = (uint64_t)(neg & 0x80000000u) << 32;
  if (E >= 1 && E <= 2045) return __longlong_as_double((long long)((((uint64_t)(uint32_t)(E - 1) << 52) + f) | sign));
  const double d = scalbn((double)f, E - 1075);
  return neg ? -d : d;
}
__device__ __forceinline__ double to_double(Sum96 s, int e) {
  return to_double(Sum128{s.w0, s.w1, s.w2, sar(s.w2, 31)}, e);
}

// j's value on i's coarser grid: (x2 x1 . x0) >>= k (0 to 63)
__device__ __forceinline__ void coarser(uint32_t& x0, uint32_t& x1, uint32_t& x2, int k) {
  const int64_t q = (int64_t)(((uint64_t)x2 << 32) | x1) >> k;
  x0 = k < 32 ? __funnelshift_r(x0, x1, k) : __funnelshift_r(x1, x2, k);
  x1 = (uint32_t)q;
  x2 = (uint32_t)((uint64_t)q >> 32);
}

// The pair (i, j): its seven terms added to a.  Returns false, and adds
// nothing, when skip is set or the pair is not one of those described above.
// SH: some lane of the warp has kx or kv > 0.  FINE: see mul.
// (Every shift by a computed amount is a funnel shift, whose amount is taken
// modulo 32: a pair that is left computes with meaningless shifts.)
template <bool SH, bool FINE>
__device__ __forceinline__ bool pair(const JFix& j, const IFix& i, bool skip, Sums& a) {
  int64_t D[3], W[3];
  uint32_t df[3], wf[3];  // fractions
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    uint32_t x0 = j.xl[c], x1 = (uint32_t)j.X[c], x2 = (uint32_t)((uint64_t)j.X[c] >> 32);
    if (SH) coarser(x0, x1, x2, i.kx);
    sub3(x0, x1, x2, i.xl[c], (uint32_t)i.X[c], (uint32_t)((uint64_t)i.X[c] >> 32));
    df[c] = x0;
    D[c] = (int64_t)(((uint64_t)x2 << 32) | x1);
    wf[c] = 0u;
    if (FINE) {
      x0 = j.vl[c], x1 = (uint32_t)j.V[c], x2 = (uint32_t)((uint64_t)j.V[c] >> 32);
      if (SH) coarser(x0, x1, x2, i.kv);
      sub3(x0, x1, x2, i.vl[c], (uint32_t)i.V[c], (uint32_t)((uint64_t)i.V[c] >> 32));
      wf[c] = x0;
      W[c] = (int64_t)(((uint64_t)x2 << 32) | x1);
    } else {
      W[c] = (SH ? j.V[c] >> i.kv : j.V[c]) - i.V[c];
    }
  }
  int32_t wh[3], wl[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) digits(W[c], wh[c], wl[c]);
  // FP32 estimate of r^2 from the high words
  const float f0 = (float)(int32_t)(D[0] >> 32), f1 = (float)(int32_t)(D[1] >> 32), f2 = (float)(int32_t)(D[2] >> 32);
  const float r2 = fmaf(f2, f2, fmaf(f1, f1, f0 * f0));
  const bool ok = !skip & (r2 >= i.rmin) &
                  ((max(max(wh[0], wh[1]), wh[2]) >= i.wmin) | (min(min(wh[0], wh[1]), wh[2]) <= -i.wmin));
  const int bits = __float_as_int(r2 + i.e2f);
  const int s = (((186 << 23) | 0x7FFFFF) - bits) >> 24;  // floor((59 - exponent) / 2): 0 to 9

  int32_t dh[3], dl[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const uint32_t lo = (uint32_t)D[c], hi = (uint32_t)((uint64_t)D[c] >> 32);
    digits((int64_t)(((uint64_t)__funnelshift_l(lo, hi, s) << 32) | __funnelshift_l(df[c], lo, s)), dh[c], dl[c]);
    df[c] = __funnelshift_l(0u, df[c], s);
  }

  // R = D.D 2^-64 + eps^2
  int64_t R = (int64_t)dh[0] * dh[0] +
              ((__mulhi(dh[0], dl[0]) + __mulhi(dh[1], dl[1]) + __mulhi(dh[2], dl[2])) << 1);
  R = (int64_t)dh[1] * dh[1] + R;
  R = (int64_t)dh[2] * dh[2] + R;
  R += (int64_t)(((uint64_t)__funnelshift_l(i.e2[1], i.e2[2], 2 * s) << 32) | __funnelshift_l(i.e2[0], i.e2[1], 2 * s));

  // 1 / (2 sigma): y0 as a 31-bit integer (a multiple of 512), then the residual
  const float y0 = nb_rsqrt_approx(__int_as_float(bits + (s << 24)));
  uint32_t Y0 = (uint32_t)__float_as_int(fmaf(y0, 0x1p60f, 0x1p32f)) << 9;
  Y0 = Y0 < 0x7FFFFE00u ? Y0 : 0x7FFFFE00u;
  const uint64_t P = umul_fl((uint64_t)R << 2, (uint64_t)Y0 * Y0);
  const int64_t e = (int64_t)((1ull << 58) - P);                  // 2^58 (1 - R y0^2)
  const int32_t eh = (int32_t)(e >> 10);
  const int64_t c2 = e + ((3 * (int64_t)__mulhi(eh, eh)) >> 8);   // 2^59 (e/2 + 3 e^2 / 8)
  const uint64_t c5 = (uint64_t)c2 << 5;
  const int64_t yc = (int64_t)(int32_t)Y0 * (int32_t)(c5 >> 32) + __umulhi(Y0, (uint32_t)c5);
  const uint64_t Y = ((uint64_t)Y0 << 32) + (uint64_t)yc;

  const uint32_t yh = (uint32_t)(Y >> 32), yl = (uint32_t)Y;
  const uint64_t Z = (uint64_t)yh * yh + (__umulhi(yh, yl) << 1);
  const uint64_t MY = umul_fl(ok ? j.M : 0ull, Y);
  const uint64_t G = umul_fl(MY, Z);

  // 6 D.W 2^-64, then T = 8 (6 D.W) Z 2^-64: A = 16 T D 2^-64 is the jerk's
  // 3 (r.v) r / s^2
  int32_t qh, ql, zh, zl, th, tl, gh, gl;
  uint32_t tf = 0u;
  digits((int64_t)Z, zh, zl);
  digits((int64_t)G, gh, gl);
  int64_t RW = (int64_t)dh[0] * wh[0];
  RW = (int64_t)dh[1] * wh[1] + RW;
  RW = (int64_t)dh[2] * wh[2] + RW;
  if (FINE) {
    int64_t t = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      t = (int64_t)dh[c] * wl[c] + t;
      t = (int64_t)dl[c] * wh[c] + t;
      t += (int64_t)__mulhi(dl[c], wl[c]);
      t += 2 * ((int64_t)__mulhi(dh[c], (int32_t)(wf[c] >> 1)) + (int64_t)__mulhi(wh[c], (int32_t)(df[c] >> 1)));
    }
    const uint64_t low = 6 * (uint64_t)(uint32_t)t;
    digits((RW + (t >> 32)) * 6 + (int64_t)(low >> 32), qh, ql);
    const uint64_t T = (uint64_t)mul<true>(zh, zl, 0u, qh, ql, (uint32_t)low, tf);
    digits((int64_t)((T << 3) | (tf >> 29)), th, tl);
    tf <<= 3;
  } else {
    int32_t cw = 3;  // (the mean of what the six lose)
#pragma unroll
    for (int c = 0; c < 3; ++c) cw = mad_hi(dl[c], wh[c], mad_hi(dh[c], wl[c], cw));
    digits((RW + cw) * 6, qh, ql);
    digits((int64_t)((uint64_t)mul_odd(zh, zl, 1, qh, ql) << 3), th, tl);
  }

  const int k = j.k;
  add_shifted(a.p, (int64_t)MY, 15 + s - k);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    uint32_t f;
    const uint64_t A = (uint64_t)mul<FINE>(th, tl, tf, dh[c], dl[c], df[c], f);
    uint32_t u0 = wf[c], u1 = (uint32_t)W[c], u2 = (uint32_t)((uint64_t)W[c] >> 32);
    sub3(u0, u1, u2, f << 4, __funnelshift_l(f, (uint32_t)A, 4), __funnelshift_l((uint32_t)A, (uint32_t)(A >> 32), 4));
    int32_t uh, ul;
    digits((int64_t)(((uint64_t)u2 << 32) | u1), uh, ul);
    int64_t t = mul<FINE>(gh, gl, 0u, dh[c], dl[c], df[c], f);
    add_shifted(a.f[c], t, f, k, 2 * s);
    t = mul<FINE>(gh, gl, 0u, uh, ul, u0, f);
    add_shifted(a.f[3 + c], t, f, k, 3 * s);
  }
  return ok;
}

}  // namespace nbx
