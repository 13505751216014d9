// fx64.cuh -- the pair arithmetic of the FP64 force path in 64-bit fixed point.
//
// What bounds the FP64 path: GB300 issues one FP64 warp instruction per 19
// cycles and SM, 64 times less than FP32, and a pair needs 34 of them (646
// cycles; measured 1.6e10 pairs/s, 89% of that).  The 32-bit integer units are
// 15 to 75 times faster (measured, lanes per clock and SM: IMAD.WIDE 25,
// IMAD.HI 32, IMAD, shifts and logic 63, adds 128), so a pair is computed here
// with mantissas of 58 to 63 bits held in two 32-bit words: the upper 64 bits
// of a product of two of them are one IMAD.WIDE and two IMAD.HI.  29 and 32 of
// those and about 220 cheaper instructions make a pair, 135 cycles per warp
// and SM (7.4e10 pairs/s at N = 65536, n = 4096); the half of the FMA pipe that
// multiplies integers is busy for three quarters of them.  Measured on the way
// there, on the same case: cross terms by IMAD.WIDE with a rounded sum 144
// cycles; C++ carries instead of add.cc chains 156; 3 or 5 CTAs of 128 threads
// per SM instead of 4, or two pairs interleaved, level to 4% slower; the cross
// terms of D.W rounded down one by one 6% faster, and the jerk's error twice
// as large, so not kept.
//
// No step holds fewer than the 53 bits of an FP64 number: each rounds at 2^-56
// of its own result or finer, and the sums over j are exact.  Measured against
// long double sums (Plummer spheres of 513 to 60000, equal and Salpeter masses,
// and sets with outliers, close pairs, wide mass ratios), the rms errors are
// 0.5 to 1.0 (acceleration), 0.35 to 1.0 (jerk) and 0.4 to 1.0 (potential)
// times those of the FP64 evaluation (1.0, 1.13 and 1.15 for 33 particles, one
// 2^30 away, whose pairs are nearly all left to FP64).
//
// Formats.  2^g bounds the coordinates of the pair and eps, 2^gv the
// velocities, em is the exponent of the largest mass near by:
//   X = x 2^(60-g), V = v 2^(60-gv)         integers, rounded to nearest
//   M in [2^62, 2^63), m = M 2^(em-k-63)    exact (k: this mass's own exponent)
// The pair is normalised by the even power 4^s that brings R = (r^2 + eps^2)
// into [2^58, 2^60) (units 2^(2(g-60)+64)); with sigma = sqrt(R 2^-60):
//   D = dX 2^s, W = dV, Y = 2^63 / (2 sigma), Z = 2^62 / (2 sigma)^2,
//   MY = M Y 2^-64, G = MY Z 2^-64, U = W - 3 (D.W) D / (D.D + eps^2),
// and the three kinds of terms are MY (potential), G D 2^-64 (acceleration)
// and G U 2^-64 (jerk), to be scaled by 2^(s-k), 2^(2s-k) and 2^(3s-k).  They
// are added up as 96-bit integers at one scale for all pairs.
// 1/sigma: the hardware's FP32 rsqrt gives y0 to 2^-18 or better; e = 1 - R y0^2
// is formed to 2^-57 and y0 (1 + e/2 + 3 e^2 / 8) keeps that.
//
// Pairs this does not cover are left to FP64 arithmetic by the caller: those
// whose difference of position (velocity) is below 2^(g-8) (2^(gv-8)), so that
// the grid would round it to fewer than 52 bits, and j whose mass is below
// 2^-kKMax of the largest, or negative.
#pragma once

#include <stdint.h>

namespace nbx {

constexpr int kKMax = 15;       // largest mass exponent below the tile's
constexpr int kFold = 512;      // pairs a 96-bit sum takes (its headroom: 2^9 terms)
constexpr int kExpLo = -300, kExpHi = 300;  // exponents the formats take
// scales of the sums: potential 2^(em-g-78), acceleration 2^(em-2g-68),
// jerk 2^(em-3g+gv-59) times the integer
constexpr int kPotScale = -78, kAccScale = -68, kJerkScale = -59;
constexpr int32_t kWMin = 1 << 20;      // high word of the smallest velocity difference taken, 2^(gv-8) ...
constexpr int32_t kNoPairs = 0x7FFFFFFF;  // ... and the value that no pair reaches

struct Sum96 {
  uint32_t w0, w1, w2;
};

// one j-particle on the tile's grid
struct JFix {
  int64_t X[3], V[3];
  uint64_t M;
  int k;
};

// one i-particle on the same grid; its softening, (eps / unit)^2 2^-64 as
// 32.32 bits above a 32-bit fraction and in FP32
struct IFix {
  int64_t X[3], V[3];
  uint32_t e2[3];
  float e2f;
  float rmin;    // square of the smallest distance taken (high words): 2^(g-8), or eps / 16
  int kx, kv;    // the i-particle lies 2^kx (2^kv) outside the tile's grid: its own grid is that much coarser
  int32_t wmin;  // kWMin; 0 where every velocity is zero; kNoPairs: take no pair
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

// a b 2^-64 for a, b in signed digits, to a unit: the cross terms are rounded
// down and the mean of that, one unit, is put back (one = min_u32(ah, 1)), the
// low digits' product is left out.  Without bias, odd in a and b (a force and
// its reaction stay opposite), zero where one of them is.
__device__ __forceinline__ int64_t mul_odd(int32_t ah, int32_t al, int32_t one, int32_t bh, int32_t bl) {
  return (int64_t)ah * bh + mad_hi(al, bh, mad_hi(ah, bl, min_u32(bh, one)));
}

// the same for positive numbers below 2^63, without the unit put back
__device__ __forceinline__ uint64_t umul_fl(uint64_t a, uint64_t b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  const uint64_t t = (uint64_t)ah * bh;
  uint32_t lo = (uint32_t)t, hi = (uint32_t)(t >> 32);
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;"
      : "+&r"(lo), "+&r"(hi)
      : "r"(__umulhi(ah, bl) + __umulhi(al, bh)));
  return ((uint64_t)hi << 32) | lo;
}

// sum += t 2^L (0 <= L < 32)
__device__ __forceinline__ void add_shifted(Sum96& s, int64_t t, int L) {
  const uint32_t t0 = (uint32_t)t, t1 = (uint32_t)((uint64_t)t >> 32);
  uint32_t a2;
  asm("shr.s32 %0, %1, %2;" : "=r"(a2) : "r"(t1), "r"(32 - L));  // (a shift by 32 gives the sign)
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
      : "+&r"(s.w0), "+&r"(s.w1), "+&r"(s.w2)
      : "r"(__funnelshift_l(0u, t0, L)), "r"(__funnelshift_l(t0, t1, L)), "r"(a2));
}

// s 2^e, rounded once to nearest: a normal FP64 number built from the sum's
// bits.  About 40 integer instructions; by FP64 conversions, products and a
// TwoSum it was eleven FP64 ones, which a warp issues 64 cycles apart, 7 sums
// 2.4 us at the end of every item of a small system.
__device__ __forceinline__ double to_double(Sum96 s, int e) {
  const uint32_t neg = (uint32_t)((int32_t)s.w2 >> 31);
  uint32_t a0 = s.w0 ^ neg, a1 = s.w1 ^ neg, a2 = s.w2 ^ neg;
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.u32 %2, %2, 0;"
      : "+&r"(a0), "+&r"(a1), "+&r"(a2)
      : "r"(neg & 1u));
  // the leading bit to bit 95: whole words, then the rest
  int n = 0;
  if (a2 == 0u) {
    n = 32;
    a2 = a1;
    a1 = a0;
    a0 = 0u;
    if (a2 == 0u) {
      n = 64;
      a2 = a1;
      a1 = 0u;
    }
  }
  if (a2 == 0u) return 0.0;
  const int z = __clz((int)a2);
  const uint32_t m1 = __funnelshift_l(a1, a2, z), m0 = __funnelshift_l(a0, a1, z), rest = __funnelshift_l(0u, a0, z);
  const int E = 95 - n - z + e + 1023;
  const uint64_t m = ((uint64_t)m1 << 32) | m0;
  const uint32_t r = m0 & 0x7FFu;
  const uint32_t up = (r > 0x400u || (r == 0x400u && (rest != 0u || (m0 & 0x800u) != 0u))) ? 1u : 0u;
  const uint64_t f = (m >> 11) + up;  // [2^52, 2^53]
  const uint64_t sign = (uint64_t)(neg & 0x80000000u) << 32;
  if (E >= 1 && E <= 2045) return __longlong_as_double((long long)((((uint64_t)(uint32_t)(E - 1) << 52) + f) | sign));
  const double d = scalbn((double)f, E - 1075);
  return neg ? -d : d;
}

// The pair (i, j): its seven terms added to a (acc, jerk, pot).  Returns
// false, and adds nothing, when skip is set or the pair is not one of those
// described above.  SH: some lane of the warp has kx or kv > 0.
// (Every shift by a computed amount is a funnel shift, whose amount is taken
// modulo 32: a pair that is left computes with meaningless shifts.)
template <bool SH>
__device__ __forceinline__ bool pair(const JFix& j, const IFix& i, bool skip, Sum96 (&a)[7]) {
  int64_t D[3], W[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    D[c] = (SH ? j.X[c] >> i.kx : j.X[c]) - i.X[c];
    W[c] = (SH ? j.V[c] >> i.kv : j.V[c]) - i.V[c];
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
    digits((int64_t)(((uint64_t)__funnelshift_l(lo, hi, s) << 32) | __funnelshift_l(0u, lo, s)), dh[c], dl[c]);
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
  const uint64_t Gn = umul_fl(MY, Z);

  // shifts of the terms: potential 15 + s - k, acceleration 9 + 2s - k, jerk
  // 3s - k; where the last is negative (light j far away) G is shifted instead.
  // (max as an instruction: written in C++, the compiler dropped it.)
  const int k = j.k, d3 = 3 * s - k;
  int Lj;
  asm("max.s32 %0, %1, 0;" : "=r"(Lj) : "r"(d3));
  const int rho = Lj - d3;  // at most kKMax
  const uint32_t g1 = (uint32_t)(Gn >> 32);
  const uint64_t G = ((uint64_t)__funnelshift_r(g1, 0u, rho) << 32) | __funnelshift_r((uint32_t)Gn, g1, rho);

  // D.W 2^-64, then T = 8 (-6 D.W) Z 2^-64: A = 16 T D 2^-64 is the jerk's
  // -3 (r.v) r / s^2.  The sum's cross terms are rounded once: their error
  // grows by up to 24 on the way to A, the largest of all.
  int64_t cw = (int64_t)dh[0] * wl[0] + 0x80000000ll;
  cw = (int64_t)dl[0] * wh[0] + cw;
  cw = (int64_t)dh[1] * wl[1] + cw;
  cw = (int64_t)dl[1] * wh[1] + cw;
  cw = (int64_t)dh[2] * wl[2] + cw;
  cw = (int64_t)dl[2] * wh[2] + cw;
  int64_t RW = (int64_t)dh[0] * wh[0] + (int64_t)(int32_t)(cw >> 32);
  RW = (int64_t)dh[1] * wh[1] + RW;
  RW = (int64_t)dh[2] * wh[2] + RW;
  int32_t qh, ql, zh, zl, th, tl, gh, gl;
  digits(RW * -6, qh, ql);
  digits((int64_t)Z, zh, zl);
  digits((int64_t)((uint64_t)mul_odd(zh, zl, 1, qh, ql) << 3), th, tl);
  digits((int64_t)G, gh, gl);

  const int32_t one_t = min_u32(th, 1), one_g = min_u32(gh, 1);
  add_shifted(a[6], (int64_t)MY, 15 + s - k);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int64_t U = W[c] + (int64_t)((uint64_t)mul_odd(th, tl, one_t, dh[c], dl[c]) << 4);
    int32_t uh, ul;
    digits(U, uh, ul);
    add_shifted(a[c], mul_odd(gh, gl, one_g, dh[c], dl[c]), Lj + 9 - s);
    add_shifted(a[3 + c], mul_odd(gh, gl, one_g, uh, ul), Lj);
  }
  return ok;
}

}  // namespace nbx
