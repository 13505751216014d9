// hermite.cuh -- per-particle arithmetic of the 4th-order Hermite block-step
// scheme, shared by every loop driver (the host-driven kernels, the body of
// the CUDA-graph loop and the persistent loop): the predictor of Sec. 4.1
// step 3 and the corrector with the power-of-two block-step rule of step 5
// (block steps of Sec. 2).  One definition, so every driver takes the same
// steps bit for bit.
#pragma once

#include <math.h>

#include "nb_internal.cuh"

namespace nbh {

// largest power of two <= x for positive finite x (clears the mantissa)
__device__ __forceinline__ double pow2_floor(double x) {
  if (!(x > 0.0)) return 0.0;
  if (isinf(x)) return x;
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  if ((b >> 52) == 0) return 0.0;  // subnormal: below any admissible step
  return __longlong_as_double((long long)(b & 0xFFF0000000000000ULL));
}

// y / x.  When x is a positive power of two (every block step, and h = t - t_i
// of every active particle) the quotient is y times 2^-k formed from the
// exponent bits: the same correctly rounded result without an FP64 divide
// (the FP64 pipe bounds the corrector).  Anything else takes the division.
__device__ __forceinline__ double div_pow2(double y, double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned long long e = b >> 52;  // sign 0 and biased exponent
  if ((b & 0x000FFFFFFFFFFFFFULL) == 0 && e >= 1 && e <= 2045)
    return y * __longlong_as_double((long long)((2046ULL - e) << 52));
  return y / x;
}

__device__ __forceinline__ double clamp_dt(double c, double dt_min, double dt_max) {
  if (c > dt_max) c = dt_max;
  if (c < dt_min) c = dt_min;
  return c;
}

// ---- exact integer forms of FP64 operations with exact results -------------
// On this GPU a warp's FP64 instruction occupies it for about 64 cycles, and
// the corrector's chain is the critical path of a small block step.  Where an
// FP64 operation's result is exact -- a power of two raised to a power, a
// constant scaled by a power of two, the power-of-two floor of a correctly
// rounded square root, comparisons -- it is formed from the exponent bits
// instead: the same bits, no FP64 instruction.  Outside the stated
// preconditions the FP64 expression is taken.

__device__ __forceinline__ unsigned long long dbits(double x) { return (unsigned long long)__double_as_longlong(x); }

// x a positive normal power of two: its exponent in e
__device__ __forceinline__ bool is_pow2(double x, int& e) {
  const unsigned long long b = dbits(x);
  const unsigned long long E = b >> 52;  // sign bit 0 and biased exponent
  e = (int)E - 1023;
  return (b & 0x000FFFFFFFFFFFFFULL) == 0 && E >= 1 && E <= 2046;
}

// 2^e, e in [-1022, 1023]
__device__ __forceinline__ double pow2i(int e) {
  return __longlong_as_double((long long)((unsigned long long)(e + 1023) << 52));
}

// c 2^k for a positive normal c whose scaled exponent stays normal (the
// callers' ranges guarantee it): exact, so equal to the FP64 product
__device__ __forceinline__ double scale_pow2(double c, int k) {
  return __longlong_as_double((long long)(dbits(c) + ((unsigned long long)(long long)k << 52)));
}

// powers of the step h = t - t_i and the constant multiples the corrector
// uses: from the exponent when h is a power of two 2^e with |e| <= 200 (every
// block step; all results normal), else by FP64 products
struct HPow {
  double ih, ih2, ih3, h2, h3, h4, h5;
  double h3_6, h4_24, h5_120, h6;  // h^3/6, h^4/24, h^5/120, 6h
  int e;                           // h = 2^e when pow2
  bool pow2;
};

// y 2^k, exact: from the exponent bits when y is finite and normal and the
// result stays normal, else the FP64 product y p2 with p2 = 2^k (the same
// value; infinities and NaNs take the product)
__device__ __forceinline__ double mul_pow2(double y, int k, double p2) {
  const unsigned long long b = dbits(y);
  const int E = (int)((b >> 52) & 0x7FF);
  if (E >= 1 && E <= 2046 && E + k >= 1 && E + k <= 2046)  // y finite and normal, so is the result
    return __longlong_as_double((long long)(b + ((unsigned long long)(long long)k << 52)));
  return y * p2;
}

// y / h^2 and y / h^3 of the corrector (products by the exact inverse powers)
__device__ __forceinline__ double div_h2(const struct HPow& q, double y) {
  return q.pow2 ? mul_pow2(y, -2 * q.e, q.ih2) : y * q.ih2;
}
__device__ __forceinline__ double div_h3(const struct HPow& q, double y) {
  return q.pow2 ? mul_pow2(y, -3 * q.e, q.ih3) : y * q.ih3;
}
// the FP64 products (the reference of the exponent form, and its fallback)
__device__ __forceinline__ HPow h_powers_fp64(double h) {
  HPow q;
  q.ih = div_pow2(1.0, h);
  q.ih2 = q.ih * q.ih;
  q.ih3 = q.ih2 * q.ih;
  q.h2 = h * h;
  q.h3 = q.h2 * h;
  q.h4 = q.h3 * h;
  q.h5 = q.h4 * h;
  q.h3_6 = q.h3 * (1.0 / 6.0);
  q.h4_24 = q.h4 * (1.0 / 24.0);
  q.h5_120 = q.h5 * (1.0 / 120.0);
  q.h6 = 6.0 * h;
  q.e = 0;
  q.pow2 = false;
  return q;
}

__device__ __forceinline__ HPow h_powers(double h) {
  HPow q;
  int e;
  if (is_pow2(h, e) && e >= -200 && e <= 200) {
    q.e = e;
    q.pow2 = true;
    q.ih = pow2i(-e);
    q.ih2 = pow2i(-2 * e);
    q.ih3 = pow2i(-3 * e);
    q.h2 = pow2i(2 * e);
    q.h3 = pow2i(3 * e);
    q.h4 = pow2i(4 * e);
    q.h5 = pow2i(5 * e);
    q.h3_6 = scale_pow2(1.0 / 6.0, 3 * e);
    q.h4_24 = scale_pow2(1.0 / 24.0, 4 * e);
    q.h5_120 = scale_pow2(1.0 / 120.0, 5 * e);
    q.h6 = scale_pow2(6.0, e);
    return q;
  }
  return h_powers_fp64(h);
}

// t (>= 0) an integer multiple of 2^s: 1 yes, 0 no, -1 undecided here
// (negative, subnormal or non-finite t, or t 2^-s below the normal range)
__device__ __forceinline__ int multiple_of_pow2(double t, int s) {
  const unsigned long long b = dbits(t);
  if (b == 0) return 1;
  const unsigned long long E = b >> 52;
  if (E == 0 || E >= 2047) return -1;
  const int d = (int)E - 1023 - s;  // t 2^-s = 1.f 2^d
  if (d < -1000) return -1;
  if (d < 0) return 0;
  if (d >= 52) return 1;
  return (b & ((1ULL << (52 - d)) - 1ULL)) == 0 ? 1 : 0;
}

// The new step (Sec. 4.1 step 5; block steps of Sec. 2) of a particle at time
// t with step dt_old, from num = na n2 + nj^2 and den = nj n3 + n2^2 (na =
// |a1|, nj = |j1|, n2 = |a2 + a3 h|, n3 = |a3|): Aarseth criterion
// crit = sqrt(eta num / den), its power-of-two floor clamped to [dt_min,
// dt_max]; the step shrinks to that freely and doubles only when t is a
// multiple of the doubled step (and the doubled step is admissible).  Counts
// criteria below dt_min; crit_nan reports a NaN criterion.  This is the FP64
// expression: the reference of new_step_nd's exponent form and its fallback.
__device__ __forceinline__ double new_step_fp64(double t, double dt_old, double num, double den, double eta,
                                                double dt_min, double dt_max, nb_dev_status* st, bool& crit_nan) {
  const double crit = (den == 0.0) ? (double)INFINITY : sqrt(eta * num / den);
  if (crit < dt_min) atomicAdd(&st->dt_underflows, 1ULL);
  crit_nan = isnan(crit);
  const double c = clamp_dt(pow2_floor(crit), dt_min, dt_max);
  if (c < dt_old) return c;
  const double two = 2.0 * dt_old;
  const double qq = div_pow2(t, two);  // exact: two is a power of two
  return (c >= two && two <= dt_max && qq == floor(qq)) ? two : dt_old;
}

// new_step_fp64's result from the exponent eq of q = fl(fl(eta num) / den), a
// finite normal positive: the power-of-two floor of the correctly rounded
// square root of q is 2^floor(eq / 2) (the square root never rounds up to a
// power of two), and crit < dt_min = 2^m exactly when eq < 2m (under).  False
// when a step bound or dt_old is not a power of two, or t is negative or
// subnormal.
__device__ __forceinline__ bool step_by_exponent(int eq, double t, double dt_old, double dt_min, double dt_max,
                                                 double& dnew, bool& under) {
  int emin, emax, eo;
  if (!(is_pow2(dt_min, emin) && is_pow2(dt_max, emax) && is_pow2(dt_old, eo) && emin <= emax)) return false;
  const int s = eo + 1;  // the doubled step 2^s
  const int mt = eq >= -1022 && eq <= 1023 ? multiple_of_pow2(t, s) : -1;
  if (mt < 0) return false;
  under = eq < 2 * emin;
  int ec = (eq - (eq & 1)) / 2;  // floor(eq / 2): exponent of the criterion's floor
  if (ec > emax) ec = emax;
  if (ec < emin) ec = emin;
  dnew = ec < eo ? pow2i(ec) : ((ec >= s && s <= emax && mt == 1) ? pow2i(s) : dt_old);
  return true;
}

// new_step_fp64's result from exponents.  For positive normal N = fl(eta num)
// and D = den, fl(N / D) has exponent e_N - e_D, less one when N's
// significand is below D's (a quotient of 53-bit significands never rounds up
// to a power of two).  So no division or square root is needed; they are taken
// (the FP64 expression) only when an operand is zero, subnormal or non-finite
// or step_by_exponent declines.
__device__ __forceinline__ double new_step_nd(double t, double dt_old, double num, double den, double eta,
                                              double dt_min, double dt_max, nb_dev_status* st, bool& crit_nan) {
  crit_nan = false;
  if (den != 0.0) {
    const double nq = eta * num;
    const unsigned long long bN = dbits(nq), bD = dbits(den);
    const unsigned long long EN = bN >> 52, ED = bD >> 52;  // sign bits 0 for positive operands
    if (EN >= 1 && EN <= 2046 && ED >= 1 && ED <= 2046) {
      const int eq = (int)EN - (int)ED - ((bN & 0x000FFFFFFFFFFFFFULL) < (bD & 0x000FFFFFFFFFFFFFULL) ? 1 : 0);
      double dnew;
      bool under;
      if (step_by_exponent(eq, t, dt_old, dt_min, dt_max, dnew, under)) {
        if (under) atomicAdd(&st->dt_underflows, 1ULL);
        return dnew;
      }
    }
  }
  return new_step_fp64(t, dt_old, num, den, eta, dt_min, dt_max, st, crit_nan);
}

// the step from the four norms' roots
__device__ __forceinline__ double new_step(double t, double dt_old, double na, double nj, double n2, double n3,
                                           double eta, double dt_min, double dt_max, nb_dev_status* st,
                                           bool& crit_nan) {
  const double num = na * n2 + nj * nj;
  const double den = nj * n3 + n2 * n2;
  return new_step_nd(t, dt_old, num, den, eta, dt_min, dt_max, st, crit_nan);
}

// The square root of a positive normal s as m 2^e, m in [1, 2), in FP32 to a few
// 2^-24; e = kNoRoot for other s.
constexpr int kNoRoot = 1 << 20;
struct Root {
  float m;
  int e;
};
__device__ __forceinline__ Root root_of(double s) {
  const unsigned long long b = dbits(s);
  const int E = (int)(b >> 52);
  Root r;
  const int k = E - 1023;
  const unsigned int m = 0x3F800000u | ((unsigned int)(b >> 29) & 0x7FFFFFu);
  const float f = __uint_as_float(m + ((unsigned int)(k & 1) << 23));
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r.m) : "f"(f));  // f in [1, 4)
  r.e = E >= 1 && E <= 2046 ? k >> 1 : kNoRoot;
  return r;
}

// 2^-k for k >= 0, in FP32 (at least 2^-100)
__device__ __forceinline__ float pow2neg(int k) { return __uint_as_float((unsigned int)(127 - min(k, 100)) << 23); }

// The exponent of the criterion's square, floor(log2(eta (na n2 + nj^2) / (nj n3
// + n2^2))), from the roots of the four squared norms in FP32.  Of the
// criterion only this exponent reaches the new step (step_by_exponent), and
// the FP64 expression rounds a few 2^-53: so where the FP32 value (truncated
// operands, roots, products, sums of positive terms, one reciprocal: below
// 1.5e-6 of it, 24 units of its last place) lies more than 64 units from a power
// of two, the FP64 expression has the same exponent.  False otherwise (15 values
// in 10^6), and where FP64 could leave its normal range: the caller then takes
// the FP64 roots, 16 to 60 more FP64 instructions of 64 cycles each.
__device__ __forceinline__ bool crit_exponent(const Root& na, const Root& nj, const Root& n2, const Root& n3,
                                              double eta, int& eq) {
  const unsigned long long be = dbits(eta);
  const int Ee = (int)(be >> 52) - 1023;
  const float fe = __uint_as_float(0x3F800000u | ((unsigned int)(be >> 29) & 0x7FFFFFu));
  const int p1 = na.e + n2.e, p2 = 2 * nj.e, q1 = nj.e + n3.e, q2 = 2 * n2.e;
  const int P = max(p1, p2), Q = max(q1, q2);
  const float num = na.m * n2.m * pow2neg(P - p1) + nj.m * nj.m * pow2neg(P - p2);  // [1, 8)
  const float den = nj.m * n3.m * pow2neg(Q - q1) + n2.m * n2.m * pow2neg(Q - q2);
  float rden;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rden) : "f"(den));
  const unsigned int r = __float_as_uint(fe * num * rden);  // 2^-3 .. 2^4
  const unsigned int frac = r & 0x7FFFFFu;
  eq = (int)(r >> 23) - 127 + Ee + P - Q;
  // (a missing root makes its sums 2^20 or so and fails the range)
  return frac >= 64u && frac <= 0x7FFFFFu - 64u && Ee >= -1000 && Ee <= 0 && P >= -900 && P <= 900 && Q >= -900 &&
         Q <= 900 && eq >= -1022 && eq <= 1023;
}

// Predictor (Sec. 4.1 step 3) of row i over h = t - t_i, Horner form:
//   xp = x + v h + a h^2/2 + jk h^3/6,   vp = v + a h + jk h^2/2
__device__ __forceinline__ void taylor1(double h, double xv, double vv, double av, double jv, double& px,
                                        double& pv) {
  px = xv + h * (vv + h * (0.5 * av + h * (jv * (1.0 / 6.0))));
  pv = vv + h * (av + h * (0.5 * jv));
}
__device__ __forceinline__ void taylor(int64_t i, int64_t n_pad, double h, const double* __restrict__ x,
                                       const double* __restrict__ v, const double* __restrict__ a,
                                       const double* __restrict__ jk, double (&px)[3], double (&pv)[3]) {
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int64_t q = d * n_pad + i;
    taylor1(h, x[q], v[q], a[q], jk[q], px[d], pv[d]);
  }
}

// the predicted row in the FP64 j-store and/or the mixed one; the
// double-single split of a position is exact: hi = fl32(xp), lo = fl32(xp - hi)
// (hi also to the caller, for the tile's box; mixed store only)
__device__ __forceinline__ void store_predicted(int64_t i, int64_t n_pad, const double (&px)[3],
                                                const double (&pv)[3], double mi, double* __restrict__ xp,
                                                double* __restrict__ vp, float4* __restrict__ jA,
                                                float4* __restrict__ jB, float2* __restrict__ jC,
                                                bool write_fp64, bool write_mixed, float (&hi)[3]) {
  if (write_fp64) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      xp[d * n_pad + i] = px[d];
      vp[d * n_pad + i] = pv[d];
    }
  }
  if (write_mixed) {
    float lo[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) nb_split(px[d], hi[d], lo[d]);
    jA[i] = make_float4(hi[0], hi[1], hi[2], nb_f32(mi));
    jB[i] = make_float4(lo[0], lo[1], lo[2], nb_f32(pv[0]));
    jC[i] = make_float2(nb_f32(pv[1]), nb_f32(pv[2]));
  }
}

// The reach of a j-memory record: a bound on every coordinate's move within a
// step d, |v_c| d + |a_c| d^2/2 + |j_c| d^3/6 summed over components, from the
// FP32 sums of the magnitudes (each rounding 2^-24, eight of them, under the
// factor 1 + 2^-20: as a bound FP32 serves, and FP64 would be 13 instructions
// of 64 cycles at the end of a correction)
__device__ __forceinline__ float reach_of(float sv, float sa, float sj, double d) {
  const float df = nb_f32(d);
  return df * (sv + df * (0.5f * sa + df * (sj * (1.0f / 6.0f)))) * (1.0f + 0x1p-20f);
}

// Corrector (Sec. 4.1 step 5) of row i at block time t from its new force
// f = (a1[3], j1[3], pot1), h = t - t_i.  Hermite interpolation of the
// acceleration through (a0, j0) and (a1, j1) gives at the start
//   a2 = [-6 (a0 - a1) - h (4 j0 + 2 j1)] / h^2,  a3 = [12 (a0 - a1) + 6 h (j0 + j1)] / h^3,
// and x1 = xp + a2 h^4/24 + a3 h^5/120,  v1 = vp + a2 h^3/6 + a3 h^4/24.
// New step: Aarseth criterion at the end of the step (a2e = a2 + a3 h),
// largest power of two below it within [dt_min, dt_max]; it may shrink
// freely and doubles only when t is a multiple of the doubled step.
// Returns the row's next due time t + dt_new.
__device__ __forceinline__ double correct_row(int64_t i, int64_t n_pad, double t, const double (&f)[7], double eta,
                                            double dt_min, double dt_max, double* __restrict__ x,
                                            double* __restrict__ v, double* __restrict__ a,
                                            double* __restrict__ jk, double* __restrict__ pot,
                                            double* __restrict__ ti, double* __restrict__ dt,
                                            const double* __restrict__ xp, const double* __restrict__ vp,
                                            nb_dev_status* __restrict__ st) {
  const double h = t - ti[i];
  const HPow hp = h_powers(h);
  double na2 = 0, nj2 = 0, n22 = 0, n32 = 0;
  bool finite = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int64_t q = c * n_pad + i;
    const double a0 = a[q], j0 = jk[q];
    const double a1 = f[c], j1 = f[3 + c];
    const double da = a0 - a1;
    const double a2 = div_h2(hp, -6.0 * da - h * (4.0 * j0 + 2.0 * j1));
    const double a3 = div_h3(hp, 12.0 * da + hp.h6 * (j0 + j1));
    const double x1 = xp[q] + a2 * hp.h4_24 + a3 * hp.h5_120;
    const double v1 = vp[q] + a2 * hp.h3_6 + a3 * hp.h4_24;
    const double a2e = a2 + a3 * h;
    x[q] = x1;
    v[q] = v1;
    a[q] = a1;
    jk[q] = j1;
    na2 += a1 * a1;
    nj2 += j1 * j1;
    n22 += a2e * a2e;
    n32 += a3 * a3;
    finite = finite && isfinite(x1) && isfinite(v1) && isfinite(a1) && isfinite(j1);
  }
  const double p1 = f[6];
  pot[i] = p1;
  const double dt0 = dt[i];
  bool crit_nan = false, under = false;
  int eq;
  double dnew;
  if (crit_exponent(root_of(na2), root_of(nj2), root_of(n22), root_of(n32), eta, eq) &&
      step_by_exponent(eq, t, dt0, dt_min, dt_max, dnew, under)) {
    if (under) atomicAdd(&st->dt_underflows, 1ULL);
  } else {
    dnew = new_step(t, dt0, sqrt(na2), sqrt(nj2), sqrt(n22), sqrt(n32), eta, dt_min, dt_max, st, crit_nan);
  }
  if (!finite || !isfinite(p1) || crit_nan) atomicOr(&st->flags, NB_ST_NUMERIC);
  ti[i] = t;
  dt[i] = dnew;
  return t + dnew;
}

// Inputs of one lane's part of a correction: the row's time and step before
// it, and component `sub` (< 3; lane 3 takes component 0) of the old
// acceleration and jerk and of the predicted position and velocity.
struct CorrIn {
  double t0, dt0, a0, j0, xp, vp;
};

// The same correction spread over four lanes of a warp: lane `sub` < 3 of
// the group takes component `sub` (the same FP64 operations in the same order
// as correct_row), the squared norms are gathered by shuffles and summed in
// component order, one on each of lanes 0-3, and lane 0 applies the step rule
// to their roots.  The result is correct_row's, bit for bit;
// the dependent FP64 chain is about a third as long, which matters where one
// particle's correction is the critical path of a block step.
//
// a1, j1: component `sub` (lane 3 and up: component 0) of the new acceleration
// and jerk; p1: the new potential (used by lane 0).
//
// Every lane of the warp must call this with the same control flow: the
// shuffles use the full mask and are taken unconditionally.  `base` is the
// warp lane of the group's lane 0; `write` says whether this group's row is
// real (lanes of groups without a row, and lanes sub >= 4, compute on a
// valid row and write nothing).  With jm the corrected row's j-memory record
// is written as well (write_jm_record's values; its mass word is left as it
// is): each lane its component, lane 0 the reach once the new step is known.
// `keep` sees what is written, for a caller that holds the rows elsewhere too.
// Returns, on the group's lane 0 of a real row, the row's next due time
// t + dt_new (0 elsewhere).
struct NoKeep {
  __device__ __forceinline__ void component(int, double, double, double, double) const {}
  __device__ __forceinline__ void record(int, float, float, float, float, float, float) const {}
  __device__ __forceinline__ void step(double, double) const {}
};
template <class Keep = NoKeep>
__device__ __forceinline__ double correct_lanes4(int64_t i, int64_t n_pad, double t, double a1, double j1,
                                                 double p1, const CorrIn& in, double eta, double dt_min, double dt_max,
                                                 double* __restrict__ x, double* __restrict__ v,
                                                 double* __restrict__ a, double* __restrict__ jk,
                                                 double* __restrict__ pot, double* __restrict__ ti,
                                                 double* __restrict__ dt, nb_dev_status* __restrict__ st, int sub,
                                                 int base, bool write, float4* __restrict__ jm = nullptr,
                                                 const Keep keep = Keep()) {
  const double h = t - in.t0;
  const HPow hp = h_powers(h);
  double sq[4] = {0.0, 0.0, 0.0, 0.0};  // a1^2, j1^2, a2e^2, a3^2 of this lane's component
  float ab[3];                          // |v1|, |a1|, |j1| of this lane's component (the record's reach)
  int fin = 1;
  const int c = sub < 3 ? sub : 0;
  {
    const int64_t q = c * n_pad + i;
    const double a0 = in.a0, j0 = in.j0;
    const double da = a0 - a1;
    const double a2 = div_h2(hp, -6.0 * da - h * (4.0 * j0 + 2.0 * j1));
    const double a3 = div_h3(hp, 12.0 * da + hp.h6 * (j0 + j1));
    const double x1 = in.xp + a2 * hp.h4_24 + a3 * hp.h5_120;
    const double v1 = in.vp + a2 * hp.h3_6 + a3 * hp.h4_24;
    const double a2e = a2 + a3 * h;
    if (write && sub < 3) {
      x[q] = x1;
      v[q] = v1;
      a[q] = a1;
      jk[q] = j1;
      if (jm) {
        float* r = reinterpret_cast<float*>(jm + i);
        float xh, xl, vh, vl;
        nb_split(x1, xh, xl);
        nb_split(v1, vh, vl);
        r[c] = xh;
        r[4 * n_pad + c] = xl;
        r[8 * n_pad + c] = vh;
        r[12 * n_pad + c] = vl;
        const float a2f = 0.5f * nb_f32(a1), j6f = nb_f32(j1 * (1.0 / 6.0));
        r[16 * n_pad + c] = a2f;
        r[4 * n_pad * (2 + c) + 3] = j6f;
        keep.record(c, xh, xl, vh, vl, a2f, j6f);
      }
      keep.component(c, x1, v1, a1, j1);
    }
    sq[0] = a1 * a1;
    sq[1] = j1 * j1;
    sq[2] = a2e * a2e;
    sq[3] = a3 * a3;
    ab[0] = jm ? fabsf(nb_f32(v1)) : 0.0f;
    ab[1] = jm ? fabsf(nb_f32(a1)) : 0.0f;
    ab[2] = jm ? fabsf(nb_f32(j1)) : 0.0f;
    fin = (isfinite(x1) && isfinite(v1) && isfinite(a1) && isfinite(j1)) ? 1 : 0;
  }
  // lane sub (< 4) sums squared norm `sub` in component order (0 + x^2 +
  // y^2 + z^2, as correct_row's running sums): three FP64 adds per lane
  // instead of all four norms on every lane; every shuffle is taken by every lane
  double own[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double t0 = __shfl_sync(0xffffffffu, sq[0], base + k);
    const double t1 = __shfl_sync(0xffffffffu, sq[1], base + k);
    const double t2 = __shfl_sync(0xffffffffu, sq[2], base + k);
    const double t3 = __shfl_sync(0xffffffffu, sq[3], base + k);
    own[k] = sub == 1 ? t1 : (sub == 2 ? t2 : (sub == 3 ? t3 : t0));
  }
  const double mine = ((0.0 + own[0]) + own[1]) + own[2];
  float sum_ab[3] = {0.0f, 0.0f, 0.0f};  // write_jm_record's sums of |v|, |a|, |j| in component order
  if (jm) {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const float s0 = __shfl_sync(0xffffffffu, ab[r], base);
      const float s1 = __shfl_sync(0xffffffffu, ab[r], base + 1);
      const float s2 = __shfl_sync(0xffffffffu, ab[r], base + 2);
      sum_ab[r] = (s0 + s1) + s2;
    }
  }
  const int f0 = __shfl_sync(0xffffffffu, fin, base);
  const int f1 = __shfl_sync(0xffffffffu, fin, base + 1);
  const int f2 = __shfl_sync(0xffffffffu, fin, base + 2);
  // one root per lane, all four on every lane
  const Root root = root_of(mine);
  Root rt[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    rt[k].m = __shfl_sync(0xffffffffu, root.m, base + k);
    rt[k].e = __shfl_sync(0xffffffffu, root.e, base + k);
  }
  int eq;
  double dnew = in.dt0;
  bool under = false;
  const bool quick = crit_exponent(rt[0], rt[1], rt[2], rt[3], eta, eq) &&
                     step_by_exponent(eq, t, in.dt0, dt_min, dt_max, dnew, under);
  double rn[4] = {0.0, 0.0, 0.0, 0.0};
  if (__any_sync(0xffffffffu, write && !quick)) {  // (rare) the FP64 roots
    const double r64 = sqrt(mine);
#pragma unroll
    for (int k = 0; k < 4; ++k) rn[k] = __shfl_sync(0xffffffffu, r64, base + k);
  }
  if (!write || sub != 0) return 0.0;
  pot[i] = p1;
  bool crit_nan = false;
  if (!quick)
    dnew = new_step(t, in.dt0, rn[0], rn[1], rn[2], rn[3], eta, dt_min, dt_max, st, crit_nan);
  else if (under)
    atomicAdd(&st->dt_underflows, 1ULL);
  const bool finite = f0 && f1 && f2;
  if (!finite || !isfinite(p1) || crit_nan) atomicOr(&st->flags, NB_ST_NUMERIC);
  ti[i] = t;
  dt[i] = dnew;
  keep.step(t, dnew);
  if (jm) reinterpret_cast<float*>(jm + n_pad + i)[3] = reach_of(sum_ab[0], sum_ab[1], sum_ab[2], dnew);
  return t + dnew;
}

// j-memory record of row i (the on-the-fly j prediction's input, Sec. 4.4
// step 4; layout in force_common.cuh): double-single position and velocity,
// a/2 and jerk/6 in FP32, the mass, and the reach Rd >= |v_c| dt + |a_c| dt^2/2
// + |j_c| dt^3/6 summed over components (a bound on every coordinate's move
// within the row's current step), rounded up.  Rows >= N: padding.
__device__ __forceinline__ void write_jm_record(int64_t i, int64_t N, int64_t n_pad, const double* __restrict__ m,
                                                const double* __restrict__ x, const double* __restrict__ v,
                                                const double* __restrict__ a, const double* __restrict__ jk,
                                                const double* __restrict__ dt, float4* __restrict__ jm) {
  float xh[3], xl[3], vh[3], vl[3], a2[3], j6[3], mf = 0.0f, reach = 0.0f;
  if (i < N) {
    float sv = 0.0f, sa = 0.0f, sj = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int64_t q = c * n_pad + i;
      const double xv = x[q], vv = v[q], av = a[q], jv = jk[q];
      nb_split(xv, xh[c], xl[c]);
      nb_split(vv, vh[c], vl[c]);
      const float af = nb_f32(av);
      a2[c] = 0.5f * af;
      j6[c] = nb_f32(jv * (1.0 / 6.0));
      sv += fabsf(vh[c]);
      sa += fabsf(af);
      sj += fabsf(nb_f32(jv));
    }
    reach = reach_of(sv, sa, sj, dt[i]);
    mf = nb_f32(m[i]);
  } else {  // padding row: massless and far away
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      xh[c] = (float)NB_PAD_POS;
      xl[c] = vh[c] = vl[c] = a2[c] = j6[c] = 0.0f;
    }
  }
  jm[i] = make_float4(xh[0], xh[1], xh[2], mf);
  jm[n_pad + i] = make_float4(xl[0], xl[1], xl[2], reach);
  jm[2 * n_pad + i] = make_float4(vh[0], vh[1], vh[2], j6[0]);
  jm[3 * n_pad + i] = make_float4(vl[0], vl[1], vl[2], j6[1]);
  jm[4 * n_pad + i] = make_float4(a2[0], a2[1], a2[2], j6[2]);
}

}  // namespace nbh
