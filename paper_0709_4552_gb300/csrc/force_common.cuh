// force_common.cuh -- the direct-sum force "work item" (Sec. 4.1 step 4,
// Eq. 3) shared by every launch shape: the grid kernels of the host-driven
// path, the persistent kernels of the graph-driven loop and of the batched
// ensemble.  One item = one i-tile (NT*IPT active particles of one list)
// against one contiguous j-range [jlo, jhi) of the j-store.
//
// For each active i and every j != i (Plummer softening eps, G = 1):
//   r = x_j - x_i, w = v_j - v_i, s^2 = r.r + eps^2,
//   acc += m_j r / s^3,  jerk += m_j (w / s^3 - 3 (r.w) r / s^5),  pot -= m_j / s.
// Items sum +m/s; the sign of the potential is applied when the item is
// final (one split) or by the split reduction.
//
// Mixed path: positions are double-single pairs (hi, lo) written by the
// predictor; r = (x_j.hi - x_i.hi) + (x_j.lo - x_i.lo) is the FP64 difference
// rounded to FP32 within about an ulp (hi difference exact for close pairs,
// Sterbenz).  Pairwise arithmetic is FP32 with one hardware rsqrt (MUFU),
// optionally refined by one Newton step (NB_MIXED_NEWTON).  The jerk term of
// a pair is formed completely before it is accumulated: its two parts
// (w / s^3 and -3 (r.w) r / s^5) cancel for close pairs, and adding them to
// the running sum one after the other costs up to 4x in the worst particle's
// error.  FP32 partial sums over one j-tile (JT pairs) are folded into
// double-single accumulators (an FP32 pair hi + lo, Knuth's TwoSum: no FP64
// instruction in the loop; NB_MIXED_DS_FOLD = 0 folds into FP64 instead).
// j-tiles (40 B per particle: float4
// hi+m, float4 lo+vx, float2 vy vz) are staged in shared memory with cp.async
// double buffering and read as warp-wide broadcasts.
//
// FP64 path: FP64 inputs and results, the pair arithmetic in 64-bit fixed
// point on the integer units (fx64.cuh; the FP64 pipe issues 2 FMA/clk/SM,
// 1/64 of FP32), exact sums of up to 512 pairs folded into (hi, lo) FP64
// accumulators with Knuth's TwoSum; the few pairs the fixed point does not
// take in IEEE FP64, 1/s from an FP32 seed refined in FP64.
//
// Self pair: excluded by index, as in the definition.  Mixed path: only the
// j-tile holding one of a warp's own i needs the test, so a warp vote picks a
// masked copy of the inner loop for that tile (no per-pair cost elsewhere).
//
// Ragged j-ranges: a tile reaching past jhi loads clamped (in-bounds)
// addresses and the slots past jhi are overwritten with a massless particle
// far away, which contributes exactly zero.
#pragma once

#include "nb_internal.cuh"

#include "fx64.cuh"

// one Newton step on the hardware rsqrt in the mixed path (1 = on)
#ifndef NB_MIXED_NEWTON
#define NB_MIXED_NEWTON 0
#endif
// FP64 accumulators of the mixed path in shared memory instead of registers
#ifndef NB_MIXED_SMEM_ACC
#define NB_MIXED_SMEM_ACC 0
#endif
// double-single (FP32 TwoSum) accumulators of the mixed path (0 = FP64)
#ifndef NB_MIXED_DS_FOLD
#define NB_MIXED_DS_FOLD 1
#endif
// unroll depth of the mixed inner loop over a j-tile
#ifndef NB_MIXED_UNROLL
#define NB_MIXED_UNROLL 4
#endif
// one i per thread: two j per instruction with the packed FP32x2 operations
// of sm_100+ (1 = on; 0 = the scalar loop)
#ifndef NB_MIXED_PACKED
#define NB_MIXED_PACKED 1
#endif
#define NB_STR_(x) #x
#define NB_PRAGMA_UNROLL(n) _Pragma(NB_STR_(unroll n))

namespace nbk {

constexpr float kFarF = 1.0e15f;

// first j-tile of split s when `tiles` tiles are shared by S splits as evenly
// as possible (split sizes differ by at most one tile)
__device__ __forceinline__ int64_t split_begin(int64_t s, int64_t S, int64_t tiles) { return s * tiles / S; }

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

template <int JT>
struct MixedSmem {
  static constexpr bool kFused = false;
  float4 A[2][JT];
  float4 B[2][JT];
  float2 C[2][JT];
};

// ---- on-the-fly prediction of the j-particles (Sec. 4.4 step 4) -------------
// GRAPE predicts the j-particles on the board, in its pipelines, as they
// stream past; the host predicts only the n active i (step 3).  Here the
// force item can do the same: instead of a predicted j-store it loads the
// "j-memory" record of each particle, written from its FP64 state after every
// correction (rows in the resident order, 5 float4 rows of stride n_pad):
//   R0 = (xh, m)   R1 = (xl, Rd)   R2 = (vh, j6.x)   R3 = (vl, j6.y)   R4 = (a2, j6.z)
// with x = xh + xl and v = vh + vl the double-single splits of the FP64
// position and velocity, a2 = fl32(a/2), j6 = fl32(jerk/6), and Rd a bound
// on the distance the particle can move within its current step (the tile
// boxes of the far test are grown by it), plus its FP64 time t_j.  The item
// predicts the tile it has staged, to the block time T, into the same
// pair-interleaved shared tile the plain loader fills:
//   h = fl32(T - t_j)  (exact: a multiple of dt_min below dt_max),
//   xp = x + h (v + h (a/2 + h j/6))  in double-single FP32 (TwoSum and an
//        FMA-exact product carry the x + v h part to ~2^-48; the a and jerk
//        terms are FP32, so their rounding is 2^-24 |a h^2 / 2| at most),
//   vp = v + h (a + h j/2)  in FP32 (the mixed path's velocities are FP32).
template <int JT>
struct FusedSmem {
  static constexpr bool kFused = true;
  float4 R[2][5][JT];  // staged j-memory records (double-buffered)
  double T[2][JT];     // their times t_j
  float4 A[JT];        // the predicted tile, pair-interleaved (PairTile)
  float4 B[JT];
  float2 C[JT];
};

// Where an item's i-particles come from.  By default they are the j-store
// rows its list names (every particle's own predicted row).  For forces on
// particles held elsewhere -- the visiting block of the ring algorithm
// (Sec. 4.3), whose positions and velocities arrive from another rank -- the
// list indexes separate arrays instead, and self[k] gives the j-store slot of
// list position k's particle when this store holds it (else -1), which keeps
// the self pair excluded by index.
struct ISrc {
  const float4* __restrict__ A = nullptr;  // mixed: (x_hi, m), (x_lo, vx), (vy, vz) like jA/jB/jC
  const float4* __restrict__ B = nullptr;
  const float2* __restrict__ C = nullptr;
  const double* __restrict__ x = nullptr;  // FP64: SoA rows x[3][stride], v[3][stride]
  const double* __restrict__ v = nullptr;
  int64_t stride = 0;
  const int32_t* __restrict__ self = nullptr;
};

struct FusedArgs {
  const float4* __restrict__ jm = nullptr;  // R0..R4 rows, stride n_pad
  int64_t stride = 0;
  const double* __restrict__ tj = nullptr;  // FP64 times of the rows
  double T = 0.0;                           // block time
};

template <int NT, int JT>
__device__ __forceinline__ void mixed_load_tile(float4* sA, float4* sB, float2* sC, const float4* __restrict__ jA,
                                                const float4* __restrict__ jB, const float2* __restrict__ jC,
                                                int64_t j0, int64_t jhi) {
#pragma unroll
  for (int q = threadIdx.x; q < JT; q += NT) {
    const int64_t j = min(j0 + q, jhi - 1);
    cp_async16(&sA[q], &jA[j]);
    cp_async16(&sB[q], &jB[j]);
    cp_async8(&sC[q], &jC[j]);
  }
}

// Pair layout of one tile buffer for the packed loop: j-particles 2u and
// 2u+1 side by side, so that one 16-byte broadcast yields two (j, j+1) pairs:
//   P0[u] = (xh, xh', yh, yh')   P1[u] = (zh, zh', m, m')   (in sA)
//   P2[u] = (vx, vx', vy, vy')   P3[u] = (vz, vz', xl, xl') (in sB)
//   P4[u] = (yl, yl', zl, zl')                              (in sC)
// (u < JT/2; same 40 B per particle as the plain layout).  The float of
// particle q, pair slot (q & 1), sits at 4 (q >> 1) + (q & 1) (+2 for the
// second pair of a vector); 4-byte asynchronous copies scatter it there.
template <int JT>
struct PairTile {
  float *p0, *p1, *p2, *p3, *p4;
  __device__ __forceinline__ PairTile(float4* sA, float4* sB, float2* sC)
      : p0((float*)sA), p1((float*)(sA + JT / 2)), p2((float*)sB), p3((float*)(sB + JT / 2)), p4((float*)sC) {}
};

template <int NT, int JT>
__device__ __forceinline__ void mixed_load_tile_pairs(float4* sA, float4* sB, float2* sC,
                                                      const float4* __restrict__ jA,
                                                      const float4* __restrict__ jB,
                                                      const float2* __restrict__ jC, int64_t j0, int64_t jhi) {
  const PairTile<JT> t(sA, sB, sC);
#pragma unroll
  for (int q = threadIdx.x; q < JT; q += NT) {
    const int64_t j = min(j0 + q, jhi - 1);
    const float* a = (const float*)&jA[j];
    const float* b = (const float*)&jB[j];
    const float* c = (const float*)&jC[j];
    const int o = 4 * (q >> 1) + (q & 1);
    cp_async4(t.p0 + o, a + 0);
    cp_async4(t.p0 + o + 2, a + 1);
    cp_async4(t.p1 + o, a + 2);
    cp_async4(t.p1 + o + 2, a + 3);
    cp_async4(t.p2 + o, b + 3);
    cp_async4(t.p2 + o + 2, c + 0);
    cp_async4(t.p3 + o, c + 1);
    cp_async4(t.p3 + o + 2, b + 0);
    cp_async4(t.p4 + o, b + 1);
    cp_async4(t.p4 + o + 2, b + 2);
  }
}

template <int NT, int JT>
__device__ __forceinline__ void jm_load_tile(FusedSmem<JT>& sm, int buf, const FusedArgs& fa, int64_t j0,
                                             int64_t jhi) {
#pragma unroll
  for (int q = threadIdx.x; q < JT; q += NT) {
    const int64_t j = min(j0 + q, jhi - 1);
#pragma unroll
    for (int k = 0; k < 5; ++k) cp_async16(&sm.R[buf][k][q], &fa.jm[k * fa.stride + j]);
    cp_async8(&sm.T[buf][q], &fa.tj[j]);
  }
}

// x + delta in double-single: (xh, xl) + (p + q) with p + q = h (s + e) exact
// up to the rounding of e; TwoSum keeps the rounding error of xh + p.  The
// velocity: v + h (a + h j/2) = vh + 2h (a/2 + (3h/2) j/6) in FP32.  F2 is
// float (one coordinate) or float2 (two coordinates in the packed FP32x2
// operations, each lane rounded exactly as the scalar form).
__device__ __forceinline__ float p_add(float a, float b) { return a + b; }
__device__ __forceinline__ float p_sub(float a, float b) { return a - b; }
__device__ __forceinline__ float p_mul(float a, float b) { return a * b; }
__device__ __forceinline__ float p_fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float p_neg(float a) { return -a; }
__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 p_neg(float2 a) { return make_float2(-a.x, -a.y); }

template <typename F2>
__device__ __forceinline__ void ds_predict(F2 xh, F2 xl, F2 vh, F2 vl, F2 a2, F2 j6, F2 h, F2 h2, F2 h15,
                                           F2& hi, F2& lo, F2& vp) {
  const F2 u = p_fma(h, j6, a2);  // a/2 + h j/6
  const F2 hu = p_mul(h, u);
  F2 s = p_add(vh, hu);  // TwoSum(vh, hu)
  F2 bb = p_sub(s, vh);
  F2 e = p_add(p_sub(vh, p_sub(s, bb)), p_sub(hu, bb));
  e = p_add(e, vl);
  const F2 p = p_mul(h, s);  // h (s + e) = p + q, the product h s exact (FMA)
  F2 q = p_fma(h, s, p_neg(p));
  q = p_fma(h, e, q);
  const F2 S = p_add(xh, p);  // TwoSum(xh, p)
  bb = p_sub(S, xh);
  F2 E = p_add(p_sub(xh, p_sub(S, bb)), p_sub(p, bb));
  E = p_add(E, p_add(xl, q));
  hi = p_add(S, E);  // renormalise: |lo| <= ulp(hi) / 2
  lo = p_sub(E, p_sub(hi, S));
  vp = p_fma(h2, p_fma(h15, j6, a2), vh);
}

// predict the staged tile `buf` into the pair tile; slots past jhi become
// massless particles far away (every float written, so no stale shared
// memory is ever read)
template <int NT, int JT>
__device__ __forceinline__ void jm_predict_tile(FusedSmem<JT>& sm, int buf, double T, int64_t jt, int64_t jhi) {
  const PairTile<JT> pt(sm.A, sm.B, sm.C);
#pragma unroll
  for (int q = threadIdx.x; q < JT; q += NT) {
    const int o = 4 * (q >> 1) + (q & 1);
    float xh[3], xl[3], vv[3], m;
    if (jt + q < jhi) {
      const float4 r0 = sm.R[buf][0][q], r1 = sm.R[buf][1][q], r2 = sm.R[buf][2][q], r3 = sm.R[buf][3][q],
                   r4 = sm.R[buf][4][q];
      const float h = nb_f32(T - sm.T[buf][q]);
      const float h2 = 2.0f * h, h15 = 1.5f * h;  // exact scalings of an exact h
      float2 hi2, lo2, vp2;
      ds_predict(make_float2(r0.x, r0.y), make_float2(r1.x, r1.y), make_float2(r2.x, r2.y),
                 make_float2(r3.x, r3.y), make_float2(r4.x, r4.y), make_float2(r2.w, r3.w), make_float2(h, h),
                 make_float2(h2, h2), make_float2(h15, h15), hi2, lo2, vp2);
      ds_predict(r0.z, r1.z, r2.z, r3.z, r4.z, r4.w, h, h2, h15, xh[2], xl[2], vv[2]);
      xh[0] = hi2.x; xh[1] = hi2.y;
      xl[0] = lo2.x; xl[1] = lo2.y;
      vv[0] = vp2.x; vv[1] = vp2.y;
      m = r0.w;
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        xh[c] = kFarF;
        xl[c] = 0.0f;
        vv[c] = 0.0f;
      }
      m = 0.0f;
    }
    pt.p0[o] = xh[0];
    pt.p0[o + 2] = xh[1];
    pt.p1[o] = xh[2];
    pt.p1[o + 2] = m;
    pt.p2[o] = vv[0];
    pt.p2[o + 2] = vv[1];
    pt.p3[o] = vv[2];
    pt.p3[o + 2] = xl[0];
    pt.p4[o] = xl[1];
    pt.p4[o + 2] = xl[2];
  }
}

template <int JT>
__device__ __forceinline__ PairTile<JT> pair_tile(MixedSmem<JT>& sm, int buf) {
  return PairTile<JT>(sm.A[buf], sm.B[buf], sm.C[buf]);
}
template <int JT>
__device__ __forceinline__ PairTile<JT> pair_tile(FusedSmem<JT>& sm, int) {
  return PairTile<JT>(sm.A, sm.B, sm.C);
}

// One j-tile against the thread's IPT i-particles; FP32 partials in p.
// MODE: kFar  -- the tile is far from every i of the warp: hi parts alone
//                (r = x_j.hi - x_i.hi, within 2^-24 (|x_i|+|x_j|) of the exact
//                difference: relative error <= 2^-24 (1/theta + 1) at the
//                far-test distance);
//       kNear -- double-single difference;
//       kSelf -- double-single difference, pairs with j == i get 1/s = 0.
constexpr int kFar = 0, kNear = 1, kSelf = 2;
// far test: box gap >= theta * (|x|max_i + |x|max_j)
#ifndef NB_FAR_THETA
#define NB_FAR_THETA 0.125f
#endif
constexpr float kFarTheta = NB_FAR_THETA;

template <int IPT, int JT, int MODE>
__device__ __forceinline__ void mixed_tile_pass(const float4* __restrict__ sA, const float4* __restrict__ sB,
                                                const float2* __restrict__ sC, const float (&xh)[IPT][3],
                                                const float (&xl)[IPT][3], const float (&vi)[IPT][3],
                                                const int (&rel)[IPT], float eps2, float (&p)[IPT][7]) {
  NB_PRAGMA_UNROLL(NB_MIXED_UNROLL)
  for (int q = 0; q < JT; ++q) {
    const float4 A = sA[q];
    const float4 B = sB[q];
    const float2 C = sC[q];
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
      const float dx = MODE == kFar ? A.x - xh[k][0] : (A.x - xh[k][0]) + (B.x - xl[k][0]);
      const float dy = MODE == kFar ? A.y - xh[k][1] : (A.y - xh[k][1]) + (B.y - xl[k][1]);
      const float dz = MODE == kFar ? A.z - xh[k][2] : (A.z - xh[k][2]) + (B.z - xl[k][2]);
      const float wx = B.w - vi[k][0];
      const float wy = C.x - vi[k][1];
      const float wz = C.y - vi[k][2];
      const float r2 = fmaf(dz, dz, fmaf(dy, dy, fmaf(dx, dx, eps2)));
      const float rw = fmaf(dz, wz, fmaf(dy, wy, dx * wx));
#if NB_MIXED_NEWTON
      // hardware 1/sqrt + one Newton step: e = 1 - s^2 y0^2, y = y0 + y0 e / 2
      const float y0 = nb_rsqrt_approx(r2);
      const float e = fmaf(-r2, y0 * y0, 1.0f);
      float rinv = fmaf(0.5f, y0 * e, y0);
#else
      float rinv = nb_rsqrt_approx(r2);
#endif
      if (MODE == kSelf) rinv = (q == rel[k]) ? 0.0f : rinv;
      const float rinv2 = rinv * rinv;
      const float mr = A.w * rinv;
      const float mr3 = mr * rinv2;
      // jerk term formed before accumulation: u = w - 3 (r.w)/s^2 r; the two
      // parts cancel for close pairs, so they must not enter the sum apart
      const float a3 = (rw * -3.0f) * rinv2;
      p[k][6] += mr;
      p[k][0] = fmaf(mr3, dx, p[k][0]);
      p[k][1] = fmaf(mr3, dy, p[k][1]);
      p[k][2] = fmaf(mr3, dz, p[k][2]);
      p[k][3] = fmaf(mr3, fmaf(a3, dx, wx), p[k][3]);
      p[k][4] = fmaf(mr3, fmaf(a3, dy, wy), p[k][4]);
      p[k][5] = fmaf(mr3, fmaf(a3, dz, wz), p[k][5]);
    }
  }
}

// The same pass on the pair layout for IPT i per thread: every FP32
// operation acts on the pair (j, j+1) at once (packed FP32x2 add/mul/fma,
// each lane rounded exactly as its scalar counterpart), which halves the
// issue slots of the FP32 work.  ni* hold the NEGATED i coordinates and
// velocity in both lanes, so x_j + (-x_i) is the scalar x_j - x_i bit for
// bit.  The two lanes of p sum the even and the odd j of the tile.
template <int IPT, int JC, int MODE, int JT>
__device__ __forceinline__ void mixed_pair_pass(const PairTile<JT>& t, const float2 (&nxh)[IPT][3],
                                                const float2 (&nxl)[IPT][3], const float2 (&nv)[IPT][3],
                                                const int (&rel)[IPT], float2 eps2, float2 (&p)[IPT][7],
                                                int j0 = 0) {
  const float4* __restrict__ P0 = (const float4*)t.p0 + j0 / 2;
  const float4* __restrict__ P1 = (const float4*)t.p1 + j0 / 2;
  const float4* __restrict__ P2 = (const float4*)t.p2 + j0 / 2;
  const float4* __restrict__ P3 = (const float4*)t.p3 + j0 / 2;
  const float4* __restrict__ P4 = (const float4*)t.p4 + j0 / 2;
  const float2 m3 = make_float2(-3.0f, -3.0f);
  NB_PRAGMA_UNROLL(NB_MIXED_UNROLL)
  for (int u = 0; u < JC / 2; ++u) {
    const float4 a = P0[u], b = P1[u], c = P2[u], d = P3[u];
    float4 e;
    if (MODE != kFar) e = P4[u];
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
      float2 dx = __fadd2_rn(make_float2(a.x, a.y), nxh[k][0]);
      float2 dy = __fadd2_rn(make_float2(a.z, a.w), nxh[k][1]);
      float2 dz = __fadd2_rn(make_float2(b.x, b.y), nxh[k][2]);
      if (MODE != kFar) {
        dx = __fadd2_rn(dx, __fadd2_rn(make_float2(d.z, d.w), nxl[k][0]));
        dy = __fadd2_rn(dy, __fadd2_rn(make_float2(e.x, e.y), nxl[k][1]));
        dz = __fadd2_rn(dz, __fadd2_rn(make_float2(e.z, e.w), nxl[k][2]));
      }
      const float2 wx = __fadd2_rn(make_float2(c.x, c.y), nv[k][0]);
      const float2 wy = __fadd2_rn(make_float2(c.z, c.w), nv[k][1]);
      const float2 wz = __fadd2_rn(make_float2(d.x, d.y), nv[k][2]);
      const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __ffma2_rn(dx, dx, eps2)));
      const float2 rw = __ffma2_rn(dz, wz, __ffma2_rn(dy, wy, __fmul2_rn(dx, wx)));
#if NB_MIXED_NEWTON
      const float2 y0 = make_float2(nb_rsqrt_approx(r2.x), nb_rsqrt_approx(r2.y));
      const float2 ee = __ffma2_rn(make_float2(-r2.x, -r2.y), __fmul2_rn(y0, y0), make_float2(1.0f, 1.0f));
      float2 rinv = __ffma2_rn(make_float2(0.5f, 0.5f), __fmul2_rn(y0, ee), y0);
#else
      float2 rinv = make_float2(nb_rsqrt_approx(r2.x), nb_rsqrt_approx(r2.y));
#endif
      if (MODE == kSelf) {
        rinv.x = (2 * u == rel[k]) ? 0.0f : rinv.x;
        rinv.y = (2 * u + 1 == rel[k]) ? 0.0f : rinv.y;
      }
      const float2 rinv2 = __fmul2_rn(rinv, rinv);
      const float2 mr = __fmul2_rn(make_float2(b.z, b.w), rinv);
      const float2 mr3 = __fmul2_rn(mr, rinv2);
      const float2 a3 = __fmul2_rn(__fmul2_rn(rw, m3), rinv2);
      p[k][6] = __fadd2_rn(p[k][6], mr);
      p[k][0] = __ffma2_rn(mr3, dx, p[k][0]);
      p[k][1] = __ffma2_rn(mr3, dy, p[k][1]);
      p[k][2] = __ffma2_rn(mr3, dz, p[k][2]);
      p[k][3] = __ffma2_rn(mr3, __ffma2_rn(a3, dx, wx), p[k][3]);
      p[k][4] = __ffma2_rn(mr3, __ffma2_rn(a3, dy, wy), p[k][4]);
      p[k][5] = __ffma2_rn(mr3, __ffma2_rn(a3, dz, wz), p[k][5]);
    }
  }
}

// (hi, lo) += (bh, bl): double-single sum (Knuth's TwoSum of the high parts,
// the low parts and the rounding error added without renormalisation, as the
// items' per-tile fold)
__device__ __forceinline__ void ds_add(float& hi, float& lo, float bh, float bl) {
  const float s = hi + bh;
  const float bb = s - hi;
  lo = (lo + bl) + ((hi - (s - bb)) + (bh - bb));
  hi = s;
}

// Sum of 7 double-single rows over the P lanes of a group (a power of two, 8 to
// 32, lanes of one warp; every lane calls): the butterfly's sums, bit for bit,
// but each lane exchanges and keeps only half of its rows in the first three
// levels, so 9 or fewer pairs cross instead of 35 (7 log2 P).  Returns the row
// this lane holds (7: none), its sum in (h, l).
__device__ __forceinline__ int ds_sum_rows(const float (&hi)[7], const float (&lo)[7], int P, float& h, float& l) {
  const int lane = threadIdx.x & 31;
  const bool u1 = (lane & (P >> 1)) != 0, u2 = (lane & (P >> 2)) != 0, u3 = (lane & (P >> 3)) != 0;
  float a[4], b[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const float h4 = r < 3 ? hi[4 + (r < 3 ? r : 0)] : 0.0f, l4 = r < 3 ? lo[4 + (r < 3 ? r : 0)] : 0.0f;
    a[r] = u1 ? h4 : hi[r];
    b[r] = u1 ? l4 : lo[r];
    const float oh = __shfl_xor_sync(0xffffffffu, u1 ? hi[r] : h4, P >> 1);
    const float ol = __shfl_xor_sync(0xffffffffu, u1 ? lo[r] : l4, P >> 1);
    ds_add(a[r], b[r], oh, ol);
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const float oh = __shfl_xor_sync(0xffffffffu, u2 ? a[r] : a[2 + r], P >> 2);
    const float ol = __shfl_xor_sync(0xffffffffu, u2 ? b[r] : b[2 + r], P >> 2);
    a[r] = u2 ? a[2 + r] : a[r];
    b[r] = u2 ? b[2 + r] : b[r];
    ds_add(a[r], b[r], oh, ol);
  }
  const float oh = __shfl_xor_sync(0xffffffffu, u3 ? a[0] : a[1], P >> 3);
  const float ol = __shfl_xor_sync(0xffffffffu, u3 ? b[0] : b[1], P >> 3);
  h = u3 ? a[1] : a[0];
  l = u3 ? b[1] : b[0];
  ds_add(h, l, oh, ol);
  for (int o = P >> 4; o > 0; o >>= 1) {
    const float qh = __shfl_xor_sync(0xffffffffu, h, o), ql = __shfl_xor_sync(0xffffffffu, l, o);
    ds_add(h, l, qh, ql);
  }
  return (u1 ? 4 : 0) + (u2 ? 2 : 0) + (u3 ? 1 : 0);
}
// the lane of a group of P that ds_sum_rows leaves row r on (the lowest one)
__device__ __forceinline__ int ds_row_lane(int r, int P) {
  return ((r & 4) ? P >> 1 : 0) + ((r & 2) ? P >> 2 : 0) + ((r & 1) ? P >> 3 : 0);
}

// an FP64 value as a double-single pair: hi = fl32(x), lo = fl32(x - hi)
__device__ __forceinline__ float2 ds_split(double x) {
  const float hi = __double2float_rn(x);
  return make_float2(hi, __double2float_rn(x - (double)hi));
}

// Groups of threads that share the j of a tile (mixed_item's JG: 1, 2, 4 or 8,
// i-tiles of 128 / JG) for n i-particles on `tiles` j-tiles with room for R
// CTAs of 128 threads: the fewest thread slots, a slot costing 1, 1.08, 1.18 or
// 1.45 with the groups (the shorter the runs of j, the more of a tile's time is
// staging and folding: n = 2000 at N = 2^20 2018, 2165, 2363, 2884 us; n = 16
// 159, 101, 70, 55; n = 48 164, 104, 121, 109; n = 160 291, 243, 224, 265); then
// more while the items still fit one wave, as each is then only latency (n = 512
// on 2048 16.5 -> 14.5 us, 16 on 30000 25 -> 21).
__host__ __device__ __forceinline__ int j_groups(int64_t n, int64_t tiles, int64_t R) {
  constexpr int kCost[4] = {100, 108, 118, 145};
  int best = 0;
  int64_t work = 0;
  for (int k = 0; k < 4; ++k) {
    const int64_t w = ((n + (128 >> k) - 1) >> (7 - k)) * (128 >> k) * kCost[k];
    if (k == 0 || w < work) {
      best = k;
      work = w;
    }
  }
  while (best < 3 && ((n + (64 >> best) - 1) >> (6 - best)) * tiles <= R) ++best;
  return 1 << best;
}

// The same for the FP64 item, 1, 2, 4 or 8 groups and i-tiles of 128, 64, 32 or
// 16, a slot costing 1, 1.02, 1.04 or 1.17; without groups the warps past n
// compute nothing, so a partial i-tile counts 96 slots (120 behind whole tiles
// with three warps).  N = 200000, with 1, 2, 4, 8 groups, us: n = 16 229, 160, 142,
// 96; n = 48 288, 247, 258, 255; n = 80 362, 401, 357, 345; n = 128 433, 454, 456, 500;
// n = 160 683, 593, 551, 611; n = 320 1114, 1013, 1042, 1187; n = 1000 3039, 3121,
// 3243, 3739.  Two groups also while the items fit about one wave, four while they
// fit half of one (N = 20000, n = 96 79, 65, 59; N = 1500, n = 320 45, 35, 32; N = n =
// 1024 45, 42, 41).
__host__ __device__ __forceinline__ int j_groups64(int64_t n, int64_t tiles, int64_t sms) {
  constexpr int kCost[4] = {100, 102, 104, 117};
  const int64_t part = n & 127;
  int best = 0;
  int64_t work = 0;
  for (int k = 0; k < 4; ++k) {
    int64_t slots = ((n + (128 >> k) - 1) >> (7 - k)) * (128 >> k);
    if (k == 0 && part > 0 && part <= 96) slots += (part > 64 && n > 128 ? 120 : 96) - 128;
    if (k == 0 || slots * kCost[k] < work) {
      best = k;
      work = slots * kCost[k];
    }
  }
  for (int k = best + 1; k <= 2; ++k)
    if (((n + (128 >> k) - 1) >> (7 - k)) * tiles <= (k == 1 ? 5 : 2) * sms) best = k;
  return 1 << best;
}

// Mixed-precision item: i-tile starting at list position ibase (n entries in
// list, entries clamped to [0, idx_hi)), j-range [jlo, jhi).  Writes 7 rows
// out[c * ostride + pos] (final: acc, jerk, pot with its sign) or raw sums.
// With FusedSmem the j-tiles come from the j-memory (fa) and are predicted
// to fa.T as they are staged; the i-particles always come from jA/jB/jC.
//
// JG > 1 (few i-particles): the CTA takes NT / JG of them, and JG groups of
// threads share the j of each tile, JT / JG each, so that a block of a few
// particles does not leave most threads to recompute its last one; the groups'
// double-single sums are added in group order at the end.
template <int NT, int IPT, int JT, int JG = 1, typename SM>
__device__ __forceinline__ void mixed_item(SM& sm, const float4* __restrict__ jA,
                                           const float4* __restrict__ jB, const float2* __restrict__ jC,
                                           int64_t jlo, int64_t jhi, int64_t idx_hi,
                                           const int32_t* __restrict__ list, int64_t n, int64_t ibase,
                                           float eps2, double* __restrict__ out, int64_t ostride,
                                           bool finalize, const float4* __restrict__ tbox = nullptr,
                                           const int32_t* __restrict__ ord = nullptr, int64_t box_origin = 0,
                                           const FusedArgs fa = FusedArgs(), const ISrc is = ISrc(),
                                           bool ds_out = false) {
  constexpr bool kFusedLoad = SM::kFused;
  // list: j-store slots of the i-particles.  ord (optional): the list
  // positions in processing order (a caller's list visited in spatial
  // order); results always go to the list positions.  tbox (optional):
  // boxes of every NB_BOX_TILE slots from slot box_origin on (j-ranges start
  // at box_origin plus a multiple of JT), which allow the far-tile pass.
  constexpr int NI = NT / JG, JC = JT / JG;  // i-particles of the CTA (IPT = 1) and j of a group and tile
  static_assert(JG == 1 || (IPT == 1 && NB_MIXED_DS_FOLD && NB_MIXED_PACKED), "groups: one i per thread, packed loop");
  static_assert(sizeof(SM) >= (JG - 1) * 7 * NI * sizeof(float2), "room for the groups' sums");
  const int tid = threadIdx.x, il = JG == 1 ? tid : tid % NI, jg = JG == 1 ? 0 : tid / NI;
  float xh[IPT][3], xl[IPT][3], vi[IPT][3];
  int64_t self[IPT];
#if NB_MIXED_DS_FOLD
  // double-single accumulators: the per-tile FP32 partial is added with
  // Knuth's TwoSum in FP32 (no FP64 instruction in the loop at all)
  float acc_hi[IPT][7], acc_lo[IPT][7];
#elif NB_MIXED_SMEM_ACC
  // FP64 accumulators in shared memory: fewer registers, more resident warps
  __shared__ double s_acc[IPT * 7 * NT];
#define NB_ACC(k, c) s_acc[((k) * 7 + (c)) * NT + tid]
#else
  double acc[IPT][7];
#define NB_ACC(k, c) acc[k][c]
#endif
#if NB_MIXED_DS_FOLD
#define NB_ACC_ZERO(k, c) (acc_hi[k][c] = acc_lo[k][c] = 0.0f)
#define NB_ACC_ADD(k, c, val)                                   \
  do {                                                          \
    const float a_ = acc_hi[k][c], b_ = (val);                  \
    const float s_ = a_ + b_;                                   \
    const float bb_ = s_ - a_;                                  \
    acc_lo[k][c] += (a_ - (s_ - bb_)) + (b_ - bb_);             \
    acc_hi[k][c] = s_;                                          \
  } while (0)
#define NB_ACC_GET(k, c) (nb_f64(acc_hi[k][c]) + nb_f64(acc_lo[k][c]))
#define NB_ACC_DS(k, c) make_float2(acc_hi[k][c], acc_lo[k][c])
#else
#define NB_ACC_ZERO(k, c) (NB_ACC(k, c) = 0.0)
#define NB_ACC_ADD(k, c, val) (NB_ACC(k, c) += (double)(val))
#define NB_ACC_GET(k, c) NB_ACC(k, c)
#define NB_ACC_DS(k, c) ds_split(NB_ACC(k, c))
#endif
#pragma unroll
  for (int k = 0; k < IPT; ++k) {
    int64_t pos = ibase + k * NI + il;
    if (pos >= n) pos = n - 1;
    if (ord) pos = ord[pos];
    int64_t p = list[pos];
    float4 A, B;
    float2 C;
    if (is.A) {  // a particle held elsewhere: list positions index the i arrays (n long)
      p = p < 0 ? 0 : (p >= n ? n - 1 : p);
      A = is.A[p];
      B = is.B[p];
      C = is.C[p];
      self[k] = is.self ? is.self[pos] : -1;
    } else {
      p = p < 0 ? 0 : (p >= idx_hi ? idx_hi - 1 : p);  // a bad list never reads out of bounds
      self[k] = p;  // j-store slot of this i
      A = jA[p];
      B = jB[p];
      C = jC[p];
    }
    xh[k][0] = A.x; xh[k][1] = A.y; xh[k][2] = A.z;
    xl[k][0] = B.x; xl[k][1] = B.y; xl[k][2] = B.z;
    vi[k][0] = B.w; vi[k][1] = C.x; vi[k][2] = C.y;
#pragma unroll
    for (int c = 0; c < 7; ++c) NB_ACC_ZERO(k, c);
  }
  // box of this thread's i-particles (hi parts) and their largest
  // |coordinate|: the far test is taken per thread and the tile is far for
  // the warp when it is far for every lane (a warp of scattered particles,
  // as a small random block forms, still finds the tiles far from all of them)
  float wlo[3], whi[3], wr = 0.0f;
  if (tbox) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      wlo[c] = xh[0][c];
      whi[c] = xh[0][c];
#pragma unroll
      for (int k = 1; k < IPT; ++k) {
        wlo[c] = fminf(wlo[c], xh[k][c]);
        whi[c] = fmaxf(whi[c], xh[k][c]);
      }
      wr = fmaxf(wr, fmaxf(fabsf(wlo[c]), fabsf(whi[c])));
    }
  }

  // packed loop: each i-particle in both lanes, negated
  constexpr bool kPk = NB_MIXED_PACKED && IPT <= 2;
  static_assert(!kFusedLoad || kPk, "on-the-fly prediction fills the pair layout of the packed loop");
  float2 nxh[IPT][3], nxl[IPT][3], nv[IPT][3];
#pragma unroll
  for (int k = 0; k < IPT; ++k)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      nxh[k][c] = make_float2(-xh[k][c], -xh[k][c]);
      nxl[k][c] = make_float2(-xl[k][c], -xl[k][c]);
      nv[k][c] = make_float2(-vi[k][c], -vi[k][c]);
    }

  const int ntiles = (int)((jhi - jlo + JT - 1) / JT);
  if (ntiles > 0) {
    if constexpr (kFusedLoad)
      jm_load_tile<NT, JT>(sm, 0, fa, jlo, jhi);
    else if constexpr (kPk)
      mixed_load_tile_pairs<NT, JT>(sm.A[0], sm.B[0], sm.C[0], jA, jB, jC, jlo, jhi);
    else
      mixed_load_tile<NT, JT>(sm.A[0], sm.B[0], sm.C[0], jA, jB, jC, jlo, jhi);
  }
  cp_async_commit();

  for (int tile = 0; tile < ntiles; ++tile) {
    const int buf = tile & 1;
    const int64_t jt = jlo + (int64_t)tile * JT;
    if (tile + 1 < ntiles) {
      if constexpr (kFusedLoad)
        jm_load_tile<NT, JT>(sm, buf ^ 1, fa, jt + JT, jhi);
      else if constexpr (kPk)
        mixed_load_tile_pairs<NT, JT>(sm.A[buf ^ 1], sm.B[buf ^ 1], sm.C[buf ^ 1], jA, jB, jC, jt + JT, jhi);
      else
        mixed_load_tile<NT, JT>(sm.A[buf ^ 1], sm.B[buf ^ 1], sm.C[buf ^ 1], jA, jB, jC, jt + JT, jhi);
    }
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    if constexpr (kFusedLoad) {
      // predict the staged tile (ragged tail included) into the pair tile
      jm_predict_tile<NT, JT>(sm, buf, fa.T, jt, jhi);
      __syncthreads();
    } else if (jt + JT > jhi) {  // ragged last tile: massless far-away particles past jhi
      for (int q = tid; q < JT; q += NT) {
        if (jt + q < jhi) continue;
        if constexpr (kPk) {
          const PairTile<JT> pt(sm.A[buf], sm.B[buf], sm.C[buf]);
          const int o = 4 * (q >> 1) + (q & 1);
          pt.p0[o] = kFarF;
          pt.p0[o + 2] = kFarF;
          pt.p1[o] = kFarF;
          pt.p1[o + 2] = 0.0f;
        } else {
          sm.A[buf][q] = make_float4(kFarF, kFarF, kFarF, 0.0f);
        }
      }
      __syncthreads();
    }

    int rel[IPT];
    bool hit = false;
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
      const int64_t d = self[k] - (jt + jg * JC);
      rel[k] = (d >= 0 && d < JC) ? (int)d : -1;
      hit = hit || rel[k] >= 0;
    }
    float p[IPT][7];
#pragma unroll
    for (int k = 0; k < IPT; ++k)
#pragma unroll
      for (int c = 0; c < 7; ++c) p[k][c] = 0.0f;

    // far test: box gap >= theta (|x|max of the thread's i + |x|max of the
    // tile) bounds the hi-only difference error of each of its pairs by
    // 2^-24 (1/theta + 1); the warp takes the far pass when every lane passes.
    // Boxes cover NB_BOX_TILE slots: a longer tile needs all of its boxes
    // far, a shorter one uses the box that contains it.
    bool far = false;
    if (tbox) {
      constexpr int kBoxes = JT >= NB_BOX_TILE ? JT / NB_BOX_TILE : 1;
      far = true;
#pragma unroll
      for (int b = 0; b < kBoxes; ++b) {
        const int64_t t = (jt - box_origin) / NB_BOX_TILE + b;
        const float4 blo = tbox[2 * t], bhi = tbox[2 * t + 1];
        const float gx = fmaxf(0.0f, fmaxf(blo.x - whi[0], wlo[0] - bhi.x));
        const float gy = fmaxf(0.0f, fmaxf(blo.y - whi[1], wlo[1] - bhi.y));
        const float gz = fmaxf(0.0f, fmaxf(blo.z - whi[2], wlo[2] - bhi.z));
        const float lim = kFarTheta * (wr + blo.w);
        far = far && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) >= lim * lim;
      }
    }
    if constexpr (kPk) {
      const PairTile<JT> pt = pair_tile(sm, buf);
      const float2 e2 = make_float2(eps2, eps2);
      float2 p2[IPT][7];
#pragma unroll
      for (int k = 0; k < IPT; ++k)
#pragma unroll
        for (int c = 0; c < 7; ++c) p2[k][c] = make_float2(0.0f, 0.0f);
      if (__any_sync(0xffffffffu, hit))
        mixed_pair_pass<IPT, JC, kSelf>(pt, nxh, nxl, nv, rel, e2, p2, jg * JC);
      else if (__all_sync(0xffffffffu, far))
        mixed_pair_pass<IPT, JC, kFar>(pt, nxh, nxl, nv, rel, e2, p2, jg * JC);
      else
        mixed_pair_pass<IPT, JC, kNear>(pt, nxh, nxl, nv, rel, e2, p2, jg * JC);
#pragma unroll
      for (int k = 0; k < IPT; ++k)
#pragma unroll
        for (int c = 0; c < 7; ++c) p[k][c] = p2[k][c].x + p2[k][c].y;
    } else {
      if (__any_sync(0xffffffffu, hit))
        mixed_tile_pass<IPT, JT, kSelf>(sm.A[buf], sm.B[buf], sm.C[buf], xh, xl, vi, rel, eps2, p);
      else if (__all_sync(0xffffffffu, far))
        mixed_tile_pass<IPT, JT, kFar>(sm.A[buf], sm.B[buf], sm.C[buf], xh, xl, vi, rel, eps2, p);
      else
        mixed_tile_pass<IPT, JT, kNear>(sm.A[buf], sm.B[buf], sm.C[buf], xh, xl, vi, rel, eps2, p);
    }

#pragma unroll
    for (int k = 0; k < IPT; ++k)
#pragma unroll
      for (int c = 0; c < 7; ++c) NB_ACC_ADD(k, c, p[k][c]);
    __syncthreads();
  }
  cp_async_wait<0>();

#if NB_MIXED_DS_FOLD
  if constexpr (JG > 1) {
    float2* red = reinterpret_cast<float2*>(&sm);
    __syncthreads();  // no copy into the tiles is in flight
    if (jg > 0)
#pragma unroll
      for (int c = 0; c < 7; ++c) red[((jg - 1) * 7 + c) * NI + il] = NB_ACC_DS(0, c);
    __syncthreads();
    if (jg == 0)
#pragma unroll
      for (int q = 0; q < JG - 1; ++q)
#pragma unroll
        for (int c = 0; c < 7; ++c) {
          const float2 v = red[(q * 7 + c) * NI + il];
          ds_add(acc_hi[0][c], acc_lo[0][c], v.x, v.y);
        }
    __syncthreads();  // (another item may load its tiles)
  }
#endif

  // final results (one split): FP64 with the potential's sign; partial sums
  // of a split: FP64, or with ds_out the double-single pair (hi, lo) in the
  // same 8-byte slot (no FP64 instruction: the FP64 pipe issues a warp
  // instruction every 64 cycles per warp on this GPU), which the split
  // reduction sums in FP32
  float2* out2 = reinterpret_cast<float2*>(out);
#pragma unroll
  for (int k = 0; k < IPT; ++k) {
    int64_t pos = ibase + k * NI + il;
    if (pos >= n || jg > 0) continue;
    if (ord) pos = ord[pos];
    if (ds_out && !finalize) {
#pragma unroll
      for (int c = 0; c < 7; ++c) out2[c * ostride + pos] = NB_ACC_DS(k, c);
    } else {
#pragma unroll
      for (int c = 0; c < 6; ++c) out[c * ostride + pos] = NB_ACC_GET(k, c);
      out[6 * ostride + pos] = finalize ? -NB_ACC_GET(k, 6) : NB_ACC_GET(k, 6);
    }
  }
#undef NB_ACC
#undef NB_ACC_ZERO
#undef NB_ACC_ADD
#undef NB_ACC_GET
#undef NB_ACC_DS
}

// ---- FP64 path --------------------------------------------------------------
// Inputs, sums and results are FP64; the pair arithmetic runs in the fixed
// point of fx64.cuh, in no component less accurate than an FP64 evaluation of
// the same formulas and 4 times as fast on this GPU.  Pairs and tiles for which
// it would not be so are evaluated in FP64.
template <int NT, int JT>
struct Fp64Smem {
  // a j-particle of the tile: (X0, X1), (X2, V0), (V1, V2), (M + k, fractions of
  // X0 and X1), (of X2 and V0, of V1 and V2).  M is a multiple of 1024; k =
  // kOdd: not for the fixed-point pair (negative, subnormal or very small mass)
  longlong2 j[JT][5];
  double hi[7][NT], lo[7][NT];  // the thread's sums (TwoSum)
  int4 red[JT / 32][4];         // a warp's bounds: X and V, minima and maxima (keys), the mass; its slow j
  int4 box[3];                  // the tile's, high words on its grid
};
constexpr int kOdd = 64;
// a tile's pairs as an i sees them (fp64_view)
constexpr int kPlain = 0, kFine = 1, kNone = 2;

__device__ __forceinline__ int64_t words(uint32_t lo, uint32_t hi) { return (int64_t)(((uint64_t)hi << 32) | lo); }

// exponent e of the largest magnitude among values whose high words (sign
// cleared) have maximum w: |x| < 2^e (NaN, Inf: 1025)
__device__ __forceinline__ int exp_above(int w) { return (w >> 20) - 1022; }
__device__ __forceinline__ int abs_hi(double x) { return __double2hiint(x) & 0x7FFFFFFF; }
__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((e + 1023) << 20, 0); }  // e in [-1022, 1023]

// the key that orders double high words, and the magnitude's word from it
__device__ __forceinline__ int hi_key(double x) {
  const int h = __double2hiint(x);
  return h ^ ((h >> 31) & 0x7FFFFFFF);
}
__device__ __forceinline__ int abs_key(int k) { return k ^ (k >> 31); }
__device__ __forceinline__ double of_hi_key(int k) { return __hiloint2double(k ^ ((k >> 31) & 0x7FFFFFFF), 0); }

// x 2^sh (|x| 2^sh <= 2^60) as an integer and 32 fraction bits, from x's bits:
// a shift of the significand costs a tenth of the FP64 instructions
__device__ __forceinline__ int64_t to_fixed(double x, int sh, uint32_t& frac) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int E = (int)(b >> 52) & 0x7FF;
  const uint64_t f = ((b & 0x000FFFFFFFFFFFFFull) | (E ? 0x0010000000000000ull : 0ull)) << 11;
  const int r = max(3, min(1086 - (E ? E : 1) - sh, 95));
  const uint64_t hi = r < 64 ? f >> (r & 63) : 0ull;
  const uint32_t lo = r < 32 ? (uint32_t)(f << ((32 - r) & 63)) : (uint32_t)(f >> ((r - 32) & 63));
  if ((int64_t)b >= 0) {
    frac = lo;
    return (int64_t)hi;
  }
  frac = 0u - lo;
  return -(int64_t)hi - (lo != 0u ? 1 : 0);
}

// (hi, lo) += p: TwoSum (Knuth), hi + p = s + e exactly
__device__ __forceinline__ void sum_add(double& hi, double& lo, double p) {
  const double s = hi + p;
  const double bp = s - hi;
  lo += (hi - (s - bp)) + (p - bp);
  hi = s;
}

// the pairs of one i with the j-particles of the bits in mask (jt + bit), in
// FP64: those that the fixed-point pair leaves, a few (closer than its grid
// resolves, odd masses) or all of a tile (fp64_view).  state: calls with a few,
// kHighUsed once the high sums have been written; returns the new one.
constexpr int kHighUsed = 1 << 30;
template <int NT, int JT>
__device__ __noinline__ int fp64_pairs(Fp64Smem<NT, JT>& sm, const double* __restrict__ xp,
                                        const double* __restrict__ vp, const double* __restrict__ m, int64_t cs,
                                        int64_t js, int64_t jt, uint64_t mask, double x0, double x1, double x2,
                                        double v0, double v1, double v2, double eps2, int state) {
  const int count = __popcll(mask);
  double p[7];
#pragma unroll
  for (int c = 0; c < 7; ++c) p[c] = 0.0;
  while (mask) {
    const int64_t j = jt + (__ffsll((long long)mask) - 1);
    mask &= mask - 1ull;
    const double* xj = xp + j * js;
    const double* vj = vp + j * js;
    const double dx = xj[0] - x0, dy = xj[cs] - x1, dz = xj[2 * cs] - x2;
    const double wx = vj[0] - v0, wy = vj[cs] - v1, wz = vj[2 * cs] - v2;
    const double r2 = fma(dz, dz, fma(dy, dy, fma(dx, dx, eps2)));
    const double rw = fma(dz, wz, fma(dy, wy, dx * wx));
    const double rinv = nb_rsqrt_fp64(r2);
    const double rinv2 = rinv * rinv;
    const double mr = m[j] * rinv;
    const double mr3 = mr * rinv2;
    const double a3 = (rw * -3.0) * rinv2;  // jerk term formed before accumulation
    p[6] += mr;
    p[0] = fma(mr3, dx, p[0]);
    p[1] = fma(mr3, dy, p[1]);
    p[2] = fma(mr3, dz, p[2]);
    p[3] = fma(mr3, fma(a3, dx, wx), p[3]);
    p[4] = fma(mr3, fma(a3, dy, wy), p[4]);
    p[5] = fma(mr3, fma(a3, dz, wz), p[5]);
  }
  // Each FP64 instruction holds the warp for 64 cycles.  A few pairs: into the
  // low sum alone, and every eighth time that into the high one without error;
  // many: a TwoSum into the high sum, none for the first
  if (count <= 4) {
    state += 1;
    if ((state & 7) != 0) {
#pragma unroll
      for (int c = 0; c < 7; ++c) sm.lo[c][threadIdx.x] += p[c];
      return state;
    }
  }
#pragma unroll
  for (int c = 0; c < 7; ++c) {
    double hi = p[c], lo = 0.0;
    if (state != 0) {
      hi = sm.hi[c][threadIdx.x];
      lo = sm.lo[c][threadIdx.x];
      if (count <= 4) {
        const double q = lo;
        lo = 0.0;
        sum_add(hi, lo, q);
      }
      sum_add(hi, lo, p[c]);
    }
    sm.hi[c][threadIdx.x] = hi;
    sm.lo[c][threadIdx.x] = lo;
  }
  return state | kHighUsed;
}

// the integer sums into the thread's FP64 sums (first: those are still zero);
// cleared
template <int NT, int JT>
__device__ __forceinline__ void fp64_fold(Fp64Smem<NT, JT>& sm, nbx::Sums& a, bool first, int g, int gv, int em) {
#pragma unroll
  for (int c = 0; c < 7; ++c) {
    const int e = c < 3 ? em - 2 * g + nbx::kAccScale
                        : (c < 6 ? em - 3 * g + gv + nbx::kJerkScale : em - g + nbx::kPotScale);
    const double p = c < 6 ? nbx::to_double(a.f[c % 6], e) : nbx::to_double(a.p, e);
    if (first)
      sm.hi[c][threadIdx.x] = p;
    else
      sum_add(sm.hi[c][threadIdx.x], sm.lo[c][threadIdx.x], p);
  }
  a = nbx::Sums{};
}

template <bool SH, bool FINE, int NT, int JT>
__device__ __forceinline__ uint32_t fx64_chunk(const Fp64Smem<NT, JT>& sm, int q0, int count, int rel,
                                               const nbx::IFix& fi, nbx::Sums& a) {
  uint32_t left = 0u;
#pragma unroll 1
  for (int q = 0; q < count; ++q) {
    const longlong2* row = sm.j[q0 + q];
    const longlong2 A = row[0], B = row[1], C = row[2], K = row[3];
    nbx::JFix fj;
    fj.X[0] = A.x; fj.X[1] = A.y; fj.X[2] = B.x;
    fj.V[0] = B.y; fj.V[1] = C.x; fj.V[2] = C.y;
    fj.k = (int)K.x & 1023;
    fj.M = (uint64_t)K.x & ~1023ull;
    fj.xl[0] = (uint32_t)K.y;
    fj.xl[1] = (uint32_t)((uint64_t)K.y >> 32);
    if (FINE) {
      const longlong2 L = row[4];
      fj.xl[2] = (uint32_t)L.x;
      fj.vl[0] = (uint32_t)((uint64_t)L.x >> 32);
      fj.vl[1] = (uint32_t)L.y;
      fj.vl[2] = (uint32_t)((uint64_t)L.y >> 32);
    } else {
      fj.xl[2] = *reinterpret_cast<const uint32_t*>(&row[4]);
    }
    const bool ok = nbx::pair<SH, FINE>(fj, fi, (q0 + q == rel) | (fj.k == kOdd), a);
    left |= ok ? 0u : 1u << q;
  }
  return left;
}

// How i sees the tile.  The fixed point holds the components of a difference,
// and of the products with it, to a fraction of what the largest one needs, so
// a tile that is flat from i (every tile of a disc) would have its small ones in
// too few bits: from 2^-kFlat of the largest extent on the pair keeps the
// products' last bits (kFine), and from 2^-kThin on it goes to FP64 (kNone), as
// does a tile of which the grid resolves few pairs (a system far from the origin,
// a common velocity: those cost a pass of their own).  kFine too where most
// velocity differences are small against the grid's unit of speed, as for
// a common velocity or most of a tile's j moving at less than 2^-kSlow of the
// fastest (a hard binary among them).  An axis on which every coordinate is zero,
// and i's, has no differences: it is judged by its velocities, the other part of
// the jerk, if there are any.  The extents are lower bounds, from the box of the
// high words.
constexpr int kFlat = 6, kThin = 16, kSlow = 4;
template <int NT, int JT>
__device__ __forceinline__ int fp64_view(const Fp64Smem<NT, JT>& sm, const nbx::IFix& fi, int zero, int qn) {
  const int4 p = sm.box[0], q = sm.box[1], r = sm.box[2];
  const int lo[6] = {p.x, p.y, p.z, p.w, q.x, q.y}, hi[6] = {q.z, q.w, r.x, r.y, r.z, r.w};
  int e[6], most[2] = {0, 0};
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const int k = min(c < 3 ? fi.kx : fi.kv, 31);
    const int64_t own = c < 3 ? fi.X[c % 3] : fi.V[c % 3];
    const uint32_t frac = c < 3 ? fi.xl[c % 3] : fi.vl[c % 3];
    const int l = lo[c] >> k, h = hi[c] >> k, x = (int)(own >> 32);
    if (own != 0 || frac != 0u) zero &= ~(1 << c);
    e[c] = max(max(h - x, x - l) - (max(abs(l), abs(h)) >> 20) - 2, 0);  // (a high word: to 2^-20 of itself)
    most[c / 3] = max(most[c / 3], e[c]);
  }
  const float ext = (float)most[0];
  int slow = 0;
#pragma unroll
  for (int w = 0; w < (NT < JT ? NT : JT) / 32; ++w) slow += sm.red[w][3].y;
  bool fine = most[1] < 3 << 24 || 2 * slow >= qn;
  bool none = ext * ext < 16.0f * fi.rmin || (fi.wmin != 0 && most[1] < 4 * nbx::kWMin);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const bool zx = (zero >> c) & 1, zv = (zero >> (3 + c)) & 1;
    fine = fine || (!zx && e[c] < most[0] >> kFlat) || (!zv && e[3 + c] < most[1] >> kFlat);
    none = none || (zx ? !zv && e[3 + c] < most[1] >> kThin : e[c] < most[0] >> kThin);
  }
  return none ? kNone : (fine ? kFine : kPlain);
}

// FP64 item: one i per thread (i-tile of NT), j-range [jlo, jhi).  Component c
// of particle j lies at xp[c cs + j js] (rows of the j-store: cs = n_pad,
// js = 1; [N][3] arrays: cs = 1, js = 3); list entries are clamped to
// [0, idx_hi).
//
// Per tile the CTA puts JT j-particles on a common grid, 2^G above the tile's
// largest coordinate (and eps), 2^GV above its largest velocity component, EM
// the exponent of its largest mass.  The grid is kept while it stays within a
// factor 2 (mass: 8) of the tile's own, so that the sums, exact
// integers, are folded into FP64 every kFold pairs and not per tile.  It
// depends on the j-range alone and on nothing the other i of the CTA hold, so
// a particle's result does not depend on which particles share its item.
//
// JG > 1: groups of NT / JG threads (whole or half warps) share the j of each tile, as in
// mixed_item; their integer sums are on one grid and add exactly.  The pairs left
// to FP64 are added up group by group, unless in_order (items of a single tile),
// which gives the bits of JG = 1.
template <int NT, int JT, int JG = 1>
__device__ __forceinline__ void fp64_item(Fp64Smem<NT, JT>& sm, const double* __restrict__ xp,
                                          const double* __restrict__ vp, const double* __restrict__ m, int64_t cs,
                                          int64_t js, int64_t jlo, int64_t jhi, int64_t idx_hi,
                                          const int32_t* __restrict__ list, int64_t n, int64_t ibase, double eps2,
                                          double* __restrict__ out, int64_t ostride, bool finalize,
                                          const ISrc is = ISrc(), bool in_order = false) {
  static_assert(JT % 32 == 0 && NT % 32 == 0, "tiles of whole warps");
  constexpr int NI = NT / JG, JC = JT / JG;  // i-particles of the CTA, j of a group and tile
  static_assert(NI % 16 == 0 && (JG == 1 || JC <= 32), "groups of whole or half warps, a chunk of a tile each");
  constexpr int kPer = (JT + NT - 1) / NT;  // j-particles a thread stages
  const int tid = threadIdx.x, il = JG == 1 ? tid : tid % NI, jg = JG == 1 ? 0 : tid / NI;
  const int64_t pos0 = ibase + il;
  const int64_t pos = pos0 < n ? pos0 : n - 1;
  int64_t self = list[pos];
  const double *xi, *vi;  // this i's position and velocity, read again when its grid changes
  int64_t ics = cs;
  if (is.x) {  // a particle held elsewhere (see ISrc)
    self = self < 0 ? 0 : (self >= n ? n - 1 : self);
    xi = is.x + self;
    vi = is.v + self;
    ics = is.stride;
    self = is.self ? is.self[pos] : -1;
  } else {
    self = self < 0 ? 0 : (self >= idx_hi ? idx_hi - 1 : self);  // a bad list never reads out of bounds
    xi = xp + self * js;
    vi = vp + self * js;
  }
  const int exi = exp_above(max(abs_hi(xi[0]), max(abs_hi(xi[ics]), abs_hi(xi[2 * ics]))));
  const int evi = exp_above(max(abs_hi(vi[0]), max(abs_hi(vi[ics]), abs_hi(vi[2 * ics]))));
  // eps < 2^eeps
  const int eeps = (exp_above(abs_hi(eps2)) + 1) >> 1;
#pragma unroll
  for (int c = 0; c < 7; ++c) sm.hi[c][tid] = sm.lo[c][tid] = 0.0;
  nbx::Sums a = {};
  nbx::IFix fi = {};
  int G = 0, GV = 0, EM = 0, g = 0, gv = 0, filled = 0;  // grid of the tiles so far, this i's grid, pairs in a
  bool have = false, in_range = false, used = false;  // used: a may hold pairs
  int tile = 0, state = 0;
  bool skip = false;
  uint64_t left64 = 0ull;
  // a warp whose list positions all lie past n computes nothing (its
  // results are not written); it still loads its share of every j-tile
  const bool wact = ibase + (int64_t)(il & ~31) < n;

  for (int64_t jt = jlo; jt < jhi; jt += JT) {
    double jx[kPer][3], jv[kPer][3], jm[kPer];
    int b[13];  // keys: minima of X and V, maxima of X and V; the mass
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      b[c] = 0x7FFFFFFF;
      b[6 + c] = ~0x7FFFFFFF;
    }
    b[12] = 0;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int q = tid + u * NT;
      const int64_t j = jt + q;
      const bool in = q < JT && j < jhi;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        jx[u][c] = in ? xp[c * cs + j * js] : 0.0;
        jv[u][c] = in ? vp[c * cs + j * js] : 0.0;
        const int kx = hi_key(jx[u][c]), kv = hi_key(jv[u][c]);
        b[c] = min(b[c], in ? kx : 0x7FFFFFFF);
        b[3 + c] = min(b[3 + c], in ? kv : 0x7FFFFFFF);
        b[6 + c] = max(b[6 + c], in ? kx : ~0x7FFFFFFF);
        b[9 + c] = max(b[9 + c], in ? kv : ~0x7FFFFFFF);
      }
      jm[u] = in ? m[j] : 0.0;
      b[12] = max(b[12], abs_hi(jm[u]));
    }
    if (tid < JT) {  // (whole warps)
#pragma unroll
      for (int c = 0; c < 13; ++c)
        b[c] = c < 6 ? __reduce_min_sync(0xffffffffu, b[c]) : __reduce_max_sync(0xffffffffu, b[c]);
      if ((tid & 31) == 0) {
        sm.red[tid >> 5][0] = make_int4(b[0], b[1], b[2], b[3]);
        sm.red[tid >> 5][1] = make_int4(b[4], b[5], b[6], b[7]);
        sm.red[tid >> 5][2] = make_int4(b[8], b[9], b[10], b[11]);
        sm.red[tid >> 5][3].x = b[12];
      }
    }
    __syncthreads();  // the previous tile is done with, the bounds are there
#pragma unroll
    for (int w = 0; w < (NT < JT ? NT : JT) / 32; ++w) {
      const int4 r0 = sm.red[w][0], r1 = sm.red[w][1], r2 = sm.red[w][2];
      const int r[13] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w, r2.x, r2.y, r2.z, r2.w, sm.red[w][3].x};
#pragma unroll
      for (int c = 0; c < 13; ++c) b[c] = w == 0 ? r[c] : (c < 6 ? min(b[c], r[c]) : max(b[c], r[c]));
    }
    int wx = 0, wv = 0, zero = 0;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const int w = max(abs_key(b[c]), abs_key(b[6 + c]));
      if (c < 3)
        wx = max(wx, w);
      else
        wv = max(wv, w);
      zero |= w == 0 ? 1 << c : 0;
    }
    const int wm = b[12];
    const int gx = max(max(exp_above(wx), eeps), nbx::kExpLo), gw = max(exp_above(wv), nbx::kExpLo),
              gm = max(exp_above(wm), nbx::kExpLo);
    const bool tile_ok = gx <= nbx::kExpHi && gw <= nbx::kExpHi && gm <= nbx::kExpHi;
    const bool moved = !have || gx > G || gx < G - 1 || gw > GV || gw < GV - 1 || gm > EM || gm < EM - 3;
    if (tile_ok && (moved || filled + JT > nbx::kFold)) {
      if (used) {
        fp64_fold(sm, a, (state & kHighUsed) == 0, g, gv, EM);
        state |= kHighUsed;
        used = false;
      }
      filled = 0;
      if (moved) {
        G = gx;
        GV = gw;
        EM = gm;
        g = max(G, exi);
        gv = max(GV, evi);
        in_range = g <= nbx::kExpHi && gv <= nbx::kExpHi;
        fi.wmin = GV == nbx::kExpLo && evi == -1022 ? 0 : nbx::kWMin;
        fi.kx = min(g - G, 63);
        fi.kv = min(gv - GV, 63);
        if (in_range) {
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            fi.X[c] = to_fixed(xi[c * ics], 60 - g, fi.xl[c]);
            fi.V[c] = to_fixed(vi[c * ics], 60 - gv, fi.vl[c]);
          }
          const double e2 = eps2 * pow2d(56 - 2 * g);
          const uint64_t e2h = (uint64_t)e2;
          fi.e2[2] = (uint32_t)(e2h >> 32);
          fi.e2[1] = (uint32_t)e2h;
          fi.e2[0] = (uint32_t)((e2 - (double)e2h) * 4294967296.0);
          fi.e2f = (float)e2;
          fi.rmin = fmaxf(0x1p40f, fi.e2f * 0x1p-8f);
        }
        have = true;
      }
    }
    if (tile_ok) {
      if (tid < 12) {
        uint32_t f;
        int key = b[0];
#pragma unroll
        for (int c = 1; c < 12; ++c) key = tid == c ? b[c] : key;
        reinterpret_cast<int*>(sm.box)[tid] = (int)(to_fixed(of_hi_key(key), tid % 6 < 3 ? 60 - G : 60 - GV, f) >> 32);
      }
      int slow = 0;  // j of less than 2^-kSlow of the grid's speed
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int q = tid + u * NT;
        if (q < JT) {
          slow += jt + q < jhi &&
                  exp_above(max(abs_hi(jv[u][0]), max(abs_hi(jv[u][1]), abs_hi(jv[u][2])))) <= GV - kSlow;
          int64_t X[3], V[3];
          uint32_t xl[3], vl[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            X[c] = to_fixed(jx[u][c], 60 - G, xl[c]);
            V[c] = to_fixed(jv[u][c], 60 - GV, vl[c]);
          }
          const uint64_t mb = (uint64_t)__double_as_longlong(jm[u]);
          const int E = (int)(mb >> 52);  // with the sign: negative masses are odd
          const int k = EM - (E - 1022);
          const bool none = mb << 1 == 0;
          const bool odd = !none && (E < 1 || E > 2046 || k > nbx::kKMax);
          const uint64_t M = none || odd ? 0ull : ((mb & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 10;
          sm.j[q][0] = make_longlong2(X[0], X[1]);
          sm.j[q][1] = make_longlong2(X[2], V[0]);
          sm.j[q][2] = make_longlong2(V[1], V[2]);
          sm.j[q][3] = make_longlong2((int64_t)(M | (uint64_t)(none ? 0 : (odd ? kOdd : k))), words(xl[0], xl[1]));
          sm.j[q][4] = make_longlong2(words(xl[2], vl[0]), words(vl[1], vl[2]));
        }
      }
      if (tid < JT) {
        slow = __reduce_add_sync(0xffffffffu, slow);
        if ((tid & 31) == 0) sm.red[tid >> 5][3].y = slow;
      }
      filled += JT;
    }
    __syncthreads();
    if (!wact) continue;  // the next tile's barrier keeps the warp in step
    const int qn = (int)min((int64_t)JT, jhi - jt);
    const int64_t d = self - jt;
    const int rel = d >= 0 && d < qn ? (int)d : -1;
    const bool shifted = __any_sync(0xffffffffu, (fi.kx | fi.kv) != 0);
    // An i that left most pairs of a tile to FP64 (one of a small core in a tile
    // with a far particle, say) leaves all of the next ones, and a warp of such i
    // skips the fixed-point pass; tried again every 256 j.  Each i decides for
    // itself, from the j-range alone.
    if (tile++ % (256 / JT) == 0) skip = false;
    const int view = tile_ok && in_range && !skip ? fp64_view(sm, fi, zero, qn) : kNone;
    used = used || view != kNone;
    // (with groups every group takes one trip, of no pairs past a ragged tile's end)
    const int qe = JG == 1 ? qn : (jg + 1) * JC;
    int left_count = 0;
#pragma unroll 1
    for (int q0 = jg * JC; q0 < qe; q0 += 32) {
      const int count = JG == 1 ? min(32, qe - q0) : max(0, min(JC, qn - q0));
      uint32_t left = JG > 1 && count == 0 ? 0u : 0xffffffffu >> (32 - count);
      if (view == kPlain)
        left = shifted ? fx64_chunk<true, false>(sm, q0, count, rel, fi, a)
                       : fx64_chunk<false, false>(sm, q0, count, rel, fi, a);
      else if (view == kFine)
        left = shifted ? fx64_chunk<true, true>(sm, q0, count, rel, fi, a)
                       : fx64_chunk<false, true>(sm, q0, count, rel, fi, a);
      if (rel >= q0 && rel < q0 + 32) left &= ~(1u << (rel - q0));
      left_count += __popc(left);
      // up to 64 pairs a call
      left64 |= (uint64_t)left << (JG == 1 ? q0 & 32 : 0);
      if (left64 && (JG > 1 ? !in_order : (q0 & 32) || q0 + 32 >= qe)) {
        state = fp64_pairs(sm, xp, vp, m, cs, js, jt + (JG == 1 ? q0 & ~32 : q0), left64, xi[0], xi[ics], xi[2 * ics],
                           vi[0], vi[ics], vi[2 * ics], eps2, state);
        left64 = 0ull;
      }
    }
    skip = skip || (view != kNone && 4 * left_count >= 3 * (JG == 1 ? qn : JC));
  }
  if constexpr (JG > 1) {
    if (in_order) {  // all of an i's left pairs in one call, as without groups
      __syncthreads();  // the tile is done with
      uint64_t* left = reinterpret_cast<uint64_t*>(sm.j);
      left[tid] = left64 << (jg * JC);
      __syncthreads();
      if (jg == 0) {
        uint64_t all = 0ull;
#pragma unroll
        for (int q = 0; q < JG; ++q) all |= left[q * NI + il];
        if (all)
          state = fp64_pairs(sm, xp, vp, m, cs, js, jlo, all, xi[0], xi[ics], xi[2 * ics], vi[0], vi[ics],
                             vi[2 * ics], eps2, state);
      }
    }
    // the groups' sums to group 0: what they hold in FP64 (early folds, pairs
    // left to FP64; rare), then, through the same slots, the integer sums, which
    // are on one grid for all groups of an i and add exactly
    if (__syncthreads_or(jg > 0 && state != 0)) {
      // (a row of an i per thread: eight FP64 instructions a group)
      for (int t = tid; t < 7 * NI; t += NT) {
        const int c = t / NI, i = t % NI;
        double hi = sm.hi[c][i], lo = sm.lo[c][i];
#pragma unroll 1
        for (int q = 1; q < JG; ++q) {
          sum_add(hi, lo, sm.hi[c][q * NI + i]);
          lo += sm.lo[c][q * NI + i];
        }
        sm.hi[c][i] = hi;
        sm.lo[c][i] = lo;
      }
      state |= kHighUsed;
      __syncthreads();
    }
    if (jg > 0)
#pragma unroll
      for (int c = 0; c < 7; ++c) {
        const uint32_t w[4] = {c < 6 ? a.f[c % 6].w0 : a.p.w0, c < 6 ? a.f[c % 6].w1 : a.p.w1,
                               c < 6 ? a.f[c % 6].w2 : a.p.w2, c < 6 ? a.f[c % 6].w3 : 0u};
        sm.hi[c][tid] = __longlong_as_double(words(w[0], w[1]));
        sm.lo[c][tid] = __longlong_as_double(words(w[2], w[3]));
      }
    __syncthreads();
    if (jg == 0)
#pragma unroll
      for (int q = 1; q < JG; ++q)
#pragma unroll
        for (int c = 0; c < 7; ++c) {
          const uint64_t b = (uint64_t)__double_as_longlong(sm.hi[c][q * NI + il]);
          const uint64_t d = (uint64_t)__double_as_longlong(sm.lo[c][q * NI + il]);
          if (c < 6)
            nbx::add4(a.f[c % 6], (uint32_t)b, (uint32_t)(b >> 32), (uint32_t)d, (uint32_t)(d >> 32));
          else
            nbx::add3(a.p.w0, a.p.w1, a.p.w2, (uint32_t)b, (uint32_t)(b >> 32), (uint32_t)d);
        }
  }
  if (used && jg == 0) fp64_fold(sm, a, (state & kHighUsed) == 0, g, gv, EM);
  __syncthreads();  // the caller may reuse shared memory for its next item
  if (pos0 >= n || jg > 0) return;
#pragma unroll
  for (int c = 0; c < 6; ++c) out[c * ostride + pos0] = sm.hi[c][tid] + sm.lo[c][tid];
  const double w = sm.hi[6][tid] + sm.lo[6][tid];
  out[6 * ostride + pos0] = finalize ? -w : w;
}

// ---- split-j reduction --------------------------------------------------------
// Sums the partials part[split][7][stride] of n list positions into F (the
// sign of the potential applied here) and the caller's row-major outputs
// (each may be null).  T = float2: double-single partials of the mixed item,
// summed in FP32 and converted once per result; T = double: FP64 partials.
//
// CTA (32 x QL threads) = 32 consecutive positions of one row c; lane y sums
// splits y, y + QL, ... in order, loaded kB at a time (one round trip per
// batch), then a fixed pairwise tree over the lanes: the result depends only
// on the number of splits, which alone chooses QL (launch_split_reduce).
// What bounds it is the latency of the partials, in L2, and for large n the
// bookkeeping of the tree: with 32 lanes for every split count 20 splits of
// n = 32768 took 46 us, with 4 lanes 12 us (the tree of 32 lanes is five
// barriers for less than one load per lane); 760 splits of n = 256 want the 32
// (13 us), and 235 of n = 1001, summed by one thread per position, took 359 us
// against 12.
__device__ __forceinline__ void part_add(float2& a, float2 b) { ds_add(a.x, a.y, b.x, b.y); }
__device__ __forceinline__ void part_add(double& a, double b) { a += b; }
__device__ __forceinline__ double part_value(float2 a) { return nb_f64(a.x) + nb_f64(a.y); }
__device__ __forceinline__ double part_value(double a) { return a; }

template <typename T, int QL>
__global__ void __launch_bounds__(32 * QL) split_reduce_kernel(const T* __restrict__ part, int64_t stride, int nsplit,
                                                               int64_t n, double* __restrict__ F, int64_t fstride,
                                                               double* __restrict__ acc, double* __restrict__ jerk,
                                                               double* __restrict__ pot) {
  constexpr int kB = 8;
  __shared__ T sm[QL][33];
  const int tx = threadIdx.x, ty = threadIdx.y, c = blockIdx.y;
  for (int64_t k0 = (int64_t)blockIdx.x * 32; k0 < n; k0 += (int64_t)gridDim.x * 32) {
    const int64_t k = k0 + tx;
    T s = T();
    if (k < n) {
      const T* src = part + (int64_t)c * stride + k;
      const int64_t step = (int64_t)QL * 7 * stride;  // QL splits further on
      int q = ty;
      for (; q + (kB - 1) * QL < nsplit; q += kB * QL) {
        T v[kB];
#pragma unroll
        for (int b = 0; b < kB; ++b) v[b] = src[(int64_t)q * 7 * stride + b * step];
#pragma unroll
        for (int b = 0; b < kB; ++b) part_add(s, v[b]);
      }
#pragma unroll 4
      for (; q < nsplit; q += QL) part_add(s, src[(int64_t)q * 7 * stride]);
    }
    sm[ty][tx] = s;
    __syncthreads();
#pragma unroll
    for (int h = QL / 2; h > 0; h >>= 1) {
      if (ty < h) {
        T a = sm[ty][tx];
        part_add(a, sm[ty + h][tx]);
        sm[ty][tx] = a;
      }
      __syncthreads();
    }
    if (ty == 0 && k < n) {
      const double w = part_value(sm[0][tx]);
      const double val = c == 6 ? -w : w;
      if (F) F[c * fstride + k] = val;
      if (c < 3) {
        if (acc) acc[3 * k + c] = val;
      } else if (c < 6) {
        if (jerk) jerk[3 * k + (c - 3)] = val;
      } else if (pot) {
        pot[k] = val;
      }
    }
    __syncthreads();
  }
}

template <typename T>
cudaError_t launch_split_reduce(const T* part, int64_t stride, int nsplit, int64_t n, double* F, int64_t fstride,
                                double* acc, double* jerk, double* pot, int sm_count, cudaStream_t stream) {
  const int64_t cols = (n + 31) / 32;
  const dim3 grid((unsigned)(cols < (int64_t)sm_count * 16 ? cols : (int64_t)sm_count * 16), 7);
  if (nsplit >= 32)
    split_reduce_kernel<T, 32><<<grid, dim3(32, 32), 0, stream>>>(part, stride, nsplit, n, F, fstride, acc, jerk, pot);
  else
    split_reduce_kernel<T, 4><<<grid, dim3(32, 4), 0, stream>>>(part, stride, nsplit, n, F, fstride, acc, jerk, pot);
  return cudaGetLastError();
}

}  // namespace nbk
