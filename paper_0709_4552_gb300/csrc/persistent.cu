// persistent.cu -- the block-step loop of one system (Sec. 4.1 steps 2-5) as
// one cooperative launch: every CTA stays resident for the whole run and the
// steps are separated by grid barriers instead of kernel boundaries.  Below
// N ~ 10^4 a block step does a few microseconds of arithmetic, and a
// launch per kernel (host loop) or a graph node per kernel (graph loop) costs
// more than the work; here a step costs three barriers.
//
// Rows are cut into 128-row tiles; CTA b of G owns the contiguous tiles
// [b T / G, (b + 1) T / G).  Per block step:
//   phase 1 (after barrier A): every CTA reads the G published slice minima
//     of t_i + dt_i with their counts and takes the block time t (step 2) and
//     its own offset in the active list; it writes its own active rows there
//     (ascending), predicts its own rows to t (step 3) and, on the mixed path
//     in spatial order, computes the boxes of its own tiles.    -> barrier B
//   phase 2: force items (i-tile of 128 list positions, fewer on the mixed
//     path when groups of threads share a tile's j, x j-split; step 4,
//     Eq. 3), the first by the CTA's place in an order that fills the SMs
//     evenly, the others from a work counter; the same items as the
//     host-driven kernels, split partials as double-single pairs. -> barrier C
//   phase 3: every CTA sums the j-splits of its own list positions in a fixed
//     order (double-single FP32), corrects them and picks their new steps
//     (step 5; own rows' due times kept in shared memory), then publishes the
//     minimum of t_i + dt_i over its rows and how many rows reach it; a block
//     time that does not increase stops the loop (no valid steps).
//                                                                 -> barrier A
// The active block is exactly the rows at the global minimum, so a CTA whose
// own minimum is larger has none, and the counts published with the minima
// give every CTA its list offset without a further barrier.
//
// Barriers count arrivals over the whole launch; each wait is bounded in
// time and polls, after which the CTA raises the timeout bit and an abort
// flag that makes every other CTA leave at its next wait.
#include <float.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "force_common.cuh"
#include "hermite.cuh"

namespace {

constexpr int kLT = 128;                     // threads per CTA = i-tile = row tile
constexpr int kLWarps = kLT / 32;
// resident CTAs per SM asked for.  Mixed: 4 (128 registers, a few spilled) where
// the force phase is the longest part of a step, 2 (no spills) where its
// latencies are (us a block step, 4 / 2: N = 4096 20.0 / 17.4, N = 12000 29.1 /
// 26.6, N = 32768 61.6 / 56.2, N = 40000 75.3 / 74.9, N = 60000 131.6 / 138.4, N =
// 65536 155.1 / 163.2).  FP64: 3 (168; with 4 the fixed-point pair spills: N =
// 1024 34.8 against 32.2 us a block step, N = 8192 81.9 against 75.5, N = 32768
// 641 against 640)
constexpr int kLPerSmMixed = 4, kLPerSmMixedSmall = 2, kLPerSm64 = 3;
constexpr int64_t kLMixedSmallHi = 32768, kLMixedTwoLo = 1024;
// j-tiles (the mixed one = the box tile).  FP64: an item's tile is its share of
// a small system's force phase, so those take 32 and at least two CTAs per SM:
// N = 1024 32.2 us a block step against 42.9 with 64 on the same grid (45.2 on
// the mixed path's; with one shared step 52.1, 49.7 and 125), N = 4096 46.9
// against 55.3 (80.3), N = 8192 75.5 against 79.8 (101); from N = 16384 the
// splits are long and 64 stages better (193 against 205).
constexpr int kLMixJT = 128, kLF64JT = 64, kLF64JTSmall = 32;
// (Up to two tiles of 64, N = 128, every loop driver splits the sums alike and
// gives the same bits.)
constexpr int64_t kLF64SmallLo = 2 * kLF64JT, kLF64SmallHi = 8192;
constexpr long long kWaitNs = 4000000000LL;  // a barrier wait of the loop gives up after 4 s
constexpr unsigned int kPollCap = 1u << 26;  // ... or after this many polls
constexpr unsigned long long kInfBits = 0x7FF0000000000000ULL;  // +inf
// force items per step: about this many per CTA.  Mixed, us a block step with 2,
// 3, 4, 6: N = 24000 40.0, 39.5, 39.5, 39.8; N = 40000 76.2, 75.4, 75.8, 77.0.
// FP64 with 2 and 4: N = 4096 46.9, 47.1; N = 16384 193, 193; N = 32768 640, 600.
constexpr int kLItemWavesMixed = 3, kLItemWaves64 = 2;
constexpr int64_t kLMaxSplits = 256;         // ... in at most this many j-splits
constexpr int kMaxSmid = 1024;               // SM ids counted by the CTA placement
constexpr int kMaxRank = 32;                 // CTAs an SM can hold

struct LoopCtl {
  unsigned long long bar;   // barrier arrivals in this launch
  unsigned long long wq;    // force-item counter of the current step
  unsigned int ranks[kMaxRank];   // CTAs of each rank on their SM
  unsigned int smrank[kMaxSmid];  // CTAs placed on each SM so far
  unsigned int abort;       // a CTA gave up waiting: every CTA leaves
  unsigned int more;        // the launch stopped after seg_steps steps
  long long steps;          // block steps taken
  long long interactions;   // sum of n N over the steps
};

struct LoopArgs {
  int64_t N, n_pad;
  double eps2;
  float eps2f;
  double eta, dt_min, dt_max, t_end;
  long long max_steps, seg_steps;
  const double* m;
  double *x, *v, *a, *jk, *pot, *t, *dt;
  double *xp, *vp;
  float4 *jA, *jB;
  float2* jC;
  float4* tbox;  // boxes of the 128-row tiles (mixed path in spatial order) or null
  int32_t* act;
  double *F, *part;
  int64_t part_elems;
  unsigned long long* smin;  // [G] slice minimum of t_i + dt_i (bit pattern)
  int32_t* scnt;             // [G] rows of the slice at that minimum
  LoopCtl* ctl;
  nb_dev_status* st;
};

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void red_release_add_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ long long globaltimer_ns() {
  long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier of G co-resident CTAs.  The k-th barrier of a launch is
// complete when the arrival count reaches k G.  Ordering: the CTA barrier
// orders every thread's writes before thread 0's gpu-scope release add
// (cumulative), and thread 0's acquire load before every thread's later
// reads.  Returns false when this CTA must leave (another CTA gave up, or
// this one waited longer than wait_ns).  In two parts, for work that passes
// between the arrival and the wait.
__device__ __forceinline__ void grid_arrive(LoopCtl* ctl, unsigned long long& epoch) {
  __syncthreads();
  if (threadIdx.x == 0) {
    epoch += 1;
    red_release_add_u64(&ctl->bar, 1ULL);
  }
}

__device__ bool grid_wait(LoopCtl* ctl, unsigned long long epoch, unsigned int G, nb_dev_status* st, int* s_ok,
                          long long wait_ns = kWaitNs) {
  if (threadIdx.x == 0) {
    const unsigned long long target = epoch * (unsigned long long)G;
    int ok = 1;
    const long long t0 = globaltimer_ns();
    unsigned int polls = 0;
    // the counter alone in the common path; the abort flag and the clock
    // every 16th poll (one L2 round trip per poll instead of two)
    while (ld_acquire_u64(&ctl->bar) < target) {
      if ((++polls & 15u) != 0u) continue;
      if (*(volatile unsigned int*)&ctl->abort) {
        ok = 0;
        break;
      }
      if (polls >= kPollCap || globaltimer_ns() - t0 > wait_ns) {
        atomicOr(&ctl->abort, 1u);
        atomicOr(&st->flags, NB_ST_TIMEOUT);
        ok = 0;
        break;
      }
      __nanosleep(32);
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

__device__ __forceinline__ bool grid_barrier(LoopCtl* ctl, unsigned long long& epoch, unsigned int G,
                                             nb_dev_status* st, int* s_ok, long long wait_ns = kWaitNs) {
  grid_arrive(ctl, epoch);
  return grid_wait(ctl, epoch, G, st, s_ok, wait_ns);
}

// (minimum, count at the minimum) combine
__device__ __forceinline__ void min_count(unsigned long long& v, int& c, unsigned long long ov, int oc) {
  if (ov < v) {
    v = ov;
    c = oc;
  } else if (ov == v) {
    c += oc;
  }
}

constexpr int kLDue = 512;  // own rows whose due times a CTA keeps in shared memory
constexpr int kOwn = 128;   // own active rows it keeps there

struct LoopSmem {
  // own rows' next due time t_i + dt_i (bit pattern), kept by the corrector
  // when the CTA owns at most kLDue rows (else read from the state)
  unsigned long long due[kLDue];
  int own[kOwn];           // own active rows (from the CTA's first), list order
  int rank;                // this CTA's rank among the CTAs on its SM
  int place;               // its place in the order of force items
  int item;
  unsigned long long wv[kLWarps];
  int wc[kLWarps];
  long long ws[2][kLWarps];
  nb_box wbox[kLWarps];
  unsigned long long tnb;  // block time (bit pattern)
  long long before, total;
  int mine;                // this CTA has active rows this step
  int mycnt;
  int ok;
};

// due time of own row i (bit pattern)
__device__ __forceinline__ unsigned long long due_of(const LoopArgs& p, const LoopSmem& s, int64_t i, int64_t r0,
                                                     bool cached) {
  return cached ? s.due[i - r0] : (unsigned long long)__double_as_longlong(p.t[i] + p.dt[i]);
}

// minimum of t_i + dt_i over rows [r0, r1) and the number of rows at it,
// published for the other CTAs (positive doubles order like their bits)
__device__ void publish_slice(const LoopArgs& p, int64_t r0, int64_t r1, LoopSmem& s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool cached = r1 - r0 <= kLDue;
  unsigned long long best = kInfBits;
  int cnt = 0;
  for (int64_t i = r0 + threadIdx.x; i < r1; i += kLT) min_count(best, cnt, due_of(p, s, i, r0, cached), 1);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long ov = __shfl_xor_sync(0xffffffffu, best, o);
    const int oc = __shfl_xor_sync(0xffffffffu, cnt, o);
    min_count(best, cnt, ov, oc);
  }
  if (lane == 0) {
    s.wv[warp] = best;
    s.wc[warp] = cnt;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kLWarps; ++w) min_count(best, cnt, s.wv[w], s.wc[w]);
    p.smin[blockIdx.x] = best;
    p.scnt[blockIdx.x] = cnt;
  }
}

// block time, total active count and this CTA's offset from the published
// slices (every CTA reads the same values, so every CTA decides alike)
constexpr int kLMaxG = 1024;  // CTAs a launch may have (slices read per thread below)
__device__ void read_slices(const LoopArgs& p, unsigned int G, LoopSmem& s) {
  constexpr int kPer = kLMaxG / kLT;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long* smin = reinterpret_cast<const long long*>(p.smin);
  unsigned long long v[kPer];
  int c[kPer];
  unsigned long long best = kInfBits;
#pragma unroll
  for (int u = 0; u < kPer; ++u) {  // one round of loads: minima and counts together
    const unsigned int q = threadIdx.x + u * kLT;
    v[u] = q < G ? (unsigned long long)__ldcg(smin + q) : kInfBits;
    c[u] = q < G ? __ldcg(p.scnt + q) : 0;
    best = v[u] < best ? v[u] : best;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long ov = __shfl_xor_sync(0xffffffffu, best, o);
    best = ov < best ? ov : best;
  }
  if (lane == 0) s.wv[warp] = best;
  __syncthreads();
  best = s.wv[0];
#pragma unroll
  for (int w = 1; w < kLWarps; ++w) best = s.wv[w] < best ? s.wv[w] : best;
  long long tot = 0, before = 0;
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const unsigned int q = threadIdx.x + u * kLT;
    if (v[u] == best) {
      tot += c[u];
      if (q < blockIdx.x) before += c[u];
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    tot += __shfl_xor_sync(0xffffffffu, tot, o);
    before += __shfl_xor_sync(0xffffffffu, before, o);
  }
  if (lane == 0) {
    s.ws[0][warp] = tot;
    s.ws[1][warp] = before;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kLWarps; ++w) {
      tot += s.ws[0][w];
      before += s.ws[1][w];
    }
    s.tnb = best;
    s.total = tot;
    s.before = before;
    const unsigned long long mv = (unsigned long long)__ldcg(smin + blockIdx.x);
    s.mine = mv == best;
    s.mycnt = s.mine ? __ldcg(p.scnt + blockIdx.x) : 0;
  }
  __syncthreads();
}

// this CTA's active rows, ascending, to act[before ...]
__device__ void write_active(const LoopArgs& p, int64_t r0, int64_t r1, unsigned long long tnb, long long base,
                             LoopSmem& s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool cached = r1 - r0 <= kLDue;
  for (int64_t r = r0; r < r1; r += kLT) {
    const int64_t i = r + threadIdx.x;
    const bool on = i < r1 && due_of(p, s, i, r0, cached) == tnb;
    const unsigned int ball = __ballot_sync(0xffffffffu, on);
    if (lane == 0) s.wc[warp] = __popc(ball);
    __syncthreads();
    int pre = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kLWarps; ++w) {
      pre += w < warp ? s.wc[w] : 0;
      all += s.wc[w];
    }
    if (on) {
      const long long k = base + pre + __popc(ball & ((1u << lane) - 1u));
      p.act[k] = (int32_t)i;
      if (k - s.before < kOwn) s.own[k - s.before] = (int)(i - r0);
    }
    base += all;
    __syncthreads();
  }
}

// predictor of this CTA's rows to tn; on the mixed path in spatial order the
// box of each 128-row tile (thread q holds row q of every tile it visits)
template <bool MIXED>
__device__ void predict_rows(const LoopArgs& p, int64_t r0, int64_t r1, double tn, LoopSmem& s) {
  static_assert(kLT == NB_BOX_TILE, "a tile of rows per pass");
  for (int64_t r = r0; r < r1; r += kLT) {
    const int64_t i = r + threadIdx.x;
    float hi[3] = {0.0f, 0.0f, 0.0f};
    if (i < r1) {
      double px[3], pv[3];
      nbh::taylor(i, p.n_pad, tn - p.t[i], p.x, p.v, p.a, p.jk, px, pv);
      nbh::store_predicted(i, p.n_pad, px, pv, p.m[i], p.xp, p.vp, p.jA, p.jB, p.jC, true, MIXED, hi);
    }
    if (MIXED && p.tbox) {
      const nb_box b = nb_warp_box(i < r1, hi);
      if ((threadIdx.x & 31) == 0) s.wbox[threadIdx.x >> 5] = b;
      __syncthreads();
      if (threadIdx.x == 0) nb_write_box(s.wbox, kLWarps, p.tbox + 2 * (r / kLT));
      __syncthreads();
    }
  }
}

// groups of threads that share the j of an item's tile (a step's i-tile is kLT
// divided by them), and the i-tiles.  (FP64: none, as the item's two more forms
// cost the loop registers: N = 1024 with one shared step 51.9 -> 61.3 us, N =
// 8192 75.2 -> 77.3, against 31.9 -> 28.9 for the small blocks of N = 1024 and
// 47.0 -> 46.4 at N = 4096.)
template <bool MIXED>
__device__ __forceinline__ int loop_groups(int64_t n, int64_t jtiles, unsigned int G) {
  return MIXED ? nbk::j_groups(n, jtiles, G) : 1;
}
__device__ __forceinline__ int64_t loop_itiles(int64_t n, int groups) {
  const int ni = kLT / groups;
  return (n + ni - 1) / ni;
}

// split-j factor of a step: a few force items per CTA (taken
// from a counter, so uneven items even out), at least one j-tile per split,
// at most kLMaxSplits splits (their sums are the corrector phase's loads),
// within the partial-sum scratch
template <bool MIXED>
__device__ __forceinline__ int64_t loop_splits(int64_t n, int64_t nI, int64_t jtiles, unsigned int G,
                                               int64_t part_elems) {
  int64_t S = ((int64_t)(MIXED ? kLItemWavesMixed : kLItemWaves64) * G + nI - 1) / nI;
  if (S > jtiles) S = jtiles;
  if (S > kLMaxSplits) S = kLMaxSplits;
  const int64_t cap = part_elems / (7 * (((n + 31) / 32) * 32));
  if (S > cap) S = cap;
  return S < 1 ? 1 : S;
}

// The own list positions are corrected up to round_of(mycnt) at a time: L =
// kLT / P' threads per position (P' = the round's positions rounded up to a
// power of two, at least 4), of which this thread is lane l of position q.
// Up to 64 positions: 32 a round, which lanes 0-3 correct together (the
// correction's FP64 chain is on the critical path of a step); more: one or two
// threads each, as the FP64 unit is then busy anyway (N = 1024 in FP64, every
// particle at every step: 52.1 us a step against 60.5 in rounds of 32).
__device__ __forceinline__ int round_of(int mycnt) { return mycnt <= 64 ? 32 : kLT; }
struct OwnRow {
  int L, l, q;
  bool have;       // position q exists in this round
  int64_t i;       // its row (without a position: some own row, read only)
  nbh::CorrIn in;  // L >= 4: what the correction reads of the row itself
};

__device__ __forceinline__ OwnRow own_row(const LoopArgs& p, const LoopSmem& s, int k0, int64_t r0) {
  OwnRow o;
  const int P = min(s.mycnt - k0, round_of(s.mycnt));
  int Pp = 4;
  while (Pp < P) Pp <<= 1;
  o.L = kLT / Pp;
  o.q = threadIdx.x / o.L;
  o.l = threadIdx.x % o.L;
  o.have = o.q < P;
  o.i = r0;
  o.in = nbh::CorrIn{};
  if (P <= 0) return o;
  const int k = k0 + (o.have ? o.q : 0);
  o.i = k < kOwn ? r0 + s.own[k] : (int64_t)p.act[s.before + k];
  if (o.L >= 4) {
    const int64_t c = (o.l < 3 ? o.l : 0) * p.n_pad + o.i;
    o.in = nbh::CorrIn{p.t[o.i], p.dt[o.i], p.a[c], p.jk[c], p.xp[c], p.vp[c]};
  }
  return o;
}

// phase 3 of a step: the j-split sums and the corrector (Sec. 4.1 step 5) of
// this CTA's own list positions [before, before + mycnt): in each round the
// lanes of a position sum its j-splits (lane l takes splits l, l + L, ... in
// order; a butterfly over the L lanes) and correct it.  `first`: the first
// round's rows, read before the forces were complete.  The active rows crowd in
// the CTAs that own a system's core, so a step waits for one CTA's L2 round
// trips: the loads of U splits are in flight per lane.
template <bool MIXED, int U, bool FIRST>
__device__ void correct_own(const LoopArgs& p, LoopSmem& s, const OwnRow& first, int64_t jtiles, unsigned int G,
                            int64_t r0, int64_t r1) {
  const long long before = s.before;
  const int mycnt = s.mycnt;
  const double tn = __longlong_as_double((long long)s.tnb);
  const int64_t n = s.total;
  const int64_t S = loop_splits<MIXED>(n, loop_itiles(n, loop_groups<MIXED>(n, jtiles, G)), jtiles, G, p.part_elems);
  const int64_t pstride = ((n + 31) / 32) * 32;
  const bool fin = S == 1;
  const bool cached = r1 - r0 <= kLDue;
  const int round = round_of(mycnt);
  for (int k0 = 0; k0 < mycnt; k0 += round) {
    const OwnRow o = FIRST && k0 == 0 ? first : own_row(p, s, k0, r0);
    const int L = o.L, l = o.l;
    const bool have = o.have;
    const int64_t k = before + k0 + (have ? o.q : 0);
    // the row's sums: final FP64 rows, double-single partials (summed and
    // exchanged in FP32), or FP64 partials
    float hi[7], lo[7];
    double f[7];
    if (fin) {
#pragma unroll
      for (int r = 0; r < 7; ++r) f[r] = have && l < 4 ? p.F[r * p.n_pad + k] : 0.0;
    } else if (MIXED) {
#pragma unroll
      for (int r = 0; r < 7; ++r) hi[r] = lo[r] = 0.0f;
      const float2* part2 = reinterpret_cast<const float2*>(p.part) + k;
      if (have)
        for (int64_t sp = l; sp < S; sp += U * L) {
          float2 v[U][7];  // (past the last split: zeros, which change nothing)
#pragma unroll
          for (int u = 0; u < U; ++u)
#pragma unroll
            for (int r = 0; r < 7; ++r)
              v[u][r] = sp + u * L < S ? part2[((sp + u * L) * 7 + r) * pstride] : make_float2(0.0f, 0.0f);
#pragma unroll
          for (int u = 0; u < U; ++u)
#pragma unroll
            for (int r = 0; r < 7; ++r) nbk::ds_add(hi[r], lo[r], v[u][r].x, v[u][r].y);
        }
      if (L >= 8) {  // each lane ends with one row; lanes 0-3 take theirs from the lanes that hold them
        float h, lw;
        nbk::ds_sum_rows(hi, lo, L, h, lw);
        const int base = (int)(threadIdx.x & 31) - l, c = l < 3 ? l : 0;
#pragma unroll
        for (int r = 0; r < 7; r += 3) {  // component c of the acceleration and the jerk, and the potential
          const int from = base + nbk::ds_row_lane(r < 6 ? r + c : 6, L);
          hi[r] = __shfl_sync(0xffffffffu, h, from);
          lo[r] = __shfl_sync(0xffffffffu, lw, from);
        }
      } else {
        for (int w = L / 2; w > 0; w >>= 1)
#pragma unroll
          for (int r = 0; r < 7; ++r) {
            const float oh = __shfl_xor_sync(0xffffffffu, hi[r], w);
            const float ol = __shfl_xor_sync(0xffffffffu, lo[r], w);
            nbk::ds_add(hi[r], lo[r], oh, ol);
          }
        if (L >= 4) {
#pragma unroll
          for (int r = 0; r < 6; r += 3) {
            hi[r] = l == 1 ? hi[r + 1] : (l == 2 ? hi[r + 2] : hi[r]);
            lo[r] = l == 1 ? lo[r + 1] : (l == 2 ? lo[r + 2] : lo[r]);
          }
        }
      }
    } else {
#pragma unroll
      for (int r = 0; r < 7; ++r) f[r] = 0.0;
      if (have)
        for (int64_t sp = l; sp < S; sp += U * L) {
          double v[U][7];
#pragma unroll
          for (int u = 0; u < U; ++u)
#pragma unroll
            for (int r = 0; r < 7; ++r)
              v[u][r] = sp + u * L < S ? p.part[((sp + u * L) * 7 + r) * pstride + k] : 0.0;
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (sp + u * L < S)
#pragma unroll
              for (int r = 0; r < 7; ++r) f[r] += v[u][r];
        }
      for (int w = L / 2; w > 0; w >>= 1)
#pragma unroll
        for (int r = 0; r < 7; ++r) f[r] += __shfl_xor_sync(0xffffffffu, f[r], w);
      f[6] = -f[6];
    }
    double nd = 0.0;
    if (L >= 4) {
      // every lane of the CTA takes this branch (L is uniform) and every
      // shuffle inside; lanes without a row write nothing.  Each lane forms the
      // FP64 values of its own component only (an FP64 addition holds the warp
      // for 64 cycles: 3 of them instead of 7, and none of the 14 conversions)
      double a1, j1, p1;
      if (MIXED && !fin) {
        a1 = nb_f64(hi[0]) + nb_f64(lo[0]);
        j1 = nb_f64(hi[3]) + nb_f64(lo[3]);
        p1 = -(nb_f64(hi[6]) + nb_f64(lo[6]));
      } else {
        a1 = l == 1 ? f[1] : (l == 2 ? f[2] : f[0]);
        j1 = l == 1 ? f[4] : (l == 2 ? f[5] : f[3]);
        p1 = f[6];
      }
      if (!(have && l < 4)) a1 = j1 = p1 = 0.0;
      nd = nbh::correct_lanes4(o.i, p.n_pad, tn, a1, j1, p1, o.in, p.eta, p.dt_min, p.dt_max, p.x, p.v, p.a, p.jk,
                               p.pot, p.t, p.dt, p.st, l, (int)(threadIdx.x & 31) - l, have);
    } else if (have && l == 0) {
      if (MIXED && !fin) {
#pragma unroll
        for (int r = 0; r < 7; ++r) f[r] = nb_f64(hi[r]) + nb_f64(lo[r]);
        f[6] = -f[6];
      }
      nd = nbh::correct_row(o.i, p.n_pad, tn, f, p.eta, p.dt_min, p.dt_max, p.x, p.v, p.a, p.jk, p.pot, p.t, p.dt,
                            p.xp, p.vp, p.st);
    }
    if (have && l == 0 && cached) s.due[o.i - r0] = (unsigned long long)__double_as_longlong(nd);
  }
}

// the next force item off the step's counter, which counts from `first`
__device__ __forceinline__ int next_item(const LoopArgs& p, LoopSmem& s, int first) {
  __syncthreads();  // every thread has read the previous item
  if (threadIdx.x == 0) s.item = first + (int)atomicAdd(&p.ctl->wq, 1ULL);
  __syncthreads();
  return s.item;
}

template <bool MIXED, int JT, int PER_SM>
__global__ void __launch_bounds__(kLT, PER_SM) loop_kernel(LoopArgs p) {
  using ForceSmem = typename std::conditional<MIXED, nbk::MixedSmem<JT>, nbk::Fp64Smem<kLT, JT>>::type;
  __shared__ __align__(16) ForceSmem fsm;
  __shared__ LoopSmem s;
  // the variants for small systems, whose steps are a chain of latencies; in
  // the others reading ahead costs the force items registers (N = 60000 mixed
  // 139.4 us a block step against 131.3), and FP64 items placed ahead of time gain
  // nothing (N = 16384 192 against 193, N = 32768 638 against 640)
  constexpr bool kShort = MIXED ? PER_SM == kLPerSmMixedSmall : JT == kLF64JTSmall;
  constexpr bool kPlaced = MIXED || kShort;  // the first item by the CTA's place
  const unsigned int G = gridDim.x;
  const int64_t N = p.N;
  const int64_t T = (N + kLT - 1) / kLT;
  const int64_t r0 = ((int64_t)blockIdx.x * T / G) * kLT;
  const int64_t r1 = min((((int64_t)blockIdx.x + 1) * T / G) * kLT, N);
  const int64_t jtiles = (N + JT - 1) / JT;
  const int64_t n_j = jtiles * JT;
  unsigned long long epoch = 0;
  long long steps = 0;
  double tn_prev = -INFINITY;  // the previous block time (they strictly increase)

  // placement: this CTA's rank among the CTAs on its SM, and its number among
  // the CTAs of that rank.  The CTAs in this order take the force items of a
  // step, so that a step with few items spreads them over the SMs.
  if (threadIdx.x == 0) {
    unsigned int smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    s.rank = (int)min(atomicAdd(&p.ctl->smrank[smid % kMaxSmid], 1u), (unsigned int)kMaxRank - 1);
    s.place = (int)atomicAdd(&p.ctl->ranks[s.rank], 1u);
  }
  // rows between N and the end of the last tile are massless far-away
  // padding in the predicted j-store (they fill the last j-tile)
  if (blockIdx.x == G - 1)
    for (int64_t i = N + threadIdx.x; i < min(T * kLT, p.n_pad); i += kLT) {
      const double px[3] = {NB_PAD_POS, NB_PAD_POS, NB_PAD_POS}, pv[3] = {0.0, 0.0, 0.0};
      float hi[3];
      nbh::store_predicted(i, p.n_pad, px, pv, 0.0, p.xp, p.vp, p.jA, p.jB, p.jC, true, MIXED, hi);
    }
  if (r1 - r0 <= kLDue)
    for (int64_t i = r0 + threadIdx.x; i < r1; i += kLT)
      s.due[i - r0] = (unsigned long long)__double_as_longlong(p.t[i] + p.dt[i]);
  __syncthreads();
  publish_slice(p, r0, r1, s);

  for (;;) {
    if (!grid_barrier(p.ctl, epoch, G, p.st, &s.ok)) return;  // A: slice minima published
    read_slices(p, G, s);
    const unsigned long long tnb = s.tnb;
    const double tn = __longlong_as_double((long long)tnb);
    const int64_t n = s.total;
    if (!isfinite(tn) || n <= 0) {  // no particle has a finite next time
      if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&p.st->flags, NB_ST_NUMERIC);
      break;
    }
    if (tn > p.t_end) break;  // every particle has reached t_end
    if (!(tn > tn_prev)) {  // no progress: a state without valid steps (dt = 0)
      if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&p.st->flags, NB_ST_STALLED);
      break;
    }
    tn_prev = tn;
    if (steps >= p.max_steps) {
      if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&p.st->flags, NB_ST_TIMEOUT);
      break;
    }
    if (steps == 0 && threadIdx.x == 0)  // (every CTA has registered before its first barrier)
      for (int r = 0; r < s.rank; ++r) s.place += (int)__ldcg(&p.ctl->ranks[r]);
    if (s.mine) write_active(p, r0, r1, tnb, s.before, s);
    predict_rows<MIXED>(p, r0, r1, tn, s);
    if (blockIdx.x == 0 && threadIdx.x == 0) p.ctl->wq = 0;  // nobody takes items before barrier B
    if (!grid_barrier(p.ctl, epoch, G, p.st, &s.ok)) return;  // B: list and j-store complete

    // forces (Sec. 4.1 step 4): items i-tile x j-split.  The first is the CTA's
    // by its place (when there are no more items than CTAs, as in every small
    // block, that is all, without counter round trips); the rest come from the
    // step's counter.
    const int groups = loop_groups<MIXED>(n, jtiles, G);
    const int64_t nI = loop_itiles(n, groups);
    const int64_t S = loop_splits<MIXED>(n, nI, jtiles, G, p.part_elems);
    const int64_t pstride = ((n + 31) / 32) * 32;
    const bool fin = S == 1;
    const int items = (int)(nI * S);
    int item = s.place;
    if (!kPlaced && item < items) item = next_item(p, s, 0);
    for (; item < items;) {
      const int itile = item % (int)nI, split = item / (int)nI;
      const int64_t jlo = nbk::split_begin(split, S, jtiles) * JT;
      // mixed: the padding rows of the last j-tile are massless far-away
      // particles in the j-store; FP64: cut at N (the item fills the tile)
      const int64_t jhi = min(nbk::split_begin(split + 1, S, jtiles) * JT, MIXED ? n_j : N);
      double* out = fin ? p.F : p.part + split * 7 * pstride;
      const int64_t ostride = fin ? p.n_pad : pstride;
      const int64_t ibase = (int64_t)itile * (kLT / groups);
      if constexpr (MIXED) {
#define NB_LOOP_ITEM(JG)                                                                                              \
  nbk::mixed_item<kLT, 1, JT, JG>(fsm, p.jA, p.jB, p.jC, jlo, jhi, n_j, p.act, n, ibase, p.eps2f, out, ostride, fin, \
                                  p.tbox, nullptr, 0, nbk::FusedArgs(), nbk::ISrc(), true)
        if (groups == 8)
          NB_LOOP_ITEM(8);
        else if (groups == 4)
          NB_LOOP_ITEM(4);
        else if (groups == 2)
          NB_LOOP_ITEM(2);
        else
          NB_LOOP_ITEM(1);
#undef NB_LOOP_ITEM
      } else {
        nbk::fp64_item<kLT, JT>(fsm, p.xp, p.vp, p.m, p.n_pad, 1, jlo, jhi, p.n_pad, p.act, n, ibase, p.eps2, out,
                                ostride, fin);
      }
      if (kPlaced && items <= (int)G) break;
      item = next_item(p, s, kPlaced ? (int)G : 0);
    }
    grid_arrive(p.ctl, epoch);
    OwnRow first;
    if (kShort) first = own_row(p, s, 0, r0);  // (its loads pass behind the wait)
    if (!grid_wait(p.ctl, epoch, G, p.st, &s.ok)) return;  // C: forces complete
    correct_own<MIXED, kShort ? 4 : 1, kShort>(p, s, first, jtiles, G, r0, r1);
    ++steps;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      p.ctl->steps = steps;
      p.ctl->interactions += (long long)s.total * (long long)N;
    }
    if (p.seg_steps > 0 && steps >= p.seg_steps) {
      if (blockIdx.x == 0 && threadIdx.x == 0) p.ctl->more = 1u;
      break;
    }
    __syncthreads();  // the corrected rows are visible to the whole CTA
    publish_slice(p, r0, r1, s);
  }
}

// the barrier alone, three times; expect = CTAs it waits for (one more than
// launched makes every wait run out)
__global__ void barrier_check_kernel(LoopCtl* ctl, unsigned int expect, long long wait_ns, nb_dev_status* st) {
  __shared__ int ok;
  unsigned long long epoch = 0;
  for (int k = 0; k < 3; ++k)
    if (!grid_barrier(ctl, epoch, expect, st, &ok, wait_ns)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->steps = 3;
}

struct PLoop {
  LoopCtl* ctl = nullptr;
  unsigned long long* smin = nullptr;
  int32_t* scnt = nullptr;
  int gmax = 0;
  int per_sm[4] = {0, 0, 0, 0};  // resident CTAs per SM of each instantiation (0 = not yet asked)
};

PLoop* ploop_of(nb_ctx* c) { return static_cast<PLoop*>(c->loop); }

// the instantiations: mixed, FP64 and each for small systems
const void* loop_variant(int v) {
  return v == 0   ? (const void*)loop_kernel<true, kLMixJT, kLPerSmMixed>
         : v == 1 ? (const void*)loop_kernel<true, kLMixJT, kLPerSmMixedSmall>
         : v == 2 ? (const void*)loop_kernel<false, kLF64JT, kLPerSm64>
                  : (const void*)loop_kernel<false, kLF64JTSmall, kLPerSm64>;
}
int variant_of(bool mixed, int64_t n) {
  if (mixed) return n <= kLMixedSmallHi ? 1 : 0;
  return n > kLF64SmallLo && n <= kLF64SmallHi ? 3 : 2;
}

int ctas_per_sm(PLoop* L, int v) {
  static const int most[4] = {kLPerSmMixed, kLPerSmMixedSmall, kLPerSm64, kLPerSm64};
  int& ps = L->per_sm[v];
  if (ps == 0) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, loop_variant(v), kLT, 0) != cudaSuccess) return -1;
    ps = std::min(occ, most[v]);
  }
  return ps;
}

}  // namespace

void nb_persistent_free(nb_ctx* c) {
  PLoop* L = c ? ploop_of(c) : nullptr;
  if (!L) return;
  if (L->ctl) cudaFree(L->ctl);
  if (L->smin) cudaFree(L->smin);
  if (L->scnt) cudaFree(L->scnt);
  delete L;
  c->loop = nullptr;
}

int nb_integrate_persistent(nb_ctx* c, double t_end) {
  if (c->n > nb_persistent_max_n(c)) return NB_EINVAL;
  const bool mixed = c->precision == NB_MIXED;
  PLoop* L = ploop_of(c);
  if (!L) {
    L = new PLoop();
    c->loop = L;
  }
  const int variant = variant_of(mixed, c->n);
  const int per_sm = ctas_per_sm(L, variant);
  if (per_sm < 1) {
    cudaGetLastError();
    return NB_ECUDA;
  }
  // as many CTAs as fit, but for a small system no more than twice its row
  // tiles, as each barrier waits for every CTA's arrival; at least 32, or two
  // CTAs per SM where the force items are a good part of a step (FP64; mixed, us
  // a block step with 32 and with two per SM: N = 300 16.2 / 16.3, N = 1024 15.5 /
  // 15.5, N = 1300 16.8 / 16.0, N = 2048 19.0 / 17.1, N = 4096 20.6 / 19.5)
  const int64_t row_tiles = (c->n + kLT - 1) / kLT;
  const bool two = variant == 3 || (variant == 1 && c->n > kLMixedTwoLo);
  const int G = (int)std::min<int64_t>(std::min(c->sm_count * per_sm, kLMaxG),
                                       std::max<int64_t>(two ? 2 * c->sm_count : 32, 2 * row_tiles));
  if (G > L->gmax) {
    if (L->smin) cudaFree(L->smin);
    if (L->scnt) cudaFree(L->scnt);
    L->smin = nullptr;
    L->scnt = nullptr;
    if (!L->ctl && cudaMalloc((void**)&L->ctl, sizeof(LoopCtl)) != cudaSuccess) return NB_ENOMEM;
    if (cudaMalloc((void**)&L->smin, G * sizeof(unsigned long long)) != cudaSuccess ||
        cudaMalloc((void**)&L->scnt, G * sizeof(int32_t)) != cudaSuccess) {
      L->gmax = 0;
      return NB_ENOMEM;
    }
    L->gmax = G;
  }
  // no valid run needs more than t_end / dt_min + 2 block steps
  const int64_t cap = std::min<int64_t>((int64_t)ceil(t_end / c->dt_min) + 2, 50000000);
  int64_t total = 0;
  for (;;) {
    long long seg = 0;
    if (mixed) {  // resident spatial order, renewed between launches
      const int rs = nb_ensure_sorted(c);
      if (rs != NB_OK) return rs;
      seg = std::max(1, c->sort_interval - c->perm_age);
    }
    LoopArgs p;
    memset(&p, 0, sizeof(p));
    p.N = c->n;
    p.n_pad = c->n_pad;
    p.eps2 = c->eps * c->eps;
    p.eps2f = (float)p.eps2;
    p.eta = c->eta;
    p.dt_min = c->dt_min;
    p.dt_max = c->dt_max;
    p.t_end = t_end;
    p.max_steps = cap;
    p.seg_steps = seg;
    p.m = c->m;
    p.x = c->x;
    p.v = c->v;
    p.a = c->a;
    p.jk = c->jk;
    p.pot = c->pot;
    p.t = c->t;
    p.dt = c->dt;
    p.xp = c->xp;
    p.vp = c->vp;
    p.jA = c->jA;
    p.jB = c->jB;
    p.jC = c->jC;
    p.tbox = mixed && c->perm_valid && c->far_tiles ? c->tbox : nullptr;
    p.act = c->act;
    p.F = c->F;
    p.part = c->part;
    p.part_elems = c->part_elems;
    p.smin = L->smin;
    p.scnt = L->scnt;
    p.ctl = L->ctl;
    p.st = c->status;
    if (cudaMemsetAsync(L->ctl, 0, sizeof(LoopCtl), c->stream) != cudaSuccess) return NB_ECUDA;
    void* args[] = {&p};
    cudaError_t e =
        cudaLaunchCooperativeKernel(loop_variant(variant), dim3((unsigned)G), dim3(kLT), args, 0, c->stream);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return NB_ECUDA;
    }
    LoopCtl h;
    if (cudaMemcpyAsync(c->hpin, L->ctl, sizeof(h), cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
        cudaStreamSynchronize(c->stream) != cudaSuccess)
      return NB_ECUDA;
    memcpy(&h, c->hpin, sizeof(h));
    c->launches += 1;
    c->steps += h.steps;
    c->perm_age += (int)h.steps;
    c->interactions += (double)h.interactions;
    total += h.steps;
    if (h.abort) return NB_ETIMEOUT;
    if (!h.more) break;
    if (total > cap) return NB_ETIMEOUT;
  }
  c->pred_valid = false;
  c->f_valid = false;
  return NB_OK;
}

// the grid barrier's bounded wait on the device: G CTAs wait for G (phantom
// = 0) or G + 1 (phantom != 0, so the first wait runs out after wait_ms)
int nb_persistent_barrier_check(nb_ctx* c, int phantom, double wait_ms) {
  PLoop* L = ploop_of(c);
  if (!L) {
    L = new PLoop();
    c->loop = L;
  }
  if (!L->ctl && cudaMalloc((void**)&L->ctl, sizeof(LoopCtl)) != cudaSuccess) return NB_ENOMEM;
  const unsigned int G = (unsigned int)c->sm_count;  // one CTA per SM is always co-resident
  const unsigned int expect = G + (phantom ? 1u : 0u);
  const long long wait_ns = (long long)(wait_ms * 1e6);
  LoopCtl* ctl = L->ctl;
  nb_dev_status* st = c->status;
  if (cudaMemsetAsync(L->ctl, 0, sizeof(LoopCtl), c->stream) != cudaSuccess) return NB_ECUDA;
  void* args[] = {&ctl, (void*)&expect, (void*)&wait_ns, &st};
  if (cudaLaunchCooperativeKernel((const void*)barrier_check_kernel, dim3(G), dim3(kLT), args, 0, c->stream) !=
      cudaSuccess) {
    cudaGetLastError();
    return NB_ECUDA;
  }
  LoopCtl h;
  if (cudaMemcpyAsync(c->hpin, L->ctl, sizeof(h), cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
      cudaStreamSynchronize(c->stream) != cudaSuccess)
    return NB_ECUDA;
  memcpy(&h, c->hpin, sizeof(h));
  c->launches += 1;
  if (h.abort) return NB_ETIMEOUT;
  return h.steps == 3 ? NB_OK : NB_ECUDA;
}
