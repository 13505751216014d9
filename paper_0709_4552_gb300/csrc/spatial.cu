// spatial.cu -- resident spatial (Morton) order of the mixed path.
//
// The mixed force kernel forms position differences from double-single pairs
// (9 FP32 adds per pair).  When a warp's i-particles and a j-tile are far apart
// compared with their distance from the origin, the FP32 "hi" parts alone give
// the difference to FP32 accuracy (1 add per coordinate).  That needs warps
// and tiles that are spatially compact, so the particle arrays are kept in
// Morton order of the positions (row s holds particle perm[s]): the predictor,
// block selection, force and corrector kernels then walk rows and every
// access is coalesced, while the j-store and the active lists come out
// spatially ordered.  The order is a pure layout choice: every sum is over
// the same pairs.
//
// nb_spatial_sort: bounding box -> 30-bit Morton keys on a 1024^3 grid ->
// stable least-significant-digit radix sort (4 passes of 8 bits, ranked with
// warp match) -> the rows gathered into a scratch block and copied back, with
// perm composed and inverted on the way.  Deterministic.
//
// A block-step run sorts every 64 steps, so at 10^4 rows the sort is a chain of
// small kernels, each the latency of its launch and a few dependent steps.
// Hence few kernels (9 up to 131072 rows, 16 above; as bounding box, keys and
// count / scan / scatter per pass it was 19 and a copy) and short chains.
// Time: 12000 rows 139 -> 47 us, 32768 rows 155 -> 55 us; at 2^20 rows, where
// one CTA's scan of all histograms was 4 x 205 us, 1125 -> 384 us.
#include <float.h>

#include <algorithm>

#include "nb_internal.cuh"

namespace {

constexpr int kSortThreads = 256;
constexpr int kRadix = 256;
static_assert(kSortThreads == kRadix, "thread = digit in the scatter");
constexpr int kSortWarps = kSortThreads / 32;
// elements per thread: short chunks while they still leave the chip mostly
// idle, long ones (longer runs of equal digits to write) above
constexpr int kItemsSmall = 2, kItemsLarge = 8;
constexpr int64_t kSmallRows = 32768;
// up to this many chunks a scatter CTA adds up the chunks' histograms itself
// (64 coalesced rows, batched) and counts the next pass's digits as it writes:
// one kernel a pass; above, a count and a prefix kernel before each scatter
constexpr int kFusedChunks = 64;

// doubles as integers of the same order (min and max without the FP64 unit)
__device__ __forceinline__ long long ord_of(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFLL);
}
__device__ __forceinline__ double of_ord(long long o) {
  return __longlong_as_double(o ^ ((o >> 63) & 0x7FFFFFFFFFFFFFFFLL));
}

// minima b[0..2] and maxima b[3..5] over the CTA; valid on threads 0-5, the
// value of component threadIdx.x
__device__ __forceinline__ long long bbox_reduce(const long long (&in)[6], long long (*sm)[6]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    long long v = in[c];
    for (int o = 16; o > 0; o >>= 1) {
      const long long u = __shfl_xor_sync(0xffffffffu, v, o);
      v = c < 3 ? min(u, v) : max(u, v);
    }
    if (lane == 0) sm[w][c] = v;
  }
  __syncthreads();
  long long r = 0;
  if (threadIdx.x < 6) {
    r = sm[0][threadIdx.x];
    for (int q = 1; q < kSortWarps; ++q)
      r = threadIdx.x < 3 ? min(r, sm[q][threadIdx.x]) : max(r, sm[q][threadIdx.x]);
  }
  return r;
}

__device__ __forceinline__ void bbox_start(long long (&b)[6]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    b[c] = ord_of(DBL_MAX);
    b[3 + c] = ord_of(-DBL_MAX);
  }
}

__global__ void __launch_bounds__(kSortThreads) bbox_partial(int64_t N, int64_t n_pad, const double* __restrict__ x,
                                                             long long* __restrict__ red) {
  long long b[6];
  bbox_start(b);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double v = x[c * n_pad + i];
      if (isnan(v)) continue;
      b[c] = min(b[c], ord_of(v));
      b[3 + c] = max(b[3 + c], ord_of(v));
    }
  __shared__ long long sm[kSortWarps][6];
  const long long r = bbox_reduce(b, sm);
  if (threadIdx.x < 6) red[blockIdx.x * 6 + threadIdx.x] = r;
}

// keys on the grid of the box of the nb partial boxes, which every CTA reduces
// for itself
__global__ void __launch_bounds__(kSortThreads) morton_keys(int64_t N, int64_t n_pad, const double* __restrict__ x,
                                                            int nb, const long long* __restrict__ red,
                                                            uint32_t* __restrict__ key, int32_t* __restrict__ val) {
  __shared__ long long sm[kSortWarps][6];
  __shared__ double box[6], s_scale;
  long long b[6];
  bbox_start(b);
  for (int k = threadIdx.x; k < nb; k += kSortThreads)
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const long long v = red[k * 6 + c];
      b[c] = c < 3 ? min(b[c], v) : max(b[c], v);
    }
  const long long r = bbox_reduce(b, sm);
  if (threadIdx.x < 6) box[threadIdx.x] = of_ord(r);
  __syncthreads();
  if (threadIdx.x == 0) {
    const double w = fmax(box[3] - box[0], fmax(box[4] - box[1], box[5] - box[2]));
    s_scale = w > 0.0 ? 1023.0 / w : 0.0;
  }
  __syncthreads();
  const double scale = s_scale;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
    uint32_t q[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)  // (the conversion saturates: below the grid, or NaN, is 0)
      q[c] = min(__double2uint_rz((x[c * n_pad + i] - box[c]) * scale), 1023u);
    key[i] = nb_spread10(q[0]) | (nb_spread10(q[1]) << 1) | (nb_spread10(q[2]) << 2);
    val[i] = (int32_t)i;
  }
}

// hist[chunk][digit] of one pass; with zero: the histograms of `zero` more
// passes cleared (they follow, gridDim.x chunks each)
template <int K>
__global__ void __launch_bounds__(kSortThreads) radix_count(const uint32_t* __restrict__ key, int64_t N, int shift,
                                                            int32_t* __restrict__ hist, int zero) {
  __shared__ int cnt[kRadix];
  cnt[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * (K * kSortThreads);
#pragma unroll
  for (int it = 0; it < K; ++it) {
    const int64_t e = base + it * kSortThreads + threadIdx.x;
    if (e < N) atomicAdd(&cnt[(key[e] >> shift) & 0xFFu], 1);
  }
  __syncthreads();
  const int64_t at = (int64_t)blockIdx.x * kRadix + threadIdx.x;
  hist[at] = cnt[threadIdx.x];
  for (int q = 1; q <= zero; ++q) hist[(int64_t)q * gridDim.x * kRadix + at] = 0;
}

// each digit's counts over the chunks -> exclusive prefixes in place, and the
// digit's total; a CTA takes 8 digits (a 32-byte sector of a row), its threads
// 128 runs of chunks
constexpr int kPrefixRuns = 128;
__global__ void __launch_bounds__(8 * kPrefixRuns) radix_prefix(int32_t* __restrict__ hist, int nblocks,
                                                                int32_t* __restrict__ tot) {
  __shared__ int32_t sm[kPrefixRuns][8];
  const int d = threadIdx.x & 7, run = threadIdx.x >> 3;
  const int per = (nblocks + kPrefixRuns - 1) / kPrefixRuns;
  const int q0 = min(run * per, nblocks), q1 = min(q0 + per, nblocks);
  int32_t* h = hist + blockIdx.x * 8 + d;
  int32_t sum = 0;
#pragma unroll 4
  for (int q = q0; q < q1; ++q) sum += h[(int64_t)q * kRadix];
  sm[run][d] = sum;
  __syncthreads();
  for (int o = 1; o < kPrefixRuns; o <<= 1) {
    const int32_t u = run >= o ? sm[run - o][d] : 0;
    __syncthreads();
    sm[run][d] += u;
    __syncthreads();
  }
  int32_t at = sm[run][d] - sum;
  if (run == kPrefixRuns - 1) tot[blockIdx.x * 8 + d] = sm[run][d];
#pragma unroll 4
  for (int q = q0; q < q1; ++q) {
    const int32_t v = h[(int64_t)q * kRadix];
    h[(int64_t)q * kRadix] = at;
    at += v;
  }
}

// Stable scatter of one chunk by one digit.  A warp owns 32 K consecutive
// elements and ranks them 32 at a time against its own running counts, so the
// CTA meets three times in all, whatever K.  FUSED: hist holds the chunks'
// counts, which thread d adds up for digit d, and next (if any) receives the
// next pass's; else hist holds exclusive prefixes and tot the digits' totals.
template <int K, bool FUSED>
__global__ void __launch_bounds__(kSortThreads) radix_scatter(
    const uint32_t* __restrict__ kin, const int32_t* __restrict__ vin, uint32_t* __restrict__ kout,
    int32_t* __restrict__ vout, int64_t N, int shift, const int32_t* __restrict__ hist,
    const int32_t* __restrict__ tot, int32_t* __restrict__ next) {
  constexpr int kChunk = K * kSortThreads;
  __shared__ int32_t at[kSortWarps][kRadix];  // counts, then first places, by warp and digit
  __shared__ int32_t wsum[kSortWarps];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t first = (int64_t)blockIdx.x * kChunk + wid * (32 * K) + lane;
  uint32_t k[K];
  int32_t v[K];
#pragma unroll
  for (int it = 0; it < K; ++it) {
    const int64_t e = first + it * 32;
    k[it] = e < N ? kin[e] : 0u;
    v[it] = e < N ? vin[e] : 0;
  }
  int32_t before = 0, total = 0;
  if (FUSED) {
#pragma unroll 8
    for (int q = 0; q < (int)gridDim.x; ++q) {
      const int32_t h = hist[q * kRadix + tid];
      total += h;
      before += q < (int)blockIdx.x ? h : 0;
    }
  } else {
    before = hist[(int64_t)blockIdx.x * kRadix + tid];
    total = tot[tid];
  }
  int32_t incl = total;
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) wsum[wid] = incl;
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) at[w][tid] = 0;
  __syncthreads();
  int32_t place = incl - total + before;  // of the chunk's first element of digit tid
  for (int w = 0; w < wid; ++w) place += wsum[w];
  int rank[K];
#pragma unroll
  for (int it = 0; it < K; ++it) {
    const bool valid = first + it * 32 < N;
    const int digit = valid ? (int)((k[it] >> shift) & 0xFFu) : kRadix;  // kRadix: no element
    const unsigned peers = __match_any_sync(0xffffffffu, digit);
    const int lower = __popc(peers & ((1u << lane) - 1u));
    const int c = valid ? at[wid][digit] : 0;
    rank[it] = c + lower;
    __syncwarp();
    if (valid && lower == 0) at[wid][digit] = c + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) {
    const int32_t c = at[w][tid];
    at[w][tid] = place;
    place += c;
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < K; ++it)
    if (first + it * 32 < N) {
      const int32_t pos = at[wid][(k[it] >> shift) & 0xFFu] + rank[it];
      kout[pos] = k[it];
      vout[pos] = v[it];
      if (FUSED && next) atomicAdd(&next[(pos / kChunk) * kRadix + ((k[it] >> (shift + 8)) & 0xFFu)], 1);
    }
}

int grid_for(int64_t n, int threads, int cap) {
  int64_t g = (n + threads - 1) / threads;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}

// pos[slot] = list position of each listed slot (clamped; pos starts at -1, a
// repeated slot keeps one of its positions) and cnt[q] = listed slots in
// [q kOrderChunk, (q + 1) kOrderChunk)
constexpr int kOrderChunk = 1024;
__global__ void order_scatter(const int32_t* __restrict__ list, int64_t n, int64_t N, int32_t* __restrict__ pos,
                              int32_t* __restrict__ cnt) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    int64_t p = list[k];
    p = p < 0 ? 0 : (p >= N ? N - 1 : p);
    if (atomicExch(&pos[p], (int32_t)k) < 0) atomicAdd(&cnt[p / kOrderChunk], 1);
  }
}

// the positions in slot order: CTA q sums the counts of the chunks before its
// own and places its chunk's positions after them.  Places left over (a list
// with repeated slots, which the caller's check reports) get position 0.
__global__ void __launch_bounds__(kOrderChunk) order_write(const int32_t* __restrict__ pos,
                                                          const int32_t* __restrict__ cnt, int chunks, int64_t n,
                                                          int64_t N, int32_t* __restrict__ ord) {
  constexpr int kWarps = kOrderChunk / 32;
  __shared__ int32_t before[kWarps], total[kWarps], own[kWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t b = 0, t = 0;
  for (int q = threadIdx.x; q < chunks; q += kOrderChunk) {
    const int32_t v = cnt[q];
    t += v;
    if (q < (int)blockIdx.x) b += v;
  }
  const int64_t s = (int64_t)blockIdx.x * kOrderChunk + threadIdx.x;
  const int32_t k = s < N ? pos[s] : -1;
  const unsigned on = __ballot_sync(0xffffffffu, k >= 0);
  b = __reduce_add_sync(0xffffffffu, b);
  t = __reduce_add_sync(0xffffffffu, t);
  if (lane == 0) {
    before[w] = b;
    total[w] = t;
    own[w] = __popc(on);
  }
  __syncthreads();
  int32_t at = __popc(on & ((1u << lane) - 1u));
  t = 0;
  for (int q = 0; q < kWarps; ++q) {
    at += before[q] + (q < w ? own[q] : 0);
    t += total[q];
  }
  if (k >= 0) ord[at] = k;
  if (blockIdx.x == 0)
    for (int64_t q = t + threadIdx.x; q < n; q += kOrderChunk) ord[q] = 0;
}

// the 16 FP64 rows of the master state: m, x[3], v[3], a[3], jerk[3], pot, t, dt
constexpr int kStateRows = 16;
struct StateRows {
  double* row[kStateRows];
};

StateRows state_rows(nb_ctx* c) {
  StateRows r;
  double* arr[8] = {c->m, c->x, c->v, c->a, c->jk, c->pot, c->t, c->dt};
  const int cnt[8] = {1, 3, 3, 3, 3, 1, 1, 1};
  int q = 0;
  for (int i = 0; i < 8; ++i)
    for (int k = 0; k < cnt[i]; ++k) r.row[q++] = arr[i] + (int64_t)k * c->n_pad;
  return r;
}

// scratch[q][s] = row_q[src[s]] for s < N (a gather of every state row); with
// order: order[s] = particle of the new row s (old row src[s] holds particle
// perm[src[s]], or src[s] when perm is null), and its inverse
__global__ void gather_state(int64_t N, int64_t n_pad, StateRows rows, const int32_t* __restrict__ src,
                             double* __restrict__ scratch, const int32_t* __restrict__ perm,
                             int32_t* __restrict__ order, int32_t* __restrict__ inverse) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)gridDim.x * blockDim.x) {
    const int64_t from = src[s];
    if (order) {
      const int32_t particle = perm ? perm[from] : (int32_t)from;
      order[s] = particle;
      inverse[particle] = (int32_t)s;
    }
#pragma unroll
    for (int q = 0; q < kStateRows; ++q) scratch[q * n_pad + s] = rows.row[q][from];
  }
}

// the gathered rows, and the order, to their places
__global__ void copy_state_back(int64_t N, int64_t n_pad, StateRows rows, const double* __restrict__ scratch,
                                const int32_t* __restrict__ order, int32_t* __restrict__ perm) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)gridDim.x * blockDim.x) {
    if (order) perm[s] = order[s];
#pragma unroll
    for (int q = 0; q < kStateRows; ++q) rows.row[q][s] = scratch[q * n_pad + s];
  }
}

// out[k] = map[in[k]] with in[k] clamped to [0, N) (in == out allowed)
__global__ void map_list(const int32_t* in, int64_t n, const int32_t* __restrict__ map, int64_t N, int32_t* out) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    int64_t p = in[k];
    p = p < 0 ? 0 : (p >= N ? N - 1 : p);
    out[k] = map[p];
  }
}

// a caller's list: NB_ST_BADLIST unless ascending within [0, N); with map,
// out[k] = map[in[k]] (in[k] clamped to [0, N))
__global__ void check_map_list(const int32_t* __restrict__ in, int64_t n, const int32_t* __restrict__ map, int64_t N,
                               int32_t* __restrict__ out, unsigned int* __restrict__ flag) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = in[k];
    if (v < 0 || v >= N || (k > 0 && in[k - 1] >= v)) atomicOr(flag, NB_ST_BADLIST);
    if (map) {
      const int64_t p = v < 0 ? 0 : (v >= N ? N - 1 : v);
      out[k] = map[p];
    }
  }
}

// dst[k * rows + r] = src[r * n_pad + iperm[first + k]]
__global__ void gather_rows(const double* __restrict__ src, int rows, int64_t n_pad, const int32_t* __restrict__ iperm,
                            int64_t first, int64_t count, double* __restrict__ dst) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < count;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = iperm[first + k];
    for (int r = 0; r < rows; ++r) dst[k * rows + r] = src[r * n_pad + s];
  }
}

// reorder every state row by src (new row s = old row src[s]) in place; with
// order (scratch of N): perm and iperm too
cudaError_t reorder_state(nb_ctx* c, const int32_t* src, int32_t* order) {
  c->state_ver++;  // rows move: any row-keyed copy of the state (the j-memory) is stale
  if (!c->pscratch) {
    cudaError_t e = cudaMalloc(&c->pscratch, (size_t)kStateRows * c->n_pad * sizeof(double));
    if (e != cudaSuccess) {
      c->pscratch = nullptr;
      return e;
    }
  }
  const StateRows rows = state_rows(c);
  const int g = grid_for(c->n, 256, c->sm_count * 16);
  gather_state<<<g, 256, 0, c->stream>>>(c->n, c->n_pad, rows, src, c->pscratch, c->perm_valid ? c->perm : nullptr,
                                         order, c->iperm);
  copy_state_back<<<g, 256, 0, c->stream>>>(c->n, c->n_pad, rows, c->pscratch, order, c->perm);
  c->launches += 2;
  return cudaGetLastError();
}

// stable LSD radix sort of (skey[0], sval[0])[0..n) on the low `bits` bits;
// *cur = the buffer holding the result
template <int K>
cudaError_t sort_pairs(nb_ctx* c, int64_t n, int bits, int* cur) {
  const int64_t chunk = K * kSortThreads;
  const int nblocks = (int)((n + chunk - 1) / chunk), passes = (bits + 7) / 8;
  const bool fused = nblocks <= kFusedChunks;
  const int64_t histogram = (int64_t)nblocks * kRadix;
  int32_t* tot = c->shist + histogram;  // (unfused: one histogram)
  int b = 0;
  for (int p = 0; p < passes; ++p, b ^= 1) {
    int32_t* hist = c->shist + (fused ? p * histogram : 0);
    if (p == 0 || !fused) {
      radix_count<K><<<nblocks, kSortThreads, 0, c->stream>>>(c->skey[b], n, 8 * p, hist, fused ? passes - 1 : 0);
      c->launches += 1;
    }
    if (fused) {
      radix_scatter<K, true><<<nblocks, kSortThreads, 0, c->stream>>>(
          c->skey[b], c->sval[b], c->skey[b ^ 1], c->sval[b ^ 1], n, 8 * p, hist, nullptr,
          p + 1 < passes ? hist + histogram : nullptr);
    } else {
      radix_prefix<<<kRadix / 8, 8 * kPrefixRuns, 0, c->stream>>>(hist, nblocks, tot);
      radix_scatter<K, false><<<nblocks, kSortThreads, 0, c->stream>>>(
          c->skey[b], c->sval[b], c->skey[b ^ 1], c->sval[b ^ 1], n, 8 * p, hist, tot, nullptr);
      c->launches += 1;
    }
    c->launches += 1;
  }
  *cur = b;
  return cudaGetLastError();
}

}  // namespace

// histogram scratch of a sort of up to n rows (and of the list order's counts)
size_t nb_sort_hist_ints(int64_t n) {
  const size_t chunks = std::max<size_t>((size_t)(n / (kItemsLarge * kSortThreads) + 1), 4 * kFusedChunks);
  return (chunks + 1) * kRadix;
}

// stable sort of the rows by the keys in skey[0] (values = row numbers in
// sval[0]) on the low `bits` bits, then the state reordered to that order
cudaError_t nb_order_rows_by_keys(nb_ctx* c, int bits) {
  const int64_t N = c->n;
  int cur = 0;
  cudaError_t e =
      N <= kSmallRows ? sort_pairs<kItemsSmall>(c, N, bits, &cur) : sort_pairs<kItemsLarge>(c, N, bits, &cur);
  if (e != cudaSuccess) return e;
  // sval[cur][s] = the current row that becomes row s
  return reorder_state(c, c->sval[cur], c->sval[cur ^ 1]);
}

cudaError_t nb_spatial_sort(nb_ctx* c) {
  const int64_t N = c->n;
  if (N <= 0) return cudaSuccess;
  // (the key kernel's CTAs read all partial boxes: two per SM are enough to
  // stream the positions)
  const int nbb = grid_for(N, kSortThreads, std::min(c->sm_count * 2, (int)(NB_RED_DOUBLES / 6)));
  long long* red = reinterpret_cast<long long*>(c->red);
  bbox_partial<<<nbb, kSortThreads, 0, c->stream>>>(N, c->n_pad, c->x, red);
  morton_keys<<<grid_for(N, kSortThreads, c->sm_count * 8), kSortThreads, 0, c->stream>>>(
      N, c->n_pad, c->x, nbb, red, c->skey[0], c->sval[0]);
  c->launches += 2;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return nb_order_rows_by_keys(c, 30);
}

cudaError_t nb_unsort(nb_ctx* c) {
  if (!c->perm_valid) return cudaSuccess;
  // particle p = old row iperm[p]
  cudaError_t e = reorder_state(c, c->iperm, nullptr);
  if (e != cudaSuccess) return e;
  c->perm_valid = false;
  c->pred_valid = false;
  c->f_valid = false;
  return cudaSuccess;
}

cudaError_t nb_map_to_slots(nb_ctx* c, const int32_t* d_list, int64_t n, const int32_t** out) {
  if (!c->perm_valid || n <= 0) {
    *out = d_list;
    return cudaSuccess;
  }
  map_list<<<grid_for(n, 256, c->sm_count * 16), 256, 0, c->stream>>>(d_list, n, c->iperm, c->n, c->mlist);
  c->launches += 1;
  *out = c->mlist;
  return cudaGetLastError();
}

cudaError_t nb_check_map_to_slots(nb_ctx* c, const int32_t* d_list, int64_t n, const int32_t** out) {
  if (n <= 0) {
    *out = d_list;
    return cudaSuccess;
  }
  c->launches += 1;
  check_map_list<<<grid_for(n, 256, c->sm_count * 16), 256, 0, c->stream>>>(
      d_list, n, c->perm_valid ? c->iperm : nullptr, c->n, c->perm_valid ? c->mlist : nullptr, &c->status->flags);
  *out = c->perm_valid ? c->mlist : d_list;
  return cudaGetLastError();
}

cudaError_t nb_map_to_particles(nb_ctx* c, const int32_t* in, int64_t n, int32_t* out) {
  if (n <= 0) return cudaSuccess;
  if (!c->perm_valid) {
    if (in == out) return cudaSuccess;
    return cudaMemcpyAsync(out, in, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, c->stream);
  }
  map_list<<<grid_for(n, 256, c->sm_count * 16), 256, 0, c->stream>>>(in, n, c->perm, c->n, out);
  c->launches += 1;
  return cudaGetLastError();
}

cudaError_t nb_gather_rows(nb_ctx* c, const double* src, int rows, int64_t first, int64_t count, double* dst) {
  if (count <= 0) return cudaSuccess;
  gather_rows<<<grid_for(count, 256, c->sm_count * 16), 256, 0, c->stream>>>(src, rows, c->n_pad, c->iperm, first,
                                                                             count, dst);
  c->launches += 1;
  return cudaGetLastError();
}

// Processing order of a caller's active list (mapped to slots) in the
// spatial order: list positions sorted by slot.  The mixed kernel then forms
// warps of nearby particles; results still go to the caller's positions.
// Returns a device array of n positions.
//
// A list of every particle is the identity (ascending and unique), so its
// order is the resident order itself.  The slots of any other list are
// distinct, so counting them in place of a sort of (slot, position) pairs
// costs two kernels and two memsets instead of two or three radix passes
// (16 us against 75 at N = 2^20, n = 4096; the radix sort took 64 of the
// 482 us of a force call on all of N = 20011).
cudaError_t nb_list_order(nb_ctx* c, const int32_t* d_list, int64_t n, const int32_t** ord) {
  if (n == c->n) {
    *ord = c->perm;
    return cudaSuccess;
  }
  const int chunks = (int)((c->n + kOrderChunk - 1) / kOrderChunk);
  int32_t* pos = reinterpret_cast<int32_t*>(c->skey[0]);
  cudaError_t e = cudaMemsetAsync(pos, 0xFF, c->n * sizeof(int32_t), c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->shist, 0, chunks * sizeof(int32_t), c->stream);
  if (e != cudaSuccess) return e;
  order_scatter<<<grid_for(n, 256, c->sm_count * 16), 256, 0, c->stream>>>(d_list, n, c->n, pos, c->shist);
  order_write<<<chunks, kOrderChunk, 0, c->stream>>>(pos, c->shist, chunks, n, c->n, c->sval[0]);
  c->launches += 2;
  *ord = c->sval[0];
  return cudaGetLastError();
}
