// force_mixed.cu -- host-driven launch of the mixed-precision force item
// (force_common.cuh; Sec. 4.1 step 4, Eq. 3) for sm_103a.
//
// Grid: (i-tiles of NT*IPT active particles, fewer in small blocks whose
// threads share the j of a tile) x (j-range splits).  With one
// split the item writes final results into F; otherwise double-single
// partials [split][7][n] (an FP32 pair per 8-byte slot) that the split-j
// reduction sums in FP32, in a fixed order (deterministic for a given launch
// configuration), and converts to FP64 once per result.
#include <algorithm>

#include "force_common.cuh"

namespace {

// minimum resident CTAs per SM asked of the register allocator for the
// 128-thread, one-i-per-thread shape (0 = no request)
#ifndef NB_MIXED_MINB
#define NB_MIXED_MINB 0
#endif
#if NB_MIXED_MINB > 0
#define NB_MIXED_BOUNDS(NT, IPT) __launch_bounds__(NT, ((IPT) == 1 && (NT) == 128) ? NB_MIXED_MINB : 1)
#else
#define NB_MIXED_BOUNDS(NT, IPT) __launch_bounds__(NT)
#endif

template <int NT, int IPT, int JT, int JG = 1>
__global__ void NB_MIXED_BOUNDS(NT, IPT) force_mixed_kernel(
    const float4* __restrict__ jA, const float4* __restrict__ jB, const float2* __restrict__ jC,
    int64_t n_j, const int32_t* __restrict__ list, int64_t n, int64_t tiles, float eps2,
    double* __restrict__ out, int64_t ostride, int finalize, const float4* __restrict__ tbox,
    const int32_t* __restrict__ ord, const nbk::ISrc is) {
  __shared__ __align__(16) nbk::MixedSmem<JT> sm;
  const int split = blockIdx.y;
  const int64_t jlo = nbk::split_begin(split, gridDim.y, tiles) * JT;
  const int64_t jhi = min(nbk::split_begin(split + 1, gridDim.y, tiles) * JT, n_j);
  double* o = finalize ? out : out + (int64_t)split * 7 * ostride;
  nbk::mixed_item<NT, IPT, JT, JG>(sm, jA, jB, jC, jlo, jhi, n_j, list, n, (int64_t)blockIdx.x * (NT / JG * IPT),
                               eps2, o, ostride, finalize != 0, tbox, ord, 0, nbk::FusedArgs(), is, true);
}

// the same item with on-the-fly prediction of the j-tiles from the j-memory
// (Sec. 4.4 step 4); the i-particles' predicted rows are in jA/jB/jC
template <int NT, int JT, int JG>
__global__ void __launch_bounds__(NT) force_mixed_fused_kernel(
    const float4* __restrict__ jA, const float4* __restrict__ jB, const float2* __restrict__ jC,
    int64_t n_j, const int32_t* __restrict__ list, int64_t n, int64_t tiles, float eps2,
    double* __restrict__ out, int64_t ostride, int finalize, const float4* __restrict__ tbox,
    const int32_t* __restrict__ ord, const float4* __restrict__ jm, int64_t jm_stride,
    const double* __restrict__ tj, double T) {
  __shared__ __align__(16) nbk::FusedSmem<JT> sm;
  const int split = blockIdx.y;
  const int64_t jlo = nbk::split_begin(split, gridDim.y, tiles) * JT;
  const int64_t jhi = min(nbk::split_begin(split + 1, gridDim.y, tiles) * JT, n_j);
  double* o = finalize ? out : out + (int64_t)split * 7 * ostride;
  nbk::FusedArgs fa;
  fa.jm = jm;
  fa.stride = jm_stride;
  fa.tj = tj;
  fa.T = T;
  nbk::mixed_item<NT, 1, JT, JG>(sm, jA, jB, jC, jlo, jhi, n_j, list, n, (int64_t)blockIdx.x * (NT / JG), eps2, o,
                                 ostride, finalize != 0, tbox, ord, 0, fa, nbk::ISrc(), true);
}

// resident CTAs per SM of a kernel (0 when the query fails); `kept`: the
// caller's place for the answer, which is the same for every call
int resident(const void* kernel, int threads, int& kept) {
  if (kept == 0 && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&kept, kernel, threads, 0) != cudaSuccess) {
    cudaGetLastError();
    kept = 0;
  }
  return kept;
}

template <int NT, int IPT, int JT>
int per_sm_of() {
  static int per_sm = 0;
  return resident((const void*)force_mixed_kernel<NT, IPT, JT>, NT, per_sm);
}

// the j-splits of a launch of shape cfg (an explicit count, or as many items as
// fill the GPU; of a single i-tile one wave: its items are short, and a second
// wave would start them all over)
int splits_for(const nb_ctx* c, int64_t n, const nb_tuning& cfg, int per_sm) {
  if (cfg.nsplit > 0) return cfg.nsplit;
  const int s = nb_auto_split(c, n, cfg, per_sm);
  return n <= (int64_t)cfg.threads * cfg.ipt ? std::min(s, std::max(1, per_sm) * c->sm_count) : s;
}

template <int NT, int IPT, int JT>
cudaError_t launch(nb_ctx* c, const int32_t* d_list, int64_t n, const nb_tuning& cfg, float eps2,
                   const int32_t* ord, const nbk::ISrc& is) {
  auto kernel = force_mixed_kernel<NT, IPT, JT>;
  int per_sm = per_sm_of<NT, IPT, JT>();
  nb_tuning shape = cfg;
  if constexpr (NT == 128 && IPT == 1 && JT == 128) {
    static int kept[3] = {0, 0, 0};
    // (an explicit split count asks for exactly that launch)
    const int jg = cfg.nsplit > 0 ? 1 : nbk::j_groups(n, (c->n + JT - 1) / JT, per_sm * (int64_t)c->sm_count);
    if (jg > 1) {
      kernel = jg == 8   ? force_mixed_kernel<NT, IPT, JT, 8>
               : jg == 4 ? force_mixed_kernel<NT, IPT, JT, 4>
                         : force_mixed_kernel<NT, IPT, JT, 2>;
      per_sm = resident((const void*)kernel, NT, kept[jg == 8 ? 2 : jg / 4]);
      shape.threads = NT / jg;
    }
  }
  if (per_sm == 0) return cudaErrorInvalidValue;
  int nsplit = splits_for(c, n, shape, per_sm);
  const int64_t per_cta = (int64_t)shape.threads * IPT;
  const int64_t itiles = (n + per_cta - 1) / per_cta;
  const int64_t n_j = ((c->n + JT - 1) / JT) * JT;  // padding particles (m = 0) fill the last tile
  const int64_t tiles = n_j / JT;
  if (nsplit > tiles) nsplit = (int)tiles;
  if (nsplit < 1) nsplit = 1;
  dim3 grid((unsigned)itiles, (unsigned)nsplit);
  const bool fin = nsplit == 1;
  const int64_t ostride = fin ? c->n_pad : ((n + 31) / 32) * 32;
  double* out = fin ? c->F : c->part;
  if (!fin && (int64_t)nsplit * 7 * ostride > c->part_elems) return cudaErrorInvalidValue;
  c->launches += fin ? 1 : 2;
  // resident spatial order: far-tile boxes when the tiles match (unless the
  // context asks for double-single differences on every tile)
  const float4* tbox = (c->perm_valid && c->far_tiles) ? c->tbox : nullptr;
  kernel<<<grid, NT, 0, c->stream>>>(c->jA, c->jB, c->jC, n_j, d_list, n, tiles, eps2, out, ostride, fin ? 1 : 0,
                                     tbox, ord, is);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || fin) return e;
  return nb_launch_split_reduce_ds(c, n, nsplit, ostride);
}

}  // namespace

// forces on d_list with the j-tiles predicted to T on the fly (default launch
// shape: 128 threads, one i per thread, 128-particle j-tiles); boxes, when
// given, are the j-memory tile boxes grown by each particle's reach
cudaError_t nb_forces_mixed_fused(nb_ctx* c, const int32_t* d_list, int64_t n, const nb_tuning& cfg,
                                  const int32_t* ord, double T, const float4* boxes) {
  constexpr int NT = 128, JT = 128;
  if (n <= 0) return cudaSuccess;
  static int kept[4] = {0, 0, 0, 0};
  const int64_t n_j = ((c->n + JT - 1) / JT) * JT;
  const int64_t tiles = n_j / JT;
  const int per_sm1 = resident((const void*)force_mixed_fused_kernel<NT, JT, 1>, NT, kept[0]);
  const int jg = cfg.nsplit > 0 ? 1 : nbk::j_groups(n, tiles, per_sm1 * (int64_t)c->sm_count);
  auto kernel = jg == 8   ? force_mixed_fused_kernel<NT, JT, 8>
                : jg == 4 ? force_mixed_fused_kernel<NT, JT, 4>
                : jg == 2 ? force_mixed_fused_kernel<NT, JT, 2>
                          : force_mixed_fused_kernel<NT, JT, 1>;
  const int per_sm = resident((const void*)kernel, NT, kept[jg == 8 ? 3 : jg / 2]);
  if (per_sm == 0) return cudaErrorInvalidValue;
  const nb_tuning shape{1, NT / jg, JT, cfg.nsplit};
  int nsplit = splits_for(c, n, shape, per_sm);
  const int64_t itiles = (n + shape.threads - 1) / shape.threads;
  if (nsplit > tiles) nsplit = (int)tiles;
  if (nsplit < 1) nsplit = 1;
  const bool fin = nsplit == 1;
  const int64_t ostride = fin ? c->n_pad : ((n + 31) / 32) * 32;
  double* out = fin ? c->F : c->part;
  if (!fin && (int64_t)nsplit * 7 * ostride > c->part_elems) return cudaErrorInvalidValue;
  c->launches += fin ? 1 : 2;
  const float eps2 = (float)(c->eps * c->eps);
  kernel<<<dim3((unsigned)itiles, (unsigned)nsplit), NT, 0, c->stream>>>(
      c->jA, c->jB, c->jC, n_j, d_list, n, tiles, eps2, out, ostride, fin ? 1 : 0, boxes, ord, c->jm, c->n_pad,
      c->t, T);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || fin) return e;
  return nb_launch_split_reduce_ds(c, n, nsplit, ostride);
}

cudaError_t nb_launch_split_reduce_ds(nb_ctx* c, int64_t n, int nsplit, int64_t stride) {
  const cudaError_t e =
      nbk::launch_split_reduce(reinterpret_cast<const float2*>(c->part), stride, nsplit, n, c->F, c->n_pad, c->fo_acc,
                               c->fo_jerk, c->fo_pot, c->sm_count, c->stream);
  if (c->fo_acc || c->fo_jerk || c->fo_pot) c->fo_done = true;
  return e;
}

int nb_mixed_ctas_per_sm(const nb_tuning& cfg) {
#define NB_PER_SM_CASE(NT_, IPT_, JT_) \
  if (cfg.threads == NT_ && cfg.ipt == IPT_ && cfg.jtile == JT_) return per_sm_of<NT_, IPT_, JT_>();
#define NB_PER_SM_JT(NT_, IPT_) NB_PER_SM_CASE(NT_, IPT_, 64) NB_PER_SM_CASE(NT_, IPT_, 128) NB_PER_SM_CASE(NT_, IPT_, 256)
#define NB_PER_SM_IPT(NT_) NB_PER_SM_JT(NT_, 1) NB_PER_SM_JT(NT_, 2) NB_PER_SM_JT(NT_, 4)
  NB_PER_SM_IPT(64)
  NB_PER_SM_IPT(128)
  NB_PER_SM_IPT(256)
#undef NB_PER_SM_IPT
#undef NB_PER_SM_JT
#undef NB_PER_SM_CASE
  return 0;
}

bool nb_mixed_supported(const nb_tuning& t) {
  const bool thr = t.threads == 64 || t.threads == 128 || t.threads == 256;
  const bool ipt = t.ipt == 1 || t.ipt == 2 || t.ipt == 4;
  const bool jt = t.jtile == 64 || t.jtile == 128 || t.jtile == 256;
  return thr && ipt && jt;
}

#define NB_MIXED_CASE(NT_, IPT_, JT_)                            \
  if (cfg.threads == NT_ && cfg.ipt == IPT_ && cfg.jtile == JT_) \
    return launch<NT_, IPT_, JT_>(c, d_list, n, cfg, eps2, ord, is);

cudaError_t nb_forces_mixed(nb_ctx* c, const int32_t* d_list, int64_t n, const nb_tuning& cfg,
                            const int32_t* ord, const nbk::ISrc* isrc) {
  if (n <= 0) return cudaSuccess;
  const nbk::ISrc is = isrc ? *isrc : nbk::ISrc();
  const float eps2 = (float)(c->eps * c->eps);
#define NB_MIXED_JT(NT_, IPT_) NB_MIXED_CASE(NT_, IPT_, 64) NB_MIXED_CASE(NT_, IPT_, 128) NB_MIXED_CASE(NT_, IPT_, 256)
#define NB_MIXED_IPT(NT_) NB_MIXED_JT(NT_, 1) NB_MIXED_JT(NT_, 2) NB_MIXED_JT(NT_, 4)
  NB_MIXED_IPT(64)
  NB_MIXED_IPT(128)
  NB_MIXED_IPT(256)
#undef NB_MIXED_IPT
#undef NB_MIXED_JT
  return cudaErrorInvalidValue;
}
