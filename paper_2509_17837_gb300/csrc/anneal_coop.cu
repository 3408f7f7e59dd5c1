// Launches of the lane-parallel annealing kernel (anneal_coop.cuh): one code
// and schedule (xzzx_anneal_warp, and xzzx_anneal when its chains do not fill
// the GPU one per thread), and batches (batch mode 2, the server's small
// batches).
#include "anneal_coop_launch.cuh"
#include "batch_internal.h"

#include <algorithm>

namespace xzzx {

xzzx_status check_anneal_args(const xzzx_code*, const xzzx_schedule*, int, int);

namespace coop {
namespace {

// Batched form: the chunks of one distance, each cut into CTAs of kCtaChains
// chains (so a CTA's chains share a segment and its thresholds).
template <class Geo, int NC, int NP>
__global__ void __launch_bounds__(Form<Geo, NC, NP>::kThreads, kMinCtas<NP>)
    coop_chunks_kernel(const __grid_constant__ batch::CoopLaunch L) {
  constexpr int kCta = Form<Geo, NC, NP>::kCtaChains;
  extern __shared__ __align__(16) uint8_t smem[];
  const int per_chunk = L.nt / kCta;
  const batch::ChunkDev ch = L.chunks[L.chunk0 + blockIdx.x / per_chunk];
  const int first = (int)(blockIdx.x % per_chunk) * kCta;
  if (first >= ch.n_chains) return;  // the whole CTA
  const batch::SegDev& sg = L.segs[ch.seg];
  core::SweepTables tab;
  tab.T = ch.T;
  tab.sig = ch.sig;
  tab.n_sweeps = ch.n_sweeps;
  tab.n_classes = ch.n_classes;
  tab.n_live = ch.n_live;
  for (int j = 0; j < 4; ++j) tab.W[j] = ch.W[j];
  tab.err = sg.code.err;
  const core::ChainOut out{sg.chain_E, nullptr, nullptr, nullptr};
  anneal_coop_cta<Geo, NC, NP>(sg.init, sg.shot0 * (uint64_t)sg.restarts * 4u, (int64_t)ch.first_chain + first,
                             min(kCta, ch.n_chains - first), out, tab, L.keys, smem);
}

template <class Geo, int NC, int NP>
xzzx_status chunks_form(const batch::CoopLaunch& L, cudaStream_t stream) {
  using F = Form<Geo, NC, NP>;
  static DeviceOnce once;
  xzzx_status st = once.run([] { return allow_shared(coop_chunks_kernel<Geo, NC, NP>); });
  if (st) return st;
  const size_t smem = std::max(F::smem_bytes(L.n_classes), (size_t)std::max(L.smem, 0));
  const int64_t grid = (int64_t)L.n_chunks * (L.nt / F::kCtaChains);
  if (grid > 0x7FFFFFFF) return fail(XZZX_EINVAL, "too many chains for one launch");
  coop_chunks_kernel<Geo, NC, NP><<<(unsigned)grid, F::kThreads, smem, stream>>>(L);
  XZZX_CUDA_TRY(cudaGetLastError());
  return XZZX_OK;
}
template <class Geo>
xzzx_status chunks_g(const batch::CoopLaunch& L, cudaStream_t stream) {
  if (L.n_chunks <= 0) return XZZX_OK;
  int n_sm = 0;
  xzzx_status st = sm_count(&n_sm);
  if (st) return st;
  // An occupancy cap (L.smem) is one of the plain form's CTAs.
  return L.smem == 0 && producing<Geo>((int64_t)L.n_chunks * L.nt, n_sm) ? chunks_form<Geo, 1, 3>(L, stream)
                                                                       : chunks_form<Geo, 4, 0>(L, stream);
}

template <class Geo>
xzzx_status configure_g(int cap, int n_classes, int* smem_out, int* ctas_per_sm) {
  using F = Form<Geo, 4, 0>;
  xzzx_status st = allow_shared(coop_chunks_kernel<Geo, 4, 0>);
  if (st) return st;
  size_t smem = F::smem_bytes(n_classes);
  int dev = 0, per_sm_bytes = 0, reserved = 0, optin = 0;
  XZZX_CUDA_TRY(cudaGetDevice(&dev));
  XZZX_CUDA_TRY(cudaDeviceGetAttribute(&per_sm_bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
  XZZX_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  XZZX_CUDA_TRY(cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev));
  if (cap > 0) {
    const long pad = ((long)per_sm_bytes / cap - reserved) & ~15L;
    smem = std::max(smem, (size_t)std::min<long>(pad, optin));
  }
  XZZX_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, coop_chunks_kernel<Geo, 4, 0>, F::kThreads, smem));
  *smem_out = cap > 0 ? (int)smem : 0;
  return XZZX_OK;
}

}  // namespace
}  // namespace coop

#define XZZX_ALL_D(M) M(3) M(5) M(7) M(9) M(11) M(13) M(15) M(17) M(19) M(21) M(23) M(25) M(27) M(29) M(31)

// Whether a launch of n_chains distance-d chains is faster with several lanes
// per chain than with one thread per chain, whose time is that of one chain's
// sweeps until its warps fill the GPU.  One thread / this kernel, ms, 400 sweeps
// at p = 0.15, eta = 100: 0.71 / 0.47 at d = 5 and 3.75 / 2.04 at d = 15 for
// 16,384 chains, 0.71 / 0.81 and 3.74 / 3.67 for 32,768; 3.45 / 2.10 at d = 17
// and 10.3 / 4.4 at d = 31 for 8,192 chains, 3.47 / 4.03 and 10.3 / 8.3 for
// 16,384 (a pair of rows per lane leaves up to 7 of 16 lanes idle at d >= 17).
xzzx_status coop_is_faster(int d, int64_t n_chains, bool* yes) {
  int n_sm = 0;
  xzzx_status st = coop::sm_count(&n_sm);
  if (st) return st;
  *yes = n_chains <= (int64_t)n_sm * (d <= 15 ? 144 : 80);
  return XZZX_OK;
}

xzzx_status launch_anneal_coop(const xzzx_code* code, const xzzx_schedule* sched, uint64_t seed, uint64_t shot0,
                               int n_shots, int restarts, const uint32_t* init, int32_t* best_E, uint32_t* best_cfg,
                               int32_t* final_E, uint32_t* final_cfg, cudaStream_t stream) {
  const coop::Args A = coop::make_args(code, sched, seed, shot0, n_shots, restarts, init, best_E, best_cfg, final_E,
                                       final_cfg);
  switch (code->d) {
#define XZZX_CASE(DD) \
  case DD:            \
    return coop::launch_g<coop::RotLanes<DD>>(A, stream);
    XZZX_ALL_D(XZZX_CASE)
#undef XZZX_CASE
    default:
      return fail(XZZX_EUNSUPPORTED, "no annealing kernel for this distance");
  }
}

namespace batch {

xzzx_status configure_coop_chunks(int d, int cap, int n_classes, int* smem, int* ctas_per_sm) {
  switch (d) {
#define XZZX_CASE(DD) \
  case DD:            \
    return coop::configure_g<coop::RotLanes<DD>>(cap, n_classes, smem, ctas_per_sm);
    XZZX_ALL_D(XZZX_CASE)
#undef XZZX_CASE
    default:
      return fail(XZZX_EUNSUPPORTED, "no annealing kernel for this distance");
  }
}

xzzx_status launch_coop_chunks(int d, const CoopLaunch& L, cudaStream_t stream) {
  switch (d) {
#define XZZX_CASE(DD) \
  case DD:            \
    return coop::chunks_g<coop::RotLanes<DD>>(L, stream);
    XZZX_ALL_D(XZZX_CASE)
#undef XZZX_CASE
    default:
      return fail(XZZX_EUNSUPPORTED, "no annealing kernel for this distance");
  }
}

}  // namespace batch
}  // namespace xzzx

using namespace xzzx;

extern "C" xzzx_status xzzx_anneal_warp(const xzzx_code* code, const xzzx_schedule* sched, uint64_t seed,
                                        uint64_t shot0, int n_shots, int restarts, const uint32_t* init,
                                        int32_t* best_E, uint32_t* best_cfg, int32_t* final_E, uint32_t* final_cfg,
                                        void* stream) {
  xzzx_status st = check_anneal_args(code, sched, n_shots, restarts);
  if (st) return st;
  if (code->layout != kLayoutRotated) return fail(XZZX_EUNSUPPORTED, "the lane-parallel kernel takes rotated codes");
  if (n_shots == 0) return XZZX_OK;
  if ((st = check_ptr(init, "init")) || (st = check_ptr(best_E, "best_E"))) return st;
  return launch_anneal_coop(code, sched, seed, shot0, n_shots, restarts, init, best_E, best_cfg, final_E, final_cfg,
                            (cudaStream_t)stream);
}
