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
template <class Geo, int NC, int NP, int PER>
__global__ void __launch_bounds__(Form<Geo, NC, NP, PER>::kThreads, Form<Geo, NC, NP, PER>::kRegCtas)
    coop_chunks_kernel(const __grid_constant__ batch::CoopLaunch L) {
  constexpr int kCta = Form<Geo, NC, NP, PER>::kCtaChains;
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
  anneal_coop_cta<Geo, NC, NP, PER>(sg.init, sg.shot0 * (uint64_t)sg.restarts * 4u, (int64_t)ch.first_chain + first,
                             min(kCta, ch.n_chains - first), out, tab, L.keys, smem);
}

template <class Geo, int NC, int NP, int PER>
xzzx_status chunks_form(const batch::CoopLaunch& L, cudaStream_t stream) {
  using F = Form<Geo, NC, NP, PER>;
  static DeviceOnce once;
  xzzx_status st = once.run([] { return allow_shared(coop_chunks_kernel<Geo, NC, NP, PER>); });
  if (st) return st;
  const size_t smem = std::max(F::smem_bytes(L.n_classes), (size_t)std::max(L.smem, 0));
  const int64_t grid = (int64_t)L.n_chunks * (L.nt / F::kCtaChains);
  if (grid > 0x7FFFFFFF) return fail(XZZX_EINVAL, "too many chains for one launch");
  coop_chunks_kernel<Geo, NC, NP, PER><<<(unsigned)grid, F::kThreads, smem, stream>>>(L);
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
  const int per = L.smem == 0 ? producing_per_sm<Geo>((int64_t)L.n_chunks * L.nt, n_sm) : 0;
  return per == 3   ? chunks_form<Geo, 1, 3, 3>(L, stream)
         : per == 4 ? chunks_form<Geo, 1, 3, 4>(L, stream)
                    : chunks_form<Geo, 4, 0, 4>(L, stream);
}

template <class Geo>
xzzx_status configure_g(int cap, int n_classes, int* smem_out, int* ctas_per_sm) {
  using F = Form<Geo, 4, 0, 4>;
  xzzx_status st = allow_shared(coop_chunks_kernel<Geo, 4, 0, 4>);
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
  XZZX_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, coop_chunks_kernel<Geo, 4, 0, 4>, F::kThreads, smem));
  *smem_out = cap > 0 ? (int)smem : 0;
  return XZZX_OK;
}

}  // namespace
}  // namespace coop

#define XZZX_ALL_D(M) M(3) M(5) M(7) M(9) M(11) M(13) M(15) M(17) M(19) M(21) M(23) M(25) M(27) M(29) M(31)

// Whether a launch of n_chains distance-d chains is faster with several lanes
// per chain than with one thread per chain, whose time is that of one chain's
// sweeps until its warps fill the GPU.  The lanes' throughput is in proportion to
// the share of them that hold rows, (d+1)/2 of a power of two.  The line is where the
// schedule with dense draws (50 sweeps near the Nishimori temperature; the first of
// each pair) crosses; the one with sparse draws (200 sweeps to 20 times it) crosses
// later.  Thread time / lane time at chains per SM:
//   d     100         140         160         180         200         220
//   5  1.18 1.29   1.08 1.19   1.09 1.19   0.79 0.83   0.73 0.80   0.73 0.80
//   7  1.48 1.56   1.42 1.47   1.40 1.44   1.03 1.06   0.96 1.00   0.96 0.99
//   9  1.07 1.21   0.96 1.04   0.91 0.97   0.79 0.91   0.71 0.80   0.67 0.75
//  11  1.18 1.32   1.04 1.12   0.96 1.06   0.84 0.98   0.75 0.86   0.72 0.81
//  15  1.51 1.45   1.36 1.37   1.27 1.27   1.10 1.18   0.99 1.03   0.94 0.97
//  17  0.97 1.15   0.88 1.09   0.80 0.99   0.70 0.89   0.64 0.79   0.58 0.74
//  21  1.04 1.22   0.96 1.21   0.88 1.09   0.77 0.96   0.70 0.87   0.64 0.80
//  25  1.19 1.25   1.23 1.37   1.11 1.23   0.98 1.08   0.89 0.97   0.80 0.89
//  29  1.29 1.30   1.33 1.44   1.20 1.29   1.05 1.14   0.96 1.02   0.87 0.94
//  31  1.42 1.42   1.48 1.57   1.33 1.41   1.17 1.24   1.07 1.11   0.96 1.02
// d = 3 stays above 0.97 up to 280.
xzzx_status coop_is_faster(int d, int64_t n_chains, bool* yes) {
  int n_sm = 0;
  xzzx_status st = sm_count(&n_sm);
  if (st) return st;
  const int pairs = (d + 1) / 2;
  int lanes = 2;
  while (lanes < pairs) lanes *= 2;
  *yes = n_chains <= (int64_t)n_sm * (d == 3 ? 280 : (d <= 15 ? 200 : d <= 23 ? 165 : 205) * pairs / lanes);
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
