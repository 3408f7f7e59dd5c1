// Launches of the lane-parallel annealing kernel (anneal_coop.cuh): one code
// and schedule (xzzx_anneal_warp, and xzzx_anneal when its chains do not fill
// the GPU one per thread), and batches (batch mode 2, the server's small
// batches).
#include "anneal_coop.cuh"
#include "batch_internal.h"

#include <algorithm>

namespace xzzx {

xzzx_status check_anneal_args(const xzzx_code*, const xzzx_schedule*, int, int);

namespace coop {
namespace {

struct Args {
  PhiloxKeys keys;
  uint64_t chain0;
  int64_t n_chains;
  core::SweepTables tab;
  const uint32_t* init;
  int32_t* best_E;
  uint32_t* best_cfg;
  int32_t* final_E;
  uint32_t* final_cfg;
};

// Resident CTAs per SM the forms are register-bounded for (what their shared
// memory allows).
template <int D, int NP>
constexpr int kMinCtas = NP ? 3 : 4;

template <int D, int NC, int NP>
__global__ void __launch_bounds__(Form<D, NC, NP>::kThreads, kMinCtas<D, NP>) anneal_coop_kernel(const __grid_constant__ Args A) {
  constexpr int kCta = Form<D, NC, NP>::kCtaChains;
  extern __shared__ __align__(16) uint8_t smem[];
  const int64_t first = (int64_t)blockIdx.x * kCta;
  const core::ChainOut out{A.best_E, A.best_cfg, A.final_E, A.final_cfg};
  anneal_coop_cta<D, NC, NP>(A.init, A.chain0, first, (int)min((int64_t)kCta, A.n_chains - first), out, A.tab, A.keys,
                             smem);
}

// Batched form: the chunks of one distance, each cut into CTAs of kCtaChains
// chains (so a CTA's chains share a segment and its thresholds).
template <int D, int NC, int NP>
__global__ void __launch_bounds__(Form<D, NC, NP>::kThreads, kMinCtas<D, NP>)
    coop_chunks_kernel(const __grid_constant__ batch::CoopLaunch L) {
  constexpr int kCta = Form<D, NC, NP>::kCtaChains;
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
  anneal_coop_cta<D, NC, NP>(sg.init, sg.shot0 * (uint64_t)sg.restarts * 4u, (int64_t)ch.first_chain + first,
                             min(kCta, ch.n_chains - first), out, tab, L.keys, smem);
}

xzzx_status sm_count(int* n_sm) {
  int dev = 0;
  XZZX_CUDA_TRY(cudaGetDevice(&dev));
  XZZX_CUDA_TRY(cudaDeviceGetAttribute(n_sm, cudaDevAttrMultiProcessorCount, dev));
  return XZZX_OK;
}

xzzx_status shared_limit(int* optin) {
  int dev = 0;
  XZZX_CUDA_TRY(cudaGetDevice(&dev));
  XZZX_CUDA_TRY(cudaDeviceGetAttribute(optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  return XZZX_OK;
}

// Allow a kernel the device's whole shared memory (the tables of a schedule
// with many energy classes, or an occupancy cap's padding).
template <typename F>
xzzx_status allow_shared(F kernel) {
  int optin = 0;
  xzzx_status st = shared_limit(&optin);
  if (st) return st;
  XZZX_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
  XZZX_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)cudaSharedmemCarveoutMaxShared));
  return XZZX_OK;
}

template <int D, int NC, int NP>
xzzx_status launch_form(const Args& A, cudaStream_t stream) {
  using F = Form<D, NC, NP>;
  static DeviceOnce once;
  xzzx_status st = once.run([] { return allow_shared(anneal_coop_kernel<D, NC, NP>); });
  if (st) return st;
  const int64_t grid = (A.n_chains + F::kCtaChains - 1) / F::kCtaChains;
  if (grid > 0x7FFFFFFF) return fail(XZZX_EINVAL, "too many chains for one launch");
  anneal_coop_kernel<D, NC, NP><<<(unsigned)grid, F::kThreads, F::smem_bytes(A.tab.n_classes), stream>>>(A);
  XZZX_CUDA_TRY(cudaGetLastError());
  return XZZX_OK;
}
// The producing form runs while every CTA (one sweeping warp, kChains chains)
// is resident at once, about three per SM; past that its unconditional draws
// cost more issue slots than they save, and four sweeping warps per CTA share
// the tables.  400 sweeps at d = 11, producing / plain form, ms: 0.24 / 0.46 at
// 128 chains, 0.30 / 0.50 at 1024, 0.40 / 0.49 at 2048, 0.69 / 0.59 at 4096.
template <int D>
bool producing(int64_t n_chains, int n_sm) {
  return n_chains <= (int64_t)3 * n_sm * Form<D, 1, 3>::kCtaChains;
}

template <int D>
xzzx_status launch_d(const Args& A, cudaStream_t stream) {
  int n_sm = 0;
  xzzx_status st = sm_count(&n_sm);
  if (st) return st;
  return producing<D>(A.n_chains, n_sm) ? launch_form<D, 1, 3>(A, stream) : launch_form<D, 4, 0>(A, stream);
}

template <int D, int NC, int NP>
xzzx_status chunks_form(const batch::CoopLaunch& L, cudaStream_t stream) {
  using F = Form<D, NC, NP>;
  static DeviceOnce once;
  xzzx_status st = once.run([] { return allow_shared(coop_chunks_kernel<D, NC, NP>); });
  if (st) return st;
  const size_t smem = std::max(F::smem_bytes(L.n_classes), (size_t)std::max(L.smem, 0));
  const int64_t grid = (int64_t)L.n_chunks * (L.nt / F::kCtaChains);
  if (grid > 0x7FFFFFFF) return fail(XZZX_EINVAL, "too many chains for one launch");
  coop_chunks_kernel<D, NC, NP><<<(unsigned)grid, F::kThreads, smem, stream>>>(L);
  XZZX_CUDA_TRY(cudaGetLastError());
  return XZZX_OK;
}
template <int D>
xzzx_status chunks_d(const batch::CoopLaunch& L, cudaStream_t stream) {
  if (L.n_chunks <= 0) return XZZX_OK;
  int n_sm = 0;
  xzzx_status st = sm_count(&n_sm);
  if (st) return st;
  // An occupancy cap (L.smem) is one of the plain form's CTAs.
  return L.smem == 0 && producing<D>((int64_t)L.n_chunks * L.nt, n_sm) ? chunks_form<D, 1, 3>(L, stream)
                                                                       : chunks_form<D, 4, 0>(L, stream);
}

template <int D>
xzzx_status configure_d(int cap, int n_classes, int* smem_out, int* ctas_per_sm) {
  using F = Form<D, 4, 0>;
  xzzx_status st = allow_shared(coop_chunks_kernel<D, 4, 0>);
  if (st) return st;
  size_t smem = F::smem_bytes(n_classes);
  int dev = 0, per_sm_bytes = 0, reserved = 0, optin = 0;
  if ((st = shared_limit(&optin))) return st;
  XZZX_CUDA_TRY(cudaGetDevice(&dev));
  XZZX_CUDA_TRY(cudaDeviceGetAttribute(&per_sm_bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
  XZZX_CUDA_TRY(cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev));
  if (cap > 0) {
    const long pad = ((long)per_sm_bytes / cap - reserved) & ~15L;
    smem = std::max(smem, (size_t)std::min<long>(pad, optin));
  }
  XZZX_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, coop_chunks_kernel<D, 4, 0>, F::kThreads, smem));
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
  coop::Args A;
  A.keys = philox_keys(seed);
  A.chain0 = shot0 * (uint64_t)restarts * 4u;
  A.n_chains = (int64_t)n_shots * restarts * 4;
  A.tab.T = sched->d_T;
  A.tab.sig = sched->d_sig;
  A.tab.n_sweeps = sched->n_sweeps;
  A.tab.n_classes = sched->n_classes;
  A.tab.n_live = sched->n_live[kLayoutRotated];
  for (int k = 0; k < 4; ++k) A.tab.W[k] = sched->noise.W[k];
  A.tab.err = code->dev.err;
  A.init = init;
  A.best_E = best_E;
  A.best_cfg = best_cfg;
  A.final_E = final_E;
  A.final_cfg = final_cfg;
  switch (code->d) {
#define XZZX_CASE(DD) \
  case DD:            \
    return coop::launch_d<DD>(A, stream);
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
    return coop::configure_d<DD>(cap, n_classes, smem, ctas_per_sm);
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
    return coop::chunks_d<DD>(L, stream);
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
