// Launch of the lane-parallel annealing kernel over one geometry's chains, shared
// by the units that instantiate it.
#pragma once

#include "anneal_coop.cuh"

namespace xzzx {
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

inline Args make_args(const xzzx_code* code, const xzzx_schedule* sched, uint64_t seed, uint64_t shot0, int n_shots,
                      int restarts, const uint32_t* init, int32_t* best_E, uint32_t* best_cfg, int32_t* final_E,
                      uint32_t* final_cfg) {
  Args A;
  A.keys = philox_keys(seed);
  A.chain0 = shot0 * (uint64_t)restarts * 4u;
  A.n_chains = (int64_t)n_shots * restarts * 4;
  A.tab.T = sched->d_T;
  A.tab.sig = sched->d_sig;
  A.tab.n_sweeps = sched->n_sweeps;
  A.tab.n_classes = sched->n_classes;
  A.tab.n_live = sched->n_live[code->layout];
  for (int k = 0; k < 4; ++k) A.tab.W[k] = sched->noise.W[k];
  A.tab.err = code->dev.err;
  A.init = init;
  A.best_E = best_E;
  A.best_cfg = best_cfg;
  A.final_E = final_E;
  A.final_cfg = final_cfg;
  return A;
}

// Resident CTAs per SM the forms are register-bounded for (what their shared
// memory allows).
template <int NP, int KB>
constexpr int kMinCtas = NP && KB > 52 ? 3 : 4;

template <class Geo, int NC, int NP, int KB>
__global__ void __launch_bounds__(Form<Geo, NC, NP, KB>::kThreads, kMinCtas<NP, KB>)
    anneal_coop_kernel(const __grid_constant__ Args A) {
  constexpr int kCta = Form<Geo, NC, NP, KB>::kCtaChains;
  extern __shared__ __align__(16) uint8_t smem[];
  const int64_t first = (int64_t)blockIdx.x * kCta;
  const core::ChainOut out{A.best_E, A.best_cfg, A.final_E, A.final_cfg};
  anneal_coop_cta<Geo, NC, NP, KB>(A.init, A.chain0, first, (int)min((int64_t)kCta, A.n_chains - first), out, A.tab,
                                   A.keys, smem);
}

xzzx_status sm_count(int* n_sm) {
  int dev = 0;
  XZZX_CUDA_TRY(cudaGetDevice(&dev));
  XZZX_CUDA_TRY(cudaDeviceGetAttribute(n_sm, cudaDevAttrMultiProcessorCount, dev));
  return XZZX_OK;
}

template <class Geo, int NC, int NP, int KB>
xzzx_status launch_form(const Args& A, cudaStream_t stream) {
  using F = Form<Geo, NC, NP, KB>;
  static DeviceOnce once;
  xzzx_status st = once.run([] { return allow_shared(anneal_coop_kernel<Geo, NC, NP, KB>); });
  if (st) return st;
  const int64_t grid = (A.n_chains + F::kCtaChains - 1) / F::kCtaChains;
  if (grid > 0x7FFFFFFF) return fail(XZZX_EINVAL, "too many chains for one launch");
  anneal_coop_kernel<Geo, NC, NP, KB><<<(unsigned)grid, F::kThreads, F::smem_bytes(A.tab.n_classes), stream>>>(A);
  XZZX_CUDA_TRY(cudaGetLastError());
  return XZZX_OK;
}
// The producing form runs while every CTA (one sweeping warp, kChains chains)
// is resident at once: three per SM with sets of 72 KB, four with sets of 52 KB
// (fewer sweeps each, so more barriers); past that its unconditional draws cost
// more issue slots than they save, and four sweeping warps per CTA share the
// tables.  400 sweeps at d = 11, producing / plain form, ms: 0.24 / 0.46 at 128
// chains, 0.30 / 0.50 at 1024, 0.40 / 0.49 at 2048, 0.69 / 0.59 at 4096; one set of
// 52 KB instead of 72: 0.26 at 128 chains.
template <class Geo>
int producing_kb(int64_t n_chains, int n_sm) {
  const int64_t ctas = (n_chains + Geo::kChains - 1) / Geo::kChains;
  return ctas <= 3 * n_sm ? 72 : ctas <= 4 * n_sm ? 52 : 0;
}

template <class Geo>
xzzx_status launch_g(const Args& A, cudaStream_t stream) {
  int n_sm = 0;
  xzzx_status st = sm_count(&n_sm);
  if (st) return st;
  const int kb = producing_kb<Geo>(A.n_chains, n_sm);
  return kb == 72   ? launch_form<Geo, 1, 3, 72>(A, stream)
         : kb == 52 ? launch_form<Geo, 1, 3, 52>(A, stream)
                    : launch_form<Geo, 4, 0, 72>(A, stream);
}

}  // namespace
}  // namespace coop
}  // namespace xzzx
