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

template <class Geo, int NC, int NP, int PER>
__global__ void __launch_bounds__(Form<Geo, NC, NP, PER>::kThreads, Form<Geo, NC, NP, PER>::kRegCtas)
    anneal_coop_kernel(const __grid_constant__ Args A) {
  constexpr int kCta = Form<Geo, NC, NP, PER>::kCtaChains;
  extern __shared__ __align__(16) uint8_t smem[];
  const int64_t first = (int64_t)blockIdx.x * kCta;
  const core::ChainOut out{A.best_E, A.best_cfg, A.final_E, A.final_cfg};
  anneal_coop_cta<Geo, NC, NP, PER>(A.init, A.chain0, first, (int)min((int64_t)kCta, A.n_chains - first), out, A.tab,
                                   A.keys, smem);
}

template <class Geo, int NC, int NP, int PER>
xzzx_status launch_form(const Args& A, cudaStream_t stream) {
  using F = Form<Geo, NC, NP, PER>;
  static DeviceOnce once;
  xzzx_status st = once.run([] { return allow_shared(anneal_coop_kernel<Geo, NC, NP, PER>); });
  if (st) return st;
  const int64_t grid = (A.n_chains + F::kCtaChains - 1) / F::kCtaChains;
  if (grid > 0x7FFFFFFF) return fail(XZZX_EINVAL, "too many chains for one launch");
  anneal_coop_kernel<Geo, NC, NP, PER><<<(unsigned)grid, F::kThreads, F::smem_bytes(A.tab.n_classes), stream>>>(A);
  XZZX_CUDA_TRY(cudaGetLastError());
  return XZZX_OK;
}
// CTAs per SM of the producing form for this launch, or 0.  It runs while every
// CTA (one sweeping warp, kChains chains) is resident at once: sized for three
// per SM, else for four (fewer sweeps per set, so more barriers); past that its
// unconditional draws cost more issue slots than they save, and four sweeping
// warps per CTA share the tables.  200 sweeps, CTAs per SM 1, 3, 4, 6, ms: d = 11
// sized for three 0.088, 0.124, 0.191, 0.228, for four 0.093, 0.125, 0.145, 0.230,
// plain form 0.204, 0.209, 0.212, 0.247; planar d = 25 0.251, 0.304, 0.525, 0.594;
// 0.217, 0.276, 0.313, 0.559; 0.468, 0.469, 0.468, 0.583.
template <class Geo>
int producing_per_sm(int64_t n_chains, int n_sm) {
  const int64_t ctas = (n_chains + Geo::kChains - 1) / Geo::kChains;
  return ctas <= 3 * n_sm ? 3 : ctas <= 4 * n_sm ? 4 : 0;
}

// CTAs per SM that the form where every warp sweeps is sized for.  Where that
// changes its sweeps per set (planar: 8 at three, 4 at four) it is three while no more
// are wanted -- fewer barriers -- and at d = 13, 15 where five or six would leave one
// or two behind four.  Form sized for four / for three, ms, 30 sweeps near the
// Nishimori temperature, d = 5: two CTAs per SM 0.050 / 0.045, four 0.079 / 0.100; 60
// sweeps to 20 times it, d = 13: four 0.200 / 0.270, five 0.310 / 0.283, six 0.334 /
// 0.317, eight 0.390 / 0.427.
template <class Geo>
int sweeping_per_sm(int64_t n_chains, int n_sm) {
  const int64_t ctas = (n_chains + 4 * Geo::kChains - 1) / (4 * Geo::kChains), c = (ctas + n_sm - 1) / n_sm;
  return c <= 3 || ((c == 5 || c == 6) && Geo::kByThree) ? 3 : 4;
}

template <class Geo>
xzzx_status launch_g(const Args& A, cudaStream_t stream) {
  int n_sm = 0;
  xzzx_status st = sm_count(&n_sm);
  if (st) return st;
  const int per = producing_per_sm<Geo>(A.n_chains, n_sm);
  if (per) return per == 3 ? launch_form<Geo, 1, 3, 3>(A, stream) : launch_form<Geo, 1, 3, 4>(A, stream);
  if constexpr (Form<Geo, 4, 0, 3>::kSweeps != Form<Geo, 4, 0, 4>::kSweeps)
    if (sweeping_per_sm<Geo>(A.n_chains, n_sm) == 3) return launch_form<Geo, 4, 0, 3>(A, stream);
  return launch_form<Geo, 4, 0, 4>(A, stream);
}

}  // namespace
}  // namespace coop
}  // namespace xzzx
