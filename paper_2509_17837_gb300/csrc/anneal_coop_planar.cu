// Lane-parallel annealing on the planar lattice (anneal_coop.cuh, PlanarLanes).
#include "anneal_coop_launch.cuh"

namespace xzzx {

// Whether a planar launch takes several lanes per chain.  d > 15: always (one
// thread per chain with its rows in shared memory leaves room for two CTAs per SM:
// 131,072 chains x 50 sweeps, 42.4 -> 11.8 ms at d = 17, 242 -> 20.8 ms at d =
// 31).  Below, against the register-resident kernel, 50 sweeps near the
// Nishimori temperature, ms: 8,192 chains 0.12 / 0.08 at d = 3, 0.42 / 0.29 at d
// = 9, 1.05 / 0.41 at d = 15; 32,768 chains 0.12 / 0.19, 0.53 / 0.96, 1.39 / 1.40.
xzzx_status coop_planar_is_faster(int d, int64_t n_chains, bool* yes) {
  int n_sm = 0;
  xzzx_status st = sm_count(&n_sm);
  if (st) return st;
  *yes = d > 15 || n_chains <= (int64_t)n_sm * (d <= 11 ? 64 : 128);
  return XZZX_OK;
}

xzzx_status launch_anneal_coop_planar(const xzzx_code* code, const xzzx_schedule* sched, uint64_t seed, uint64_t shot0,
                                      int n_shots, int restarts, const uint32_t* init, int32_t* best_E,
                                      uint32_t* best_cfg, int32_t* final_E, uint32_t* final_cfg, cudaStream_t stream) {
  const coop::Args A = coop::make_args(code, sched, seed, shot0, n_shots, restarts, init, best_E, best_cfg, final_E,
                                       final_cfg);
  switch (code->d) {
#define XZZX_CASE(DD) \
  case DD:            \
    return coop::launch_g<coop::PlanarLanes<DD>>(A, stream);
    XZZX_CASE(3) XZZX_CASE(5) XZZX_CASE(7) XZZX_CASE(9) XZZX_CASE(11) XZZX_CASE(13) XZZX_CASE(15)
    XZZX_CASE(17) XZZX_CASE(19) XZZX_CASE(21) XZZX_CASE(23) XZZX_CASE(25) XZZX_CASE(27) XZZX_CASE(29)
    XZZX_CASE(31)
#undef XZZX_CASE
    default:
      return fail(XZZX_EUNSUPPORTED, "no annealing kernel for this distance");
  }
}

}  // namespace xzzx
