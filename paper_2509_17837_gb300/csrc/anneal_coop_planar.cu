// Lane-parallel annealing on the planar lattice (anneal_coop.cuh, PlanarLanes).
#include "anneal_coop_launch.cuh"

namespace xzzx {

// Whether a planar launch takes several lanes per chain.  d > 15: always (one
// thread per chain with its rows in shared memory leaves room for two CTAs per SM:
// 131,072 chains x 50 sweeps, 42.4 -> 11.8 ms at d = 17, 242 -> 20.8 ms at d =
// 31).  Below, against the register-resident kernel, by the share of the lanes that
// hold rows (d of a power of two), at the crossing with dense draws.  Thread time /
// lane time, 50 sweeps near the Nishimori temperature and 200 to 20 times it, at
// chains per SM:
//   d      60          80         100         150         180         200
//   3  1.11 1.19   0.94 1.06   0.78 0.91   0.74 0.79   0.64 0.70   0.53 0.59
//   5  1.41 1.44   1.19 1.22   0.83 0.91   0.72 0.80   0.60 0.69   0.57 0.64
//   7  2.11 2.19   1.52 1.61   1.21 1.43   1.07 1.18   0.93 1.01   0.85 0.93
//   9  1.29 1.59   1.03 1.23   0.81 1.01   0.73 0.93   0.61 0.78   0.56 0.72
//  11  1.51 1.79   1.21 1.41   0.95 1.15   0.84 1.06   0.70 0.92   0.64 0.83
//  13  1.90 2.10   1.52 1.65   1.19 1.35   1.05 1.29   0.88 1.10   0.80 1.00
//  15  2.23 2.40   1.77 1.84   1.39 1.51   1.24 1.47   1.04 1.29   0.95 1.18
xzzx_status coop_planar_is_faster(int d, int64_t n_chains, bool* yes) {
  int n_sm = 0;
  xzzx_status st = sm_count(&n_sm);
  if (st) return st;
  int lanes = 4;
  while (lanes < d) lanes *= 2;
  *yes = d > 15 || n_chains <= (int64_t)n_sm * (d == 3 ? 64 : (8 * d > 6 * lanes ? 190 : 135) * d / lanes);
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
