// Choice of the annealing kernel on the planar layout (the paper's own lattice;
// Alg. 2 with the Metropolis step of Alg. 3, colour sweep, minimum per colour
// phase).  The literal forms are in anneal_literal.cu.
#include "internal.h"

namespace xzzx {

xzzx_status coop_planar_is_faster(int d, int64_t n_chains, bool* yes);
xzzx_status launch_anneal_coop_planar(const xzzx_code* code, const xzzx_schedule* sched, uint64_t seed, uint64_t shot0,
                                      int n_shots, int restarts, const uint32_t* init, int32_t* best_E,
                                      uint32_t* best_cfg, int32_t* final_E, uint32_t* final_cfg, cudaStream_t stream);
xzzx_status launch_anneal_planar_reg(const xzzx_code* code, const xzzx_schedule* sched, uint64_t seed, uint64_t shot0,
                                     int n_shots, int restarts, const uint32_t* init, int32_t* best_E,
                                     uint32_t* best_cfg, int32_t* final_E, uint32_t* final_cfg, cudaStream_t stream);

// Launch for a planar code (arguments checked by the caller): one thread per chain
// in registers, or several lanes per chain (small launches, and d > 15, where a
// chain's rows outgrow one thread's registers).
xzzx_status launch_anneal_planar(const xzzx_code* code, const xzzx_schedule* sched, uint64_t seed, uint64_t shot0,
                                 int n_shots, int restarts, const uint32_t* init, int32_t* best_E, uint32_t* best_cfg,
                                 int32_t* final_E, uint32_t* final_cfg, cudaStream_t stream) {
  bool coop = false;
  xzzx_status st = coop_planar_is_faster(code->d, (int64_t)n_shots * restarts * 4, &coop);
  if (st) return st;
  return coop ? launch_anneal_coop_planar(code, sched, seed, shot0, n_shots, restarts, init, best_E, best_cfg, final_E,
                                          final_cfg, stream)
              : launch_anneal_planar_reg(code, sched, seed, shot0, n_shots, restarts, init, best_E, best_cfg, final_E,
                                         final_cfg, stream);
}

}  // namespace xzzx
