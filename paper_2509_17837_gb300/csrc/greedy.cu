// Randomised greedy matching (Algs. 5 and 6): the per-launch entry point.
// The per-CTA work is greedy::greedy_cta (greedy_core.cuh).
#include "greedy_core.cuh"

namespace xzzx {
namespace {

using namespace greedy;

struct GreedyArgs {
  DevCode code;
  PhiloxKeys keys;
  uint64_t shot0;
  int n_shots, restarts, randomised, groups, cols, room;
  int32_t Wt_x, Wt_z;
  const uint32_t* syndromes;
  uint32_t* init;
  uint8_t* cbits;
};

template <class G, int kWarps>
__global__ void __launch_bounds__(kWarps * 32, 32 / kWarps) greedy_kernel(const __grid_constant__ GreedyArgs A) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int k = blockIdx.x / A.groups;
  greedy_cta<G, kWarps>(A.code, A.keys, A.shot0 + (uint64_t)k, blockIdx.x % A.groups, A.groups, A.cols, A.room,
                        A.restarts, A.randomised, A.Wt_x, A.Wt_z, A.syndromes + (size_t)k * A.code.sw,
                        A.init + (size_t)k * A.restarts * 2 * A.code.w, A.cbits + (size_t)k * A.restarts, smem);
}

template <class G, int kWarps>
xzzx_status launch_g(const GreedyArgs& A, unsigned grid, size_t smem, cudaStream_t stream) {
  static DeviceOnce once;
  xzzx_status st = once.run([] { return allow_shared(greedy_kernel<G, kWarps>); });
  if (st) return st;
  greedy_kernel<G, kWarps><<<grid, kWarps * 32, smem, stream>>>(A);
  XZZX_CUDA_TRY(cudaGetLastError());
  return XZZX_OK;
}
template <class G>
xzzx_status launch_w(const GreedyArgs& A, int warps, unsigned grid, size_t smem, cudaStream_t stream) {
  return warps == kLargeWarps   ? launch_g<G, kLargeWarps>(A, grid, smem, stream)
         : warps == kSmallWarps ? launch_g<G, kSmallWarps>(A, grid, smem, stream)
                                : launch_g<G, kFewWarps>(A, grid, smem, stream);
}

}  // namespace

xzzx_status launch_greedy(const xzzx_code* code, const xzzx_noise* noise, uint64_t seed, uint64_t shot0, int n_shots,
                          int restarts, int randomised, const uint32_t* syndromes, uint32_t* init, uint8_t* cbits,
                          cudaStream_t stream) {
  NvtxRange nvtx_range("xzzx K1 greedy");
  GreedyArgs A;
  A.code = code->dev;
  A.keys = philox_keys(seed);
  A.shot0 = shot0;
  A.n_shots = n_shots;
  A.restarts = restarts;
  A.randomised = randomised;
  int n_sm = 0;
  xzzx_status st = sm_count(&n_sm);
  if (st) return st;
  const bool scan = randomised != kInitBoundary && scans(A.code, *noise, restarts);
  const int warps = choose_warps(A.code, n_shots, restarts, randomised, scan, n_sm);
  int rpw = 1;
  for (int r = kMaxRestartsPerWarp; r > 1 && rpw == 1 && !scan; r >>= 1)  // a scan has no lists to share
    if ((int64_t)n_shots * greedy_groups(restarts, warps, r) >= min_ctas(is_large(A.code), n_sm)) rpw = r;
  const bool few = few_ctas((int64_t)n_shots * greedy_groups(restarts, warps, 1), n_sm);
  const Cut cut = cut_of(A.code, warps, restarts, randomised, rpw, few, scan);
  A.groups = cut.groups;
  A.cols = cut.cols;
  A.room = cut.room;
  A.Wt_x = noise->Wt_x;
  A.Wt_z = noise->Wt_z;
  A.syndromes = syndromes;
  A.init = init;
  A.cbits = cbits;
  const uint64_t grid = (uint64_t)n_shots * A.groups;
  if (grid > 0x7FFFFFFFull) return fail(XZZX_EINVAL, "too many shots x restarts for one launch");
  return code->layout == kLayoutPlanar ? launch_w<PlanarGeo>(A, warps, (unsigned)grid, cut.smem, stream)
                                       : launch_w<RotGeo>(A, warps, (unsigned)grid, cut.smem, stream);
}

}  // namespace xzzx

using namespace xzzx;

extern "C" xzzx_status xzzx_greedy_init(const xzzx_code* code, const xzzx_noise* noise, uint64_t seed, uint64_t shot0,
                                        int n_shots, int restarts, int randomised, const uint32_t* syndromes,
                                        uint32_t* init, uint8_t* cbits, void* stream) {
  xzzx_status st = check_code(code);
  if (st) return st;
  if (!noise) return fail(XZZX_EINVAL, "noise is NULL");
  if (n_shots < 0) return fail(XZZX_EINVAL, "n_shots < 0");
  if (restarts < 1 || restarts > 65535) return fail(XZZX_EINVAL, "restarts must be in [1, 65535]");
  if (randomised < 0 || randomised > 2) return fail(XZZX_EINVAL, "init mode must be 0, 1 or 2");
  if (noise->Wt_x <= 0 || noise->Wt_z <= 0) return fail(XZZX_EINVAL, "matching weights must be positive");
  if ((int64_t)noise->Wt_x * 4 * code->nq > kInf || (int64_t)noise->Wt_z * 4 * code->nq > kInf)
    return fail(XZZX_EINVAL, "matching weights too large for int32 path lengths");
  if (n_shots == 0) return XZZX_OK;
  if ((st = check_ptr(syndromes, "syndromes")) || (st = check_ptr(init, "init")) || (st = check_ptr(cbits, "cbits")))
    return st;
  return launch_greedy(code, noise, seed, shot0, n_shots, restarts, randomised, syndromes, init, cbits,
                       (cudaStream_t)stream);
}
