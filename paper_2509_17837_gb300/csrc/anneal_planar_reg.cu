// Register-resident annealing on the planar layout (colour sweep, minimum per
// colour phase): the planar counterpart of anneal_cta, for d <= 15.
//
// State.  One chain per thread, one 32-bit word per grid row in registers
// (row r holds its d or d-1 qubits as two bits per slot k, column c = 2k +
// (r&1)).  A phase packs the up and down corners of each of its rows' faces into
// one word first (Packed), so a face is two nibbles at shifts fixed by the column
// step, and a move two XORs.
//
// Sweep.  Colour C holds the faces (i, j) with i & 1 = C & 1 and
// ((i+j-1)/2) & 1 = C >> 1.  With m = i >> 1 (the row inside the class) and
// t = j >> 2 (the column step), the faces of one step t sit in every row of
// the class at slot kl = 2t + kl0(m), kl0 alternating with m; their draw block
// (C, t, m>>2) serves four consecutive rows, exactly as four faces of one
// column share a block on the rotated lattice.  The step loop runs at run
// time with the rows unrolled; the edge steps of the odd-row class (left
// boundary at t = 0, right boundary at the last step) are peeled.
//
// Results equal the lane-parallel kernel (same draws, same
// acceptance, same per-phase minimum), which the parity tests check.
#include "anneal_core.cuh"

namespace xzzx {
namespace {

constexpr int kRThreads = 128;
constexpr int kRLut = kSigPlanar;
constexpr uint32_t kPOffNoUp = (uint32_t)(planar_sig_base(kPNoUp) - kSigRot);
constexpr uint32_t kPOffNoDown = (uint32_t)(planar_sig_base(kPNoDown) - kSigRot);
constexpr uint32_t kPOffNoLeft = (uint32_t)(planar_sig_base(kPNoLeft) - kSigRot);
constexpr uint32_t kPOffNoRight = (uint32_t)(planar_sig_base(kPNoRight) - kSigRot);

template <int D>
struct PShape {
  static constexpr int G = 2 * D - 1;
  static constexpr int NQ = D * D + (D - 1) * (D - 1);
  static constexpr int kW = (NQ + 31) / 32;
};

__host__ __device__ constexpr int prow_start(int d, int r) { return (r >> 1) * (2 * d - 1) + ((r & 1) ? d : 0); }
__host__ __device__ constexpr int prow_len(int d, int r) { return (r & 1) ? d - 1 : d; }

struct RegArgs {
  PhiloxKeys keys;
  uint64_t chain0;
  int64_t n_chains;
  int n_sweeps, n_classes, n_live;
  int32_t W[4];
  const uint32_t* T;
  const int2* sig;
  const uint32_t* init;
  int32_t* best_E;
  uint32_t* best_cfg;
  int32_t* final_E;
  uint32_t* final_cfg;
  uint32_t* err;
};

template <int D>
__device__ __forceinline__ void pload(const uint32_t* __restrict__ cfg, uint32_t (&R)[PShape<D>::G]) {
  constexpr int W = PShape<D>::kW;
#pragma unroll
  for (int r = 0; r < PShape<D>::G; ++r) {
    const uint32_t x = core::plane_field(cfg, W, prow_start(D, r), prow_len(D, r));
    const uint32_t z = core::plane_field(cfg + W, W, prow_start(D, r), prow_len(D, r));
    R[r] = (uint32_t)(core::spread2(z) | (core::spread2(x) << 1));
  }
}

template <int D>
__device__ __forceinline__ void pstore(const uint32_t (&R)[PShape<D>::G], uint32_t* __restrict__ cfg) {
  constexpr int W = PShape<D>::kW;
  uint32_t px[W], pz[W];
#pragma unroll
  for (int j = 0; j < W; ++j) px[j] = pz[j] = 0u;
#pragma unroll
  for (int r = 0; r < PShape<D>::G; ++r) {
    const uint32_t fz = core::gather2(R[r]), fx = core::gather2((uint64_t)R[r] >> 1);
    const int start = prow_start(D, r), len = prow_len(D, r), wi = start >> 5, off = start & 31;
    pz[wi] |= fz << off;
    px[wi] |= fx << off;
    if (wi + 1 < W && off + len > 32) {
      pz[wi + 1] |= fz >> (32 - off);
      px[wi + 1] |= fx >> (32 - off);
    }
  }
#pragma unroll
  for (int j = 0; j < W; ++j) {
    cfg[j] = px[j];
    cfg[W + j] = pz[j];
  }
}

// Face kinds of one row at one step.
enum { kKBulk = 0, kKNoUp = 1, kKNoDown = 2, kKNoLeft = 3, kKNoRight = 4, kKNone = 5 };

// kl0 of row m of colour C: the slot of its face at step 0.
template <int C>
__host__ __device__ constexpr int kl0_of(int m) {
  return (C & 1) ? -(((C >> 1) - m - 1) & 1) : (((C >> 1) - m) & 1);
}

// Kind of the face of row m at a step of the given position (0 interior,
// 1 first step of the odd-row class, 2 its last step).
template <int D, int C, int POS>
__host__ __device__ constexpr int kind_of(int m) {
  return (C & 1) == 0 ? (m == 0 ? kKNoUp : (m == D - 1 ? kKNoDown : kKBulk))
                      : (POS == 0 ? kKBulk
                                  : POS == 1 ? (kl0_of<C>(m) == -1 ? kKNoLeft : kKBulk)
                                             : (kl0_of<C>(m) == -1 ? kKNoRight : kKNone));
}

// The up and down corners of the faces of one row and colour, packed for the
// phase.  Their faces use every second slot of the rows above and below (slots of
// parity KL + CL, KL the row's first slot in the colour); U holds the upper row's
// at those slots and the lower row's at the slots between, so that a face's up and
// down bits are a nibble at the bit of its left corner (CL: one slot on).
template <int KL, int CL>
struct Packed {
  static constexpr int P = (KL + CL) & 1;
  static constexpr uint32_t kMask = P ? 0xCCCCCCCCu : 0x33333333u;  // slots of parity P
  __device__ static uint32_t pack(uint32_t up, uint32_t down) {
    return P ? ((up & kMask) >> 2) | (down & kMask) : (up & kMask) | ((down & kMask) << 2);
  }
  // The row above's slots of parity P, and the row below's, from U.
  __device__ static uint32_t up(uint32_t U) { return P ? (U & 0x33333333u) << 2 : U & 0x33333333u; }
  __device__ static uint32_t down(uint32_t U) { return P ? U & 0xCCCCCCCCu : (U & 0xCCCCCCCCu) >> 2; }
};

// All faces of colour C at column step `step` (POS as kind_of) of a sweep; U: the
// packed corners of the class's rows.  A face (row m, slot kl = 2 step + kl0(m))
// has its left and right corners at bit 2 kl of row i = 2m + CL, its up and down
// ones at bit 4 step of U[m] when kl0 + CL is 0 or 1, which the packing arranges.
template <int D, int C, int POS, bool LIVE>
__device__ __forceinline__ void pstep(uint32_t (&R)[PShape<D>::G], uint32_t (&U)[D], int32_t& E, uint32_t Lb,
                                      uint32_t step, const core::SaDraws& dr, const PhiloxKeys& K, uint32_t* err) {
  constexpr int CL = C & 1;
  constexpr int M = CL ? D - 1 : D;
  constexpr int NG = (M + 3) / 4;
  uint2 e[M];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int i = 2 * m + CL;
    const int kind = kind_of<D, C, POS>(m);
    const int sm = 4 * (int)step + 2 * kl0_of<C>(m);
    const uint32_t smid = (uint32_t)(sm < 0 ? 0 : sm);
    e[m] = make_uint2(0u, 0u);
    if (kind == kKNone) continue;
    const uint32_t ud = (U[m] >> (4 * (int)step)) & (kind == kKNoUp ? 0xCu : kind == kKNoDown ? 0x3u : 0xFu);
    uint32_t a;
    // Entry address: 8 (lr | ud << 4), a missing corner closed up; the bulk's
    // products by factors the compiler cannot see, on the multiply pipe.
    if (kind == kKNoLeft) a = ud * 32u + ((R[i] & 3u) * 8u + (Lb + 8u * kPOffNoLeft));
    else if (kind == kKNoRight) a = ud * 32u + (((R[i] >> smid) & 3u) * 8u + (Lb + 8u * kPOffNoRight));
    else if (kind == kKNoUp) a = ud * 32u + (((R[i] >> smid) & 0xFu) * 8u + (Lb + 8u * kPOffNoUp));
    else if (kind == kKNoDown) a = ud * 128u + (((R[i] >> smid) & 0xFu) * 8u + (Lb + 8u * kPOffNoDown));
    else a = ud * K.c128 + (((R[i] >> smid) & 0xFu) * K.c8 + Lb);
    e[m] = XZZX_CHECK(err, a - Lb <= 8u * (kRLut - 1) && !injected(err, XZZX_DEVERR_BOUNDS)) ? core::lds_u2(a)
                                                                                           : make_uint2(0u, 0u);
  }
  uint4 r[NG];
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    uint32_t need = 0;
#pragma unroll
    for (int m = 0; m < M; ++m)
      if ((m >> 2) == g) need |= e[m].y;
    r[g] = make_uint4(0u, 0u, 0u, 0u);
    if (LIVE && __any_sync(0xFFFFFFFFu, need != 0u)) r[g] = dr.block(((uint32_t)C << 16) | (step << 8) | (uint32_t)g, K);
  }
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int kind = kind_of<D, C, POS>(m);
    if (kind == kKNone) continue;
    const int i = 2 * m + CL;
    const int sm = 4 * (int)step + 2 * kl0_of<C>(m);
    const uint32_t smid = (uint32_t)(sm < 0 ? 0 : sm);
    const uint32_t u = lane_of(r[m >> 2], m & 3);
    const int32_t dE = (int32_t)e[m].x;
    if ((dE <= 0) | (LIVE && u < e[m].y)) {
      core::add_energy(E, dE, K);
      if (kind == kKNoLeft) R[i] ^= 2u;
      else if (kind == kKNoRight) R[i] ^= 2u << smid;
      else R[i] ^= 0xAu << smid;
      U[m] ^= (kind == kKNoUp ? 0x4u : kind == kKNoDown ? 0x1u : 0x5u) << (4 * (int)step);
    }
  }
}

// One colour phase: pack the class's neighbours, its column steps, unpack.
template <int D, int C, bool LIVE>
__device__ __forceinline__ void pphase(uint32_t (&R)[PShape<D>::G], int32_t& E, uint32_t Lb, const core::SaDraws& dr,
                                       const PhiloxKeys& K, uint32_t* err) {
  constexpr int CL = C & 1, M = CL ? D - 1 : D, G = PShape<D>::G;
  constexpr int NS = (D - 1) / 2;  // column steps of the even-row class; the odd-row class has NS + 1
  constexpr int K0 = kl0_of<C>(0), K1 = kl0_of<C>(1);  // even and odd m
  uint32_t U[D];
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int i = 2 * m + CL;
    const uint32_t up = i > 0 ? R[i > 0 ? i - 1 : 0] : 0u, dn = i + 1 < G ? R[i + 1 < G ? i + 1 : i] : 0u;
    U[m] = (m & 1) ? Packed<K1, CL>::pack(up, dn) : Packed<K0, CL>::pack(up, dn);
  }
  if (CL == 0) {
#pragma unroll 1
    for (int s = 0; s < NS; ++s) pstep<D, C, 0, LIVE>(R, U, E, Lb, (uint32_t)s, dr, K, err);
  } else {
    pstep<D, C, 1, LIVE>(R, U, E, Lb, 0u, dr, K, err);
#pragma unroll 1
    for (int s = 1; s < NS; ++s) pstep<D, C, 0, LIVE>(R, U, E, Lb, (uint32_t)s, dr, K, err);
    pstep<D, C, 2, LIVE>(R, U, E, Lb, (uint32_t)NS, dr, K, err);
  }
  // The row between face rows m and m + 1: m's lower corners and m + 1's upper ones.
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const int i = 2 * m + CL;
    if (m == 0 && i > 0)  // the row above the class's first: its other slots are untouched
      R[i - 1] = (R[i - 1] & ~Packed<K0, CL>::kMask) | Packed<K0, CL>::up(U[0]);
    if (i + 1 >= G) continue;
    const uint32_t dn = (m & 1) ? Packed<K1, CL>::down(U[m]) : Packed<K0, CL>::down(U[m]);
    if (m + 1 < M) R[i + 1] = dn | ((m & 1) ? Packed<K0, CL>::up(U[m + 1]) : Packed<K1, CL>::up(U[m + 1]));
    else R[i + 1] = (R[i + 1] & ~((m & 1) ? Packed<K1, CL>::kMask : Packed<K0, CL>::kMask)) | dn;
  }
}

// Shared memory: one table per warp, the list of entries whose threshold changes
// per sweep, one configuration per chain.
template <int D>
constexpr size_t reg_smem_bytes() {
  return (kRThreads / 32) * kRLut * sizeof(uint2) + kRLut * sizeof(uint32_t) + 16 +
         (size_t)PShape<D>::G * kRThreads * sizeof(uint32_t);
}

// Bound by the pipe of shifts and logic together with the wide multiplies of the
// draws.  600 shots x 64 restarts, against three-row faces, a table rebuilt every
// sweep and no frozen sweeps: 50 sweeps near the Nishimori temperature d = 9 1.65 ->
// 1.49 ms, d = 15 5.58 -> 4.3 ms; 200 sweeps to 20 times it d = 9 4.95 -> 4.09 ms, d =
// 15 18.7 -> 14.6 ms.  Held to seven CTAs per SM (72 registers) d = 9 takes 1.56 ms.
template <int D>
__global__ void __launch_bounds__(kRThreads, 1) anneal_planar_reg_kernel(const __grid_constant__ RegArgs A) {
  constexpr int G = PShape<D>::G;
  constexpr int W = PShape<D>::kW;
  extern __shared__ __align__(16) uint8_t smem[];
  const int tid = threadIdx.x, lane = tid & 31;
  uint32_t* upd = reinterpret_cast<uint32_t*>(smem + (kRThreads / 32) * kRLut * sizeof(uint2));
  int* n_upd_s = reinterpret_cast<int*>(upd + kRLut);
  uint32_t* kept = reinterpret_cast<uint32_t*>(n_upd_s + 4);  // [G][kRThreads]
  const uint32_t L0 = (uint32_t)__cvta_generic_to_shared(smem), Lb = L0 + (uint32_t)(tid >> 5) * kRLut * 8u;
  const int64_t c_raw = (int64_t)blockIdx.x * kRThreads + tid;
  const bool active = c_raw < A.n_chains;
  const int64_t c = active ? c_raw : A.n_chains - 1;  // inactive threads shadow a real chain
  const uint64_t chain = A.chain0 + (uint64_t)c;
  const int P = (int)(c & 3);

  // Every warp's table for the first sweep, in full, and the list of the entries
  // whose threshold changes.
  if (tid == 0) n_upd_s[0] = 0;
  __syncthreads();
  static_assert(kRLut % kRThreads == 0, "whole warps in every pass");
  for (int k = tid; k < kRLut; k += kRThreads) {
    const int2 sg = __ldg(&A.sig[kSigRot + k]);
    const uint2 entry = make_uint2((uint32_t)sg.x, sg.y >= 0 && A.n_sweeps > 0 ? __ldg(&A.T[sg.y]) : 0u);
#pragma unroll
    for (int w = 0; w < kRThreads / 32; ++w) core::sts_u2(L0 + (uint32_t)(w * kRLut + k) * 8u, entry);
    core::append_entry(sg.y >= 0, ((uint32_t)k << 16) | (uint32_t)sg.y, upd, n_upd_s);
  }
  __syncthreads();  // the last CTA barrier: warps then sweep independently
  const int n_upd = n_upd_s[0];

  uint32_t R[G];
  pload<D>(A.init + (size_t)(c >> 2) * 2 * W, R);
  // L_X: X on column 0 (slot 0 of the even rows); L_Z: Z on every qubit of row 0.
  if (P == 1 || P == 2) {
#pragma unroll
    for (int r = 0; r < G; r += 2) R[r] ^= 2u;
  }
  if (P == 2 || P == 3) R[0] ^= (uint32_t)(0x55555555u & ((1u << (2 * D)) - 1u));
  int32_t nx = 0, ny = 0, nz = 0;
#pragma unroll
  for (int r = 0; r < G; ++r) {
    const uint32_t z = R[r] & 0x55555555u, x = (R[r] >> 1) & 0x55555555u;
    ny += __popc(x & z);
    nx += __popc(x & ~z);
    nz += __popc(z & ~x);
  }
  int32_t E = nx * A.W[2] + ny * A.W[3] + nz * A.W[1];
  int32_t E_best = E;
  const bool keep = A.best_cfg != nullptr;
  auto save = [&] {
#pragma unroll
    for (int r = 0; r < G; ++r) kept[r * kRThreads + tid] = R[r];
  };
  if (keep) save();

  core::SaDraws dr;
  dr.init((uint32_t)chain, kTagSA | ((uint32_t)(chain >> 32) << 8), A.keys);
#define XZZX_PPHASE(CC, LIVE)                               \
  pphase<D, CC, LIVE>(R, E, Lb, dr, A.keys, A.err);         \
  if (E < E_best) {                                         \
    E_best = E;                                             \
    if (keep) save();                                       \
  }
  for (int t = 0; t < A.n_live; ++t) {
    dr.sweep((uint32_t)t, A.keys);
    XZZX_PPHASE(0, true)
    XZZX_PPHASE(1, true)
    XZZX_PPHASE(2, true)
    XZZX_PPHASE(3, true)
    if (t + 1 < A.n_live) {  // next sweep's thresholds, once every lane is done with these
      __syncwarp();
      core::update_lut_pair(Lb, upd, n_upd, A.T + (size_t)(t + 1) * A.n_classes, lane);
      __syncwarp();
    }
  }
  // The frozen sweeps (see anneal_core.cuh); the saved configuration takes the
  // place of the minimum's when nobody asks for that.
  const bool may_stop = !A.final_E && !A.final_cfg && !keep;
  bool done = false;
  for (int t = A.n_live, i = 0; t < A.n_sweeps; ++t, ++i) {
    if (may_stop && (i & (i + 1)) == 0) save();
    XZZX_PPHASE(0, false)
    XZZX_PPHASE(1, false)
    XZZX_PPHASE(2, false)
    XZZX_PPHASE(3, false)
    if (may_stop) {
      uint32_t diff = 0;
#pragma unroll
      for (int r = 0; r < G; ++r) diff |= R[r] ^ kept[r * kRThreads + tid];
      done |= diff == 0u;
      if (__all_sync(0xFFFFFFFFu, done)) break;
    }
  }
#undef XZZX_PPHASE

  if (!active) return;
  A.best_E[c] = E_best;
  if (A.final_E) A.final_E[c] = E;
  if (A.final_cfg) pstore<D>(R, A.final_cfg + (size_t)c * 2 * W);
  if (keep) {
#pragma unroll
    for (int r = 0; r < G; ++r) R[r] = kept[r * kRThreads + tid];
    pstore<D>(R, A.best_cfg + (size_t)c * 2 * W);
  }
}

template <int D>
xzzx_status launch_d(const RegArgs& A, cudaStream_t stream) {
  const size_t smem = reg_smem_bytes<D>();
  static DeviceOnce once;
  xzzx_status st = once.run([&]() -> xzzx_status {
    XZZX_CUDA_TRY(cudaFuncSetAttribute(anneal_planar_reg_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem));
    return XZZX_OK;
  });
  if (st) return st;
  const int64_t grid = (A.n_chains + kRThreads - 1) / kRThreads;
  if (grid > 0x7FFFFFFF) return fail(XZZX_EINVAL, "too many chains for one launch");
  anneal_planar_reg_kernel<D><<<(unsigned)grid, kRThreads, smem, stream>>>(A);
  XZZX_CUDA_TRY(cudaGetLastError());
  return XZZX_OK;
}

}  // namespace

// Colour sweep with per-phase minima on a planar code, d <= 15 (arguments
// checked by the caller).
xzzx_status launch_anneal_planar_reg(const xzzx_code* code, const xzzx_schedule* sched, uint64_t seed, uint64_t shot0,
                                     int n_shots, int restarts, const uint32_t* init, int32_t* best_E,
                                     uint32_t* best_cfg, int32_t* final_E, uint32_t* final_cfg, cudaStream_t stream) {
  RegArgs A;
  A.keys = philox_keys(seed);
  A.chain0 = shot0 * (uint64_t)restarts * 4u;
  A.n_chains = (int64_t)n_shots * restarts * 4;
  A.n_sweeps = sched->n_sweeps;
  A.n_classes = sched->n_classes;
  A.n_live = sched->n_live[kLayoutPlanar];
  for (int k = 0; k < 4; ++k) A.W[k] = sched->noise.W[k];
  A.T = sched->d_T;
  A.sig = sched->d_sig;
  A.init = init;
  A.best_E = best_E;
  A.best_cfg = best_cfg;
  A.final_E = final_E;
  A.final_cfg = final_cfg;
  A.err = code->dev.err;
  switch (code->d) {
    case 3: return launch_d<3>(A, stream);
    case 5: return launch_d<5>(A, stream);
    case 7: return launch_d<7>(A, stream);
    case 9: return launch_d<9>(A, stream);
    case 11: return launch_d<11>(A, stream);
    case 13: return launch_d<13>(A, stream);
    case 15: return launch_d<15>(A, stream);
    default: return fail(XZZX_EUNSUPPORTED, "no register-resident planar kernel for this distance");
  }
}

}  // namespace xzzx
