// Lane-parallel annealing (the colour sweep of Alg. 2 / Alg. 3 with several
// lanes per chain), for launches whose chains do not fill the GPU one per
// thread.
//
// State.  Lane k of a chain's group of G lanes (G = 2, 4, 8 or 16, the power of
// two at or above the H = (d+1)/2 pairs of rows) holds one pair word of the
// layout of anneal_core.cuh: rows 2k and 2k+1 (even layout, colours 0 and 2) or
// rows 2k-1 and 2k (odd layout, colours 1 and 3), four bits per column in one
// to four registers.  Every face of a colour then lies inside one lane's word,
// a layout change is one shuffle per register, and a lane takes the faces of
// its pair of rows, column by column, with every shift a compile-time constant.
// The face row of lane k has draw coordinate ia = k in all four colours.
//
// Draws.  The block of a column serves the four rows of a quad of lanes, so the
// quad computes four columns' blocks at once, one per lane, and trades words
// through shared memory (quads 20 words apart: conflict-free).
//
// Acceptance table.  One table of (dE, A) per sweep for the whole CTA, 512
// entries in pair order, kept for kSweeps sweeps at a time: the thresholds of
// the next kSweeps sweeps are copied in asynchronously while these run, so the
// warps meet at two barriers per kSweeps sweeps and none of them rebuilds a
// table.  Entry order: 256 bulk signatures (TL | BL << 2 | TR << 4 | BR << 6);
// then 256 "edge" ones: a top face keeps its byte's bits 2-3 and 6-7, a bottom
// face bits 0-1 and 4-5 (both give the all-identity entry at 0); the left and
// right boundary nibbles and the entry of idle lanes (never accepted) fill
// index ranges that neither can reach.
//
// Minimum.  A chain's energy is kept as one partial sum per lane.  A phase can
// only set a new minimum if some lane's change is negative, so the sums over
// the group after each phase of a sweep are taken, at its end, only when a vote
// finds one.
//
// What bounds it: at one warp per scheduler the dependent chain of a phase
// (layout shuffle, table load, compare) and the issue slots of its lanes'
// faces, not throughput; the one-thread-per-chain kernel spends a sweep's whole
// work on that chain.
#pragma once

#include "anneal_core.cuh"

namespace xzzx {
namespace coop {

constexpr int kEntries = 512;               // entries of one sweep's table
constexpr uint32_t kTable = kEntries * 8u;  // bytes of one sweep's table
constexpr uint32_t kEdge = 256u * 8u, kLeft = (256u + 0x50u) * 8u, kRight = (256u + 0x90u) * 8u,
                   kIdle = (256u + 0x60u) * 8u;
constexpr int kBatchWords = 128;            // one batch of a warp's draws

template <int D>
struct Shape {
  static constexpr int H = (D + 1) / 2;
  static constexpr int NW = (4 * D + 31) / 32;
  static constexpr int G = H <= 2 ? 2 : H <= 4 ? 4 : H <= 8 ? 8 : 16;  // lanes per chain
  static constexpr int kChains = 32 / G;                              // chains per warp
  static constexpr int Q = G < 4 ? G : 4;                             // columns drawn at once
  // Batches of draws of the four phases of a sweep, and where each phase's begin.
  static constexpr int NCB = (D - 1) / 2, kB0 = (NCB + Q - 1) / Q, kB1 = (NCB + Q) / Q;
  static constexpr int kBatches = 2 * (kB0 + kB1);
  static constexpr int kW = (D * D + 31) / 32;
};

// Entry of the schedule's rotated signature table for table index p, -1 for
// the entry of idle lanes and unreachable indices.
__device__ __forceinline__ int sig_source(int p) {
  if (p < 256) return core::pair_sig_source(p);
  const int e = p - 256;
  if ((e & 0x33) == 0) return sig_base(kTop) + (((e >> 2) & 3) | (((e >> 6) & 3) << 2));
  if ((e & 0xCC) == 0) return sig_base(kBottom) + ((e & 3) | (((e >> 4) & 3) << 2));
  if ((e & 0xF0) == 0x50) return sig_base(::xzzx::kLeft) + (e & 15);
  if ((e & 0xF0) == 0x90) return sig_base(::xzzx::kRight) + (e & 15);
  return -1;
}

// A launch form: NC warps that sweep and NP warps that produce for them, per
// CTA.  NP = 0: every warp sweeps, draws its own blocks where a vote finds a
// need, and the CTA rebuilds the tables of the next kSweeps sweeps together.
// NP > 0: the producing warps draw every block of the next kSweeps sweeps and
// write their tables while the sweeping warps run the current ones from shared
// memory (two sets of each).
template <int D, int NC, int NP>
struct Form {
  static constexpr int kThreads = 32 * (NC + NP);
  static constexpr int kCtaChains = NC * Shape<D>::kChains;
  static constexpr int kSets = NP ? 2 : 1;
  // sweeps per set: as many as keep them within 72 KB (three CTAs per SM)
  static constexpr int kDrawBytes = NP ? NC * Shape<D>::kBatches * kBatchWords * 4 : 0;
  static constexpr int kFit = 72 * 1024 / (kSets * ((int)kTable + kDrawBytes));
  static constexpr int kSweeps = kFit >= 8 ? 8 : kFit >= 4 ? 4 : kFit >= 2 ? 2 : 1;
  static constexpr int kDrawWords = NP ? kSets * kSweeps * NC * Shape<D>::kBatches * kBatchWords
                                       : NC * 2 * kBatchWords;
  // Dynamic shared memory: alignment slack, the tables, the list of entries
  // with a threshold, the draws, the output staging of each chain and, for NP =
  // 0, the raw thresholds of the next kSweeps sweeps.
  static constexpr size_t smem_bytes(int n_classes) {
    return kTable + (size_t)kSets * kSweeps * kTable + kEntries * sizeof(uint32_t) + 16 + (size_t)kDrawWords * 4 +
           (size_t)kCtaChains * 2 * Shape<D>::kW * 4 + (NP ? 0 : (size_t)kSweeps * n_classes * 4);
  }
};

// Constants of a lane for one colour: byte mask and table offset of its faces
// (idle lanes: the entry that is never accepted) and the rows a move changes.
struct LaneColour {
  uint32_t mask, base, rows;
};

template <int D, int C>
__device__ __forceinline__ LaneColour lane_colour(int k) {
  constexpr int H = Shape<D>::H;
  LaneColour c;
  const bool on = k < H && !(C == 1 && k == 0) && !(C == 2 && k == H - 1);
  const bool top = C == 3 && k == 0, bottom = C == 0 && k == H - 1;
  c.mask = on ? 0x7F8u : 0u;
  c.base = !on ? kIdle : (top || bottom) ? kEdge : 0u;
  c.rows = top ? 0xCCCCCCCCu : bottom ? 0x33333333u : 0xFFFFFFFFu;
  if (top) c.mask &= 0xCCu << 3;
  if (bottom) c.mask &= 0x33u << 3;
  return c;
}

// Table byte offset of the face at column b (-1: the left boundary nibble, d-1:
// the right one) of word w, before the lane's mask.
template <int D, int B, int NW>
__device__ __forceinline__ uint32_t face_bits(const uint32_t (&w)[NW]) {
  if constexpr (B < 0) {
    return w[0] << 3;
  } else {
    constexpr int RG = (4 * B) >> 5, OFF = (4 * B) & 31;
    if constexpr (OFF == 0) return w[RG] << 3;
    else if constexpr (OFF == 28 && RG + 1 < NW) return __funnelshift_r(w[RG], w[RG + 1], 25);
    else return w[RG] >> (OFF - 3);
  }
}

template <int D, int B, int NW>
__device__ __forceinline__ void face_flip(uint32_t (&w)[NW], uint32_t rows) {
  if constexpr (B < 0) {
    w[0] ^= 0x9u;  // Z on TR, X on BR
  } else {
    constexpr int RG = (4 * B) >> 5, OFF = (4 * B) & 31;
    if constexpr (B == D - 1) {
      w[RG] ^= 0x6u << OFF;  // X on TL, Z on BL
    } else {
      w[RG] ^= (0x96u << OFF) & rows;  // X on TL, Z on BL, Z on TR, X on BR
      if constexpr (OFF == 28) w[RG + 1] ^= (0x96u >> 4) & rows;
    }
  }
}

__device__ __forceinline__ uint2 table_entry(uint32_t a, uint32_t tbl, uint32_t* err) {
  return XZZX_CHECK(err, a - tbl <= kTable - 8u && !injected(err, XZZX_DEVERR_BOUNDS)) ? core::lds_u2(a)
                                                                                       : make_uint2(0u, 0u);
}

// Column ib of colour C (the draw coordinate) as the face column b.
template <int C>
__host__ __device__ constexpr int column_of(int ib) {
  return (C >> 1) == 0 ? 2 * ib : 2 * ib - 1;
}

// Compile-time loop over n columns from IB.
template <int IB, int N, typename F>
__device__ __forceinline__ void for_columns(F&& f) {
  if constexpr (N > 0) {
    f(std::integral_constant<int, IB>{});
    for_columns<IB + 1, N - 1>(f);
  }
}

// The columns of colour C: draw coordinates ib in [first, first + n).
template <int D, int C>
struct Columns {
  static constexpr int NCB = (D - 1) / 2;
  static constexpr int first = C == 3 ? 1 : 0;
  static constexpr int n = (C == 0 ? NCB - 1 : NCB) - first + 1;
  static constexpr int batches = (n + Shape<D>::Q - 1) / Shape<D>::Q;
};
// One batch of draws for the lanes of a warp: each lane computes one column's
// block of its chain and hands the quad's four lanes (G = 2: the pair) their
// words, so that lane l finds the draws of columns first, first + 1, ... of the
// batch at x[Q l], x[Q l + 1], ...  c0: the block's counter word.
template <int D>
__device__ __forceinline__ void draw_batch(uint32_t c0, const core::SaDraws& dr, const PhiloxKeys& K, uint32_t* x,
                                           int lane) {
  constexpr int Q = Shape<D>::Q;
  const uint4 r = dr.block(c0, K);
  uint32_t* d = x + Q * (lane & ~(Q - 1)) + (lane & (Q - 1));
  d[0] = r.x;
  d[Q] = r.y;
  if constexpr (Q == 4) {
    d[2 * Q] = r.z;
    d[3 * Q] = r.w;
  }
}
template <int D>
__device__ __forceinline__ void load_draws(const uint32_t* x, int lane, uint32_t (&u)[4]) {
  if constexpr (Shape<D>::Q == 4) {
    const uint4 v = *reinterpret_cast<const uint4*>(x + 4 * lane);
    u[0] = v.x; u[1] = v.y; u[2] = v.z; u[3] = v.w;
  } else {
    const uint2 v = *reinterpret_cast<const uint2*>(x + 2 * lane);
    u[0] = v.x; u[1] = v.y;
  }
}
// Counter word of lane k's block in batch bt of colour C (columns from first).
template <int D>
__device__ __forceinline__ uint32_t batch_counter(uint32_t C, uint32_t first, uint32_t bt, int k) {
  constexpr int Q = Shape<D>::Q;
  return (C << 16) | ((first + bt * Q + (uint32_t)(k & (Q - 1))) << 8) | (uint32_t)(k >> 2);
}

// One colour phase; returns the lane's energy change.  tbl: this sweep's
// table (shared address).  kStaged: x holds the phase's draws.  kVote: each
// batch of columns draws into x (two areas, taken in turn) when a vote finds a
// lane that needs it.  kFrozen: no threshold is above zero, nothing is drawn.
enum Draws { kVote, kStaged, kFrozen };
template <int D, int C, Draws MODE>
__device__ __forceinline__ int32_t phase(uint32_t (&P)[Shape<D>::NW], uint32_t tbl, const LaneColour& lc,
                                         const core::SaDraws& dr, const PhiloxKeys& K, uint32_t* x, int lane,
                                         uint32_t* err) {
  using Col = Columns<D, C>;
  constexpr int Q = Shape<D>::Q;
  auto entry = [&](auto ic) {
    constexpr int B = column_of<C>(decltype(ic)::value);
    uint32_t base = lc.base, mask = lc.mask;
    if constexpr (B < 0 || B == D - 1) {
      base = mask ? (B < 0 ? kLeft : kRight) : kIdle;
      mask &= 0x78u;
    }
    return table_entry((face_bits<D, B>(P) & mask) | (base | tbl), tbl, err);
  };
  int32_t dsum = 0;
  auto move = [&](auto ic, const uint2& e, uint32_t u) {
    const int32_t dE = (int32_t)e.x;
    if ((dE <= 0) | (u < e.y)) {
      dsum += dE;
      face_flip<D, column_of<C>(decltype(ic)::value)>(P, lc.rows);
    }
  };
  if constexpr (MODE == kFrozen) {
    int32_t dE[Col::n];
    for_columns<0, Col::n>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      dE[i] = (int32_t)entry(std::integral_constant<int, Col::first + i>{}).x;
    });
    for_columns<0, Col::n>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      if (dE[i] <= 0) {
        dsum += dE[i];
        face_flip<D, column_of<C>(Col::first + i)>(P, lc.rows);
      }
    });
  } else if constexpr (MODE == kStaged) {
    uint2 e[Col::n];
    uint32_t u[Col::batches][4];
    for_columns<0, Col::n>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      e[i] = entry(std::integral_constant<int, Col::first + i>{});
    });
#pragma unroll
    for (int bt = 0; bt < Col::batches; ++bt) load_draws<D>(x + bt * kBatchWords, lane, u[bt]);
    for_columns<0, Col::n>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      move(std::integral_constant<int, Col::first + i>{}, e[i], u[i / Q][i % Q]);
    });
  } else {
    for_columns<0, Col::batches>([&](auto bc) {
      constexpr int BT = decltype(bc)::value;
      constexpr int N = Col::n - BT * Q < Q ? Col::n - BT * Q : Q;
      uint2 e[Q];
      uint32_t u[4] = {0u, 0u, 0u, 0u}, need = 0;
      for_columns<0, N>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        e[i] = entry(std::integral_constant<int, Col::first + BT * Q + i>{});
        need |= e[i].y;
      });
      if (__any_sync(0xFFFFFFFFu, need != 0u)) {
        uint32_t* xb = x + (BT & 1) * kBatchWords;
        __syncwarp();
        draw_batch<D>(batch_counter<D>(C, Col::first, BT, lane & (Shape<D>::G - 1)), dr, K, xb, lane);
        __syncwarp();
        load_draws<D>(xb, lane, u);
      }
      for_columns<0, N>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        move(std::integral_constant<int, Col::first + BT * Q + i>{}, e[i], u[i]);
      });
    });
  }
  return dsum;
}

// Layout changes of a lane's word: row 2k-1 comes from lane k-1 (m_up: the
// first-row slots, none in the group's first lane), row 2k+1 from lane k+1
// (m_dn: the second-row slots, none in its last lane).
template <int NW>
__device__ __forceinline__ void to_odd(uint32_t (&P)[NW], uint32_t m_up) {
#pragma unroll
  for (int j = 0; j < NW; ++j) {
    const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, P[j], 1);
    P[j] = ((up >> 2) & m_up) | ((P[j] << 2) & 0xCCCCCCCCu);
  }
}
template <int NW>
__device__ __forceinline__ void to_even(uint32_t (&P)[NW], uint32_t m_dn) {
#pragma unroll
  for (int j = 0; j < NW; ++j) {
    const uint32_t dn = __shfl_down_sync(0xFFFFFFFFu, P[j], 1);
    P[j] = ((P[j] >> 2) & 0x33333333u) | ((dn << 2) & m_dn);
  }
}
template <int NW>
__device__ __forceinline__ void copy_words(const uint32_t (&a)[NW], uint32_t (&b)[NW]) {
#pragma unroll
  for (int j = 0; j < NW; ++j) b[j] = a[j];
}

template <int G>
__device__ __forceinline__ int32_t group_sum(int32_t v) {
#pragma unroll
  for (int off = G / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
  return v;
}

__device__ __forceinline__ void copy_async_u32(uint32_t dst, const uint32_t* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// What a producing warp does for one set of sweeps [t0, t0 + ns): the draws of
// every sweeping warp and the thresholds of the tables.
template <int D, int NC, int NP>
__device__ __forceinline__ void produce(int t0, int ns, const core::SaDraws (&base)[NC], const core::SweepTables& tab,
                                        const PhiloxKeys& K, uint32_t tables, const uint32_t* upd, int n_upd,
                                        uint32_t* draws, int pw, int lane) {
  using S = Shape<D>;
  const int k = lane & (S::G - 1);
  constexpr int kSweeps = Form<D, NC, NP>::kSweeps;
  for (int j = pw * 32 + lane; j < n_upd; j += NP * 32) {
    const uint32_t v = upd[j], a = tables + 8u * (v >> 16) + 4u;
    const uint32_t* T = tab.T + (size_t)t0 * tab.n_classes + (v & 0xFFFFu);
    uint32_t A[kSweeps];
#pragma unroll
    for (int s = 0; s < kSweeps; ++s) A[s] = s < ns ? __ldg(&T[(size_t)s * tab.n_classes]) : 0u;
#pragma unroll
    for (int s = 0; s < kSweeps; ++s) core::sts_u32(a + (uint32_t)s * kTable, A[s]);
  }
#pragma unroll
  for (int w = 0; w < NC; ++w) {
    core::SaDraws dr = base[w];
    for (int s = 0; s < ns; ++s) {
      dr.sweep((uint32_t)(t0 + s), K);
      uint32_t* x = draws + (s * NC + w) * S::kBatches * kBatchWords;
      // phases hold kB0, kB1, kB1, kB0 batches
#pragma unroll 2
      for (int j = (pw + s) % NP; j < S::kBatches; j += NP) {
        const int C = j < S::kB0 ? 0 : j < S::kB0 + S::kB1 ? 1 : j < S::kB0 + 2 * S::kB1 ? 2 : 3;
        const int j0 = C == 0 ? 0 : C == 1 ? S::kB0 : C == 2 ? S::kB0 + S::kB1 : S::kB0 + 2 * S::kB1;
        draw_batch<D>(batch_counter<D>((uint32_t)C, C == 3 ? 1u : 0u, (uint32_t)(j - j0), k), dr, K,
                      x + j * kBatchWords, lane);
      }
    }
  }
}

// Anneal the n_chains (1 to kCtaChains) chains of a segment from chain first by
// one CTA.  chain0, init0 and out0 are those of the segment's chain 0; groups
// past n_chains run a copy of the last chain and write nothing.  smem: Form::smem_bytes(tab.n_classes) bytes.
template <int D, int NC, int NP>
__device__ __forceinline__ void anneal_coop_cta(const uint32_t* __restrict__ init0, uint64_t chain0, int64_t first,
                                                int n_chains, const core::ChainOut& out0, const core::SweepTables& tab,
                                                const PhiloxKeys& K, uint8_t* smem) {
  using S = Shape<D>;
  using F = Form<D, NC, NP>;
  constexpr int G = S::G, NW = S::NW, W = S::kW, kSweeps = F::kSweeps;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = lane & (G - 1);
  const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t pad = ((s0 + kTable - 1u) & ~(kTable - 1u)) - s0, tables = s0 + pad;
  uint32_t* draws = reinterpret_cast<uint32_t*>(smem + pad + F::kSets * kSweeps * kTable);
  uint32_t* upd = draws + F::kDrawWords;                                   // [kEntries]
  int* n_upd_s = reinterpret_cast<int*>(upd + kEntries);                   // [4]
  uint32_t* stage_all = reinterpret_cast<uint32_t*>(n_upd_s + 4);
  uint32_t* stage = stage_all + (tid / G) * 2 * W;                         // sweeping warps only
  uint32_t* raw = stage_all + F::kCtaChains * 2 * W;                       // NP = 0: [kSweeps][n_classes]
  const uint32_t raw_s = (uint32_t)__cvta_generic_to_shared(raw);
  const int n_sweeps = tab.n_sweeps, ncls = tab.n_classes, n_live = min(tab.n_live, n_sweeps);

  // The energy changes are the same in every sweep; the thresholds (zero
  // where no draw can accept) follow per set of sweeps.
  if (tid == 0) n_upd_s[0] = 0;
  __syncthreads();
  for (int e = tid; e < kEntries; e += F::kThreads) {
    const int src = sig_source(e);
    const int2 sg = src >= 0 ? __ldg(&tab.sig[src]) : make_int2(1, -1);
#pragma unroll
    for (int s = 0; s < F::kSets * kSweeps; ++s)
      core::sts_u2(tables + (uint32_t)s * kTable + 8u * (uint32_t)e, make_uint2((uint32_t)sg.x, 0u));
    if (sg.y >= 0) upd[atomicAdd(n_upd_s, 1)] = ((uint32_t)e << 16) | (uint32_t)sg.y;
  }
  __syncthreads();
  const int n_upd = n_upd_s[0];

  if constexpr (NP > 0) if (warp >= NC) {  // a producing warp: one set ahead of the sweeping ones
    core::SaDraws base[NC];
#pragma unroll
    for (int w = 0; w < NC; ++w) {
      const uint64_t ch = chain0 + (uint64_t)(first + min(w * S::kChains + lane / G, n_chains - 1));
      base[w].init((uint32_t)ch, kTagSA | ((uint32_t)(ch >> 32) << 8), K);
    }
    for (int t0 = 0, set = 0; t0 < n_live; t0 += kSweeps, set ^= 1) {
      produce<D, NC, NP>(t0, min(kSweeps, n_live - t0), base, tab, K, tables + (uint32_t)(set * kSweeps) * kTable, upd,
                          n_upd, draws + set * (F::kDrawWords / 2), warp - NC, lane);
      __syncthreads();
    }
    if (n_live > 0) __syncthreads();
    return;
  }
  auto fetch = [&](int t0) {  // thresholds of sweeps [t0, t0 + kSweeps) into raw, asynchronously
    const int n = min(kSweeps, n_live - t0) * ncls;
    for (int j = tid; j < n; j += F::kThreads) copy_async_u32(raw_s + 4u * (uint32_t)j, tab.T + (size_t)t0 * ncls + j);
  };
  if (NP == 0 && n_live > 0) fetch(0);

  const bool active = tid / G < n_chains;
  const int64_t ci = first + (active ? tid / G : n_chains - 1);
  const uint64_t chain = chain0 + (uint64_t)ci;
  const int P_coset = (int)(ci & 3);
  const uint32_t* init = init0 + (size_t)(ci >> 2) * 2 * W;
  core::ChainOut out;
  out.best_E = out0.best_E + ci;
  out.best_cfg = out0.best_cfg ? out0.best_cfg + (size_t)ci * 2 * W : nullptr;
  out.final_E = out0.final_E ? out0.final_E + ci : nullptr;
  out.final_cfg = out0.final_cfg ? out0.final_cfg + (size_t)ci * 2 * W : nullptr;

  // Rows 2k and 2k+1 of R_i L_P as an even-layout pair word.
  uint32_t P[NW];
  int32_t e_lane = 0;
  {
    uint64_t row[2] = {0ull, 0ull};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = 2 * k + h;
      if (r < D) {
        const uint32_t x = core::plane_field(init, W, r * D, D), z = core::plane_field(init + W, W, r * D, D);
        uint64_t v = core::spread2(z) | (core::spread2(x) << 1);
        if (P_coset == 1 || P_coset == 2) v ^= h ? 1ull : 2ull;
        if ((P_coset == 2 || P_coset == 3) && r == 0)
          v ^= 0x9999999999999999ull & ((2 * D >= 64) ? ~0ull : ((1ull << (2 * D)) - 1ull));
        const uint64_t zz = v & 0x5555555555555555ull, xx = (v >> 1) & 0x5555555555555555ull;
        e_lane += __popcll(xx & ~zz) * tab.W[2] + __popcll(xx & zz) * tab.W[3] + __popcll(zz & ~xx) * tab.W[1];
        row[h] = v;
      }
    }
    const uint64_t lo = core::spread_pairs((uint32_t)row[0]) | (core::spread_pairs((uint32_t)row[1]) << 2);
    const uint64_t hi =
        core::spread_pairs((uint32_t)(row[0] >> 32)) | (core::spread_pairs((uint32_t)(row[1] >> 32)) << 2);
#pragma unroll
    for (int j = 0; j < NW; ++j) P[j] = (uint32_t)((j < 2 ? lo : hi) >> (32 * (j & 1)));
  }
  const LaneColour c0 = lane_colour<D, 0>(k), c1 = lane_colour<D, 1>(k), c2 = lane_colour<D, 2>(k),
                   c3 = lane_colour<D, 3>(k);
  const uint32_t m_up = k == 0 ? 0u : 0x33333333u, m_dn = k == G - 1 ? 0u : 0xCCCCCCCCu;
  core::SaDraws dr;
  dr.init((uint32_t)chain, kTagSA | ((uint32_t)(chain >> 32) << 8), K);
  int32_t E_best = group_sum<G>(e_lane);
  uint32_t best[NW];
#pragma unroll
  for (int j = 0; j < NW; ++j) best[j] = P[j];

  // One sweep; x: its draws (kStaged) or the warp's two areas (kVote).
  auto sweep = [&](auto mode, uint32_t tbl, uint32_t* x) {
    constexpr Draws M = decltype(mode)::value;
    // The words after colours 0, 1 and 2 (even layout), for the minimum.
    uint32_t P0[NW], P1[NW], P2[NW];
    const int32_t d0 = phase<D, 0, M>(P, tbl, c0, dr, K, x, lane, tab.err);
    copy_words(P, P0);
    to_odd(P, m_up);
    const int32_t d1 = phase<D, 1, M>(P, tbl, c1, dr, K, M == kStaged ? x + S::kB0 * kBatchWords : x, lane, tab.err);
    to_even(P, m_dn);
    copy_words(P, P1);
    const int32_t d2 =
        phase<D, 2, M>(P, tbl, c2, dr, K, M == kStaged ? x + (S::kB0 + S::kB1) * kBatchWords : x, lane, tab.err);
    copy_words(P, P2);
    to_odd(P, m_up);
    const int32_t d3 =
        phase<D, 3, M>(P, tbl, c3, dr, K, M == kStaged ? x + (S::kB0 + 2 * S::kB1) * kBatchWords : x, lane, tab.err);
    to_even(P, m_dn);
    if (__any_sync(0xFFFFFFFFu, (d0 < 0) | (d1 < 0) | (d2 < 0) | (d3 < 0))) {
      const int32_t e0 = e_lane + d0, e1 = e0 + d1, e2 = e1 + d2, e3 = e2 + d3;
      const int32_t E0 = group_sum<G>(e0), E1 = group_sum<G>(e1), E2 = group_sum<G>(e2), E3 = group_sum<G>(e3);
      if (min(min(E0, E1), min(E2, E3)) < E_best) {  // the earliest phase with the lowest energy
        if (E0 < E_best) E_best = E0, copy_words(P0, best);
        if (E1 < E_best) E_best = E1, copy_words(P1, best);
        if (E2 < E_best) E_best = E2, copy_words(P2, best);
        if (E3 < E_best) E_best = E3, copy_words(P, best);
      }
    }
    e_lane += d0 + d1 + d2 + d3;
  };

  for (int t0 = 0, set = 0; t0 < n_live; t0 += kSweeps, set ^= (F::kSets - 1)) {
    const int ns = min(kSweeps, n_live - t0);
    if constexpr (NP == 0) {
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();  // the fetched thresholds are in, and every warp is done with the tables
      for (int j = tid; j < n_upd; j += F::kThreads) {
        const uint32_t v = upd[j], a = tables + 8u * (v >> 16) + 4u;
        const uint32_t* r = raw + (v & 0xFFFFu);
#pragma unroll
        for (int s = 0; s < kSweeps; ++s)
          if (s < ns) core::sts_u32(a + (uint32_t)s * kTable, r[s * ncls]);
      }
    }
    __syncthreads();  // this set is ready (NP > 0: and the producing warps may refill the other one)
    if (NP == 0 && t0 + kSweeps < n_live) fetch(t0 + kSweeps);
    for (int s = 0; s < ns; ++s) {
      const uint32_t tbl = tables + (uint32_t)(set * kSweeps + s) * kTable;
      if (NP == 0) dr.sweep((uint32_t)(t0 + s), K);
      uint32_t* x = NP ? draws + set * (F::kDrawWords / 2) + (s * NC + warp) * S::kBatches * kBatchWords
                       : draws + warp * 2 * kBatchWords;
      sweep(std::integral_constant<Draws, NP ? kStaged : kVote>{}, tbl, x);
    }
  }
  if (NP > 0 && n_live > 0) __syncthreads();  // pairs with the producing warps' last
  // The frozen sweeps (see anneal_core.cuh).
  uint32_t saved[NW];
  const bool may_stop = !out.final_E && !out.final_cfg;
  bool done = false;
  for (int t = n_live, i = 0; t < n_sweeps; ++t, ++i) {
    if ((i & (i + 1)) == 0) copy_words(P, saved);
    sweep(std::integral_constant<Draws, kFrozen>{}, tables, nullptr);
    if (may_stop) {
      uint32_t diff = 0;
#pragma unroll
      for (int j = 0; j < NW; ++j) diff |= P[j] ^ saved[j];
      const uint32_t same = __ballot_sync(0xFFFFFFFFu, diff == 0u) >> (lane & ~(G - 1));
      done |= (same & ((1u << G) - 1u)) == (1u << G) - 1u;
      if (__all_sync(0xFFFFFFFFu, done)) break;
    }
  }

  const int32_t E_final = group_sum<G>(e_lane);
  if (active && k == 0) {
    *out.best_E = E_best;
    if (out.final_E) *out.final_E = E_final;
  }
  // Pair words -> planar words: each lane places its two rows' bits.
  auto emit = [&](const uint32_t (&w)[NW], uint32_t* dst) {
    for (int i = k; i < 2 * W; i += G) stage[i] = 0u;
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = 2 * k + h;
      if (r < D) {
        const uint64_t lo = (uint64_t)w[0] | (NW > 1 ? (uint64_t)w[NW > 1 ? 1 : 0] << 32 : 0ull);
        const uint64_t hi = (NW > 2 ? (uint64_t)w[NW > 2 ? 2 : 0] : 0ull) |
                            (NW > 3 ? (uint64_t)w[NW > 3 ? 3 : 0] << 32 : 0ull);
        const uint64_t v = (uint64_t)core::gather_pairs(lo >> (2 * h)) | ((uint64_t)core::gather_pairs(hi >> (2 * h)) << 32);
        const uint64_t fz = core::gather2(v), fx = core::gather2(v >> 1);
        const int start = r * D, wi = start >> 5, off = start & 31;
        atomicOr(&stage[W + wi], (uint32_t)(fz << off));
        atomicOr(&stage[wi], (uint32_t)(fx << off));
        if (wi + 1 < W && off + D > 32) {
          atomicOr(&stage[W + wi + 1], (uint32_t)(fz >> (32 - off)));
          atomicOr(&stage[wi + 1], (uint32_t)(fx >> (32 - off)));
        }
      }
    }
    __syncwarp();
    if (active)
      for (int i = k; i < 2 * W; i += G) dst[i] = stage[i];
    __syncwarp();
  };
  if (out.final_cfg) emit(P, out.final_cfg);
  if (out.best_cfg) emit(best, out.best_cfg);
}

}  // namespace coop
}  // namespace xzzx
