// Lane-parallel annealing (the colour sweep of Alg. 2 / Alg. 3 with several
// lanes per chain), for launches whose chains do not fill the GPU one per
// thread, and for planar codes past the register-resident kernel.
//
// State.  Lane k of a chain's group of G lanes (a power of two) holds a pair of
// lattice rows: the geometries below (RotLanes, PlanarLanes) say how.  Every
// face of a colour has its draw coordinate's row part equal to its lane's k, and
// a lane takes its rows' faces column by column with compile-time shifts.
//
// Draws.  The block of a column serves the four rows of a quad of lanes, so the
// quad computes four columns' blocks at once, one per lane, and trades words
// through shared memory.
//
// Acceptance table.  One table of (dE, A) per sweep for the whole CTA, for
// several sweeps at a time, instead of one per warp rebuilt every sweep.
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

constexpr int kBatchWords = 128;  // one batch of a warp's draws

// Compile-time loop over n indices from I.
template <int I, int N, typename F>
__device__ __forceinline__ void for_each(F&& f) {
  if constexpr (N > 0) {
    f(std::integral_constant<int, I>{});
    for_each<I + 1, N - 1>(f);
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
// Sets len bits of plane p from bit start to the low bits of v.
__device__ __forceinline__ void place_bits(uint32_t* p, int start, int len, uint32_t v) {
  const int wi = start >> 5, off = start & 31;
  atomicOr(&p[wi], v << off);
  if (off + len > 32) atomicOr(&p[wi + 1], v >> (32 - off));
}
__device__ __forceinline__ int32_t row_energy(uint64_t v, const int32_t (&W)[4]) {
  const uint64_t z = v & 0x5555555555555555ull, x = (v >> 1) & 0x5555555555555555ull;
  return __popcll(x & ~z) * W[2] + __popcll(x & z) * W[3] + __popcll(z & ~x) * W[1];
}

// ---------------------------------------------------------------------------
// Draws.
// ---------------------------------------------------------------------------

// What a geometry fixes for the draws: lanes per chain, columns drawn at once
// (a quad's, or a pair's when G = 2), and the batches of each colour's phase.
template <int G_, int N0, int N1, int N2, int N3, int FIRST3>
struct LaneShape {
  static constexpr int G = G_, kChains = 32 / G;
  static constexpr int Q = G < 4 ? G : 4;
  // Columns of colour C and the first one's draw coordinate.
  __host__ __device__ static constexpr int cols(int C) { return C == 0 ? N0 : C == 1 ? N1 : C == 2 ? N2 : N3; }
  __host__ __device__ static constexpr int first(int C) { return C == 3 ? FIRST3 : 0; }
  __host__ __device__ static constexpr int batches(int C) { return (cols(C) + Q - 1) / Q; }
  __host__ __device__ static constexpr int start(int C) {
    int b = 0;
    for (int c = 0; c < C; ++c) b += batches(c);
    return b;
  }
  static constexpr int kBatches = (N0 + Q - 1) / Q + (N1 + Q - 1) / Q + (N2 + Q - 1) / Q + (N3 + Q - 1) / Q;
};

// One batch of draws for the lanes of a warp: each lane computes one column's
// block of its chain and hands the quad's four lanes (G = 2: the pair) their
// words, so that lane l finds the draws of the batch's columns at x[Q l], x[Q l +
// 1], ...  c0: the block's counter word.
template <int Q>
__device__ __forceinline__ void draw_batch(uint32_t c0, const core::SaDraws& dr, const PhiloxKeys& K, uint32_t* x,
                                           int lane) {
  const uint4 r = dr.block(c0, K);
  uint32_t* d = x + Q * (lane & ~(Q - 1)) + (lane & (Q - 1));
  d[0] = r.x;
  d[Q] = r.y;
  if constexpr (Q == 4) {
    d[2 * Q] = r.z;
    d[3 * Q] = r.w;
  }
}
template <int Q>
__device__ __forceinline__ void load_draws(const uint32_t* x, int lane, uint32_t (&u)[4]) {
  if constexpr (Q == 4) {
    const uint4 v = *reinterpret_cast<const uint4*>(x + 4 * lane);
    u[0] = v.x; u[1] = v.y; u[2] = v.z; u[3] = v.w;
  } else {
    const uint2 v = *reinterpret_cast<const uint2*>(x + 2 * lane);
    u[0] = v.x; u[1] = v.y;
  }
}
// Counter word of lane k's block in batch bt of colour C (columns from first).
template <class S>
__device__ __forceinline__ uint32_t batch_counter(uint32_t C, uint32_t first, uint32_t bt, int k) {
  return (C << 16) | ((first + bt * S::Q + (uint32_t)(k & (S::Q - 1))) << 8) | (uint32_t)(k >> 2);
}

// How a phase gets its draws.  kStaged: they wait in x.  kVote: each batch of
// columns draws into x (two areas, taken in turn) when a vote finds a lane that
// needs it.  kFrozen: no threshold is above zero, nothing is drawn.
enum Draws { kVote, kStaged, kFrozen };

// The faces of one colour phase.  entry(i) loads the table entry of the lane's
// face in column i; move(i, dE) takes the move.
template <class S, int C, Draws MODE, typename Entry, typename Move>
__device__ __forceinline__ void faces(const core::SaDraws& dr, const PhiloxKeys& K, uint32_t* x, int lane,
                                      Entry&& entry, Move&& move) {
  constexpr int N = S::cols(C), Q = S::Q, NB = S::batches(C);
  if constexpr (MODE == kFrozen) {
    int32_t dE[N];
    for_each<0, N>([&](auto ic) { dE[ic] = (int32_t)entry(ic).x; });
    for_each<0, N>([&](auto ic) {
      if (dE[ic] <= 0) move(ic, dE[ic]);
    });
  } else if constexpr (MODE == kStaged) {
    uint2 e[N];
    uint32_t u[NB][4];
    for_each<0, N>([&](auto ic) { e[ic] = entry(ic); });
#pragma unroll
    for (int bt = 0; bt < NB; ++bt) load_draws<Q>(x + bt * kBatchWords, lane, u[bt]);
    for_each<0, N>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      if (((int32_t)e[i].x <= 0) | (u[i / Q][i % Q] < e[i].y)) move(ic, (int32_t)e[i].x);
    });
  } else {
    for_each<0, NB>([&](auto bc) {
      constexpr int BT = decltype(bc)::value, I0 = BT * Q, n = N - I0 < Q ? N - I0 : Q;
      uint2 e[Q];
      uint32_t u[4] = {0u, 0u, 0u, 0u}, need = 0;
      for_each<0, n>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        e[i] = entry(std::integral_constant<int, I0 + i>{});
        need |= e[i].y;
      });
      if (__any_sync(0xFFFFFFFFu, need != 0u)) {
        uint32_t* xb = x + (BT & 1) * kBatchWords;
        __syncwarp();
        draw_batch<Q>(batch_counter<S>(C, S::first(C), BT, lane & (S::G - 1)), dr, K, xb, lane);
        __syncwarp();
        load_draws<Q>(xb, lane, u);
      }
      for_each<0, n>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        if (((int32_t)e[i].x <= 0) | (u[i] < e[i].y)) move(std::integral_constant<int, I0 + i>{}, (int32_t)e[i].x);
      });
    });
  }
}

// Table entry at shared address a of a table of the given bytes at tbl.
__device__ __forceinline__ uint2 table_entry(uint32_t a, uint32_t tbl, uint32_t bytes, uint32_t* err) {
  return XZZX_CHECK(err, a - tbl <= bytes - 8u && !injected(err, XZZX_DEVERR_BOUNDS)) ? core::lds_u2(a)
                                                                                      : make_uint2(0u, 0u);
}

// ---------------------------------------------------------------------------
// Rotated lattice.  Lane k holds one pair word of the layout of
// anneal_core.cuh: rows 2k and 2k+1 (even layout, colours 0 and 2) or rows 2k-1
// and 2k (odd layout, colours 1 and 3), four bits per column in one to four
// registers, so that a face lies inside its lane's word and a layout change is
// one shuffle per register.
//
// Table order: 256 bulk signatures (TL | BL << 2 | TR << 4 | BR << 6); then 256
// "edge" ones: a top face keeps its byte's bits 2-3 and 6-7, a bottom face bits
// 0-1 and 4-5 (both give the all-identity entry at 0); the left and right
// boundary nibbles and the entry of idle lanes (never accepted) fill index
// ranges that neither can reach.
// ---------------------------------------------------------------------------
template <int D>
struct RotLanes : LaneShape<(D + 1) / 2 <= 2 ? 2 : (D + 1) / 2 <= 4 ? 4 : (D + 1) / 2 <= 8 ? 8 : 16, (D - 1) / 2,
                            (D + 1) / 2, (D + 1) / 2, (D - 1) / 2, 1> {
  using S = LaneShape<(D + 1) / 2 <= 2 ? 2 : (D + 1) / 2 <= 4 ? 4 : (D + 1) / 2 <= 8 ? 8 : 16, (D - 1) / 2, (D + 1) / 2,
                      (D + 1) / 2, (D - 1) / 2, 1>;
  static constexpr int H = (D + 1) / 2;
  static constexpr int NW = (4 * D + 31) / 32;
  static constexpr int kW = (D * D + 31) / 32;
  static constexpr int kEntries = 512;
  static constexpr uint32_t kTable = kEntries * 8u;
  static constexpr uint32_t kEdgeAt = 256u * 8u, kLeftAt = (256u + 0x50u) * 8u, kRightAt = (256u + 0x90u) * 8u,
                            kIdleAt = (256u + 0x60u) * 8u;

  // Entry of the schedule's signature table for table index p, -1 for the
  // entry of idle lanes and unreachable indices.
  __device__ static int sig_source(int p) {
    if (p < 256) return core::pair_sig_source(p);
    const int e = p - 256;
    if ((e & 0x33) == 0) return sig_base(kTop) + (((e >> 2) & 3) | (((e >> 6) & 3) << 2));
    if ((e & 0xCC) == 0) return sig_base(kBottom) + ((e & 3) | (((e >> 4) & 3) << 2));
    if ((e & 0xF0) == 0x50) return sig_base(kLeft) + (e & 15);
    if ((e & 0xF0) == 0x90) return sig_base(kRight) + (e & 15);
    return -1;
  }

  uint32_t w[NW];  // the pair word, even layout between phases

  // Constants of a lane: per colour, the byte mask and table offset of its
  // faces (idle lanes: the entry that is never accepted) and the rows a move
  // changes; the slots a layout change brings in.
  struct Lane {
    uint32_t mask[4], base[4], rows[4], m_up, m_dn;
    __device__ explicit Lane(int k) {
#pragma unroll
      for (int C = 0; C < 4; ++C) {
        const bool on = k < H && !(C == 1 && k == 0) && !(C == 2 && k == H - 1);
        const bool top = C == 3 && k == 0, bottom = C == 0 && k == H - 1;
        mask[C] = !on ? 0u : top ? 0xCCu << 3 : bottom ? 0x33u << 3 : 0x7F8u;
        base[C] = !on ? kIdleAt : (top || bottom) ? kEdgeAt : 0u;
        rows[C] = top ? 0xCCCCCCCCu : bottom ? 0x33333333u : 0xFFFFFFFFu;
      }
      m_up = k == 0 ? 0u : 0x33333333u;         // row 2k-1 comes from lane k-1
      m_dn = k == S::G - 1 ? 0u : 0xCCCCCCCCu;  // row 2k+1 from lane k+1
    }
  };

  // Rows 2k and 2k+1 of R_i L_P (L_X: column 0, X on even rows, Z on odd ones;
  // L_Z: row 0, Z on even columns, X on odd ones).  Returns their energy.
  __device__ __forceinline__ int32_t load(const uint32_t* __restrict__ init, int P, int k, const int32_t (&W)[4]) {
    uint64_t row[2] = {0ull, 0ull};
    int32_t e = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = 2 * k + h;
      if (r < D) {
        uint64_t v = core::spread2(core::plane_field(init + kW, kW, r * D, D)) |
                     (core::spread2(core::plane_field(init, kW, r * D, D)) << 1);
        if (P == 1 || P == 2) v ^= h ? 1ull : 2ull;
        if ((P == 2 || P == 3) && r == 0) v ^= 0x9999999999999999ull & ((2 * D >= 64) ? ~0ull : ((1ull << (2 * D)) - 1ull));
        e += row_energy(v, W);
        row[h] = v;
      }
    }
    const uint64_t lo = core::spread_pairs((uint32_t)row[0]) | (core::spread_pairs((uint32_t)row[1]) << 2);
    const uint64_t hi =
        core::spread_pairs((uint32_t)(row[0] >> 32)) | (core::spread_pairs((uint32_t)(row[1] >> 32)) << 2);
#pragma unroll
    for (int j = 0; j < NW; ++j) w[j] = (uint32_t)((j < 2 ? lo : hi) >> (32 * (j & 1)));
    return e;
  }
  // The lane's rows of state v into the planes at stage (x then z).
  __device__ static void place(const uint32_t (&v)[NW], uint32_t* stage, int k) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = 2 * k + h;
      if (r < D) {
        const uint64_t lo = (uint64_t)v[0] | (NW > 1 ? (uint64_t)v[NW > 1 ? 1 : 0] << 32 : 0ull);
        const uint64_t hi = (NW > 2 ? (uint64_t)v[NW > 2 ? 2 : 0] : 0ull) |
                            (NW > 3 ? (uint64_t)v[NW > 3 ? 3 : 0] << 32 : 0ull);
        const uint64_t f = (uint64_t)core::gather_pairs(lo >> (2 * h)) | ((uint64_t)core::gather_pairs(hi >> (2 * h)) << 32);
        place_bits(stage, r * D, D, core::gather2(f >> 1));
        place_bits(stage + kW, r * D, D, core::gather2(f));
      }
    }
  }

  // Table byte offset of the face at column B (-1: the left boundary nibble,
  // d-1: the right one), before the lane's mask.
  template <int B>
  __device__ __forceinline__ uint32_t bits() const {
    if constexpr (B < 0) {
      return w[0] << 3;
    } else {
      constexpr int RG = (4 * B) >> 5, OFF = (4 * B) & 31;
      if constexpr (OFF == 0) return w[RG] << 3;
      else if constexpr (OFF == 28 && RG + 1 < NW) return __funnelshift_r(w[RG], w[RG + 1], 25);
      else return w[RG] >> (OFF - 3);
    }
  }
  template <int B>
  __device__ __forceinline__ void flip(uint32_t rows) {
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

  // One colour phase; returns the lane's energy change.
  template <int C, Draws MODE>
  __device__ __forceinline__ int32_t phase(const Lane& ln, uint32_t tbl, const core::SaDraws& dr, const PhiloxKeys& K,
                                           uint32_t* x, int lane, uint32_t* err) {
    if constexpr (C & 1) {
#pragma unroll
      for (int j = 0; j < NW; ++j) {
        const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, w[j], 1);
        w[j] = ((up >> 2) & ln.m_up) | ((w[j] << 2) & 0xCCCCCCCCu);
      }
    }
    int32_t dsum = 0;
    const uint32_t base = tbl + ln.base[C], base_side = tbl + (ln.mask[C] ? (C == 1 ? kRightAt : kLeftAt) : kIdleAt);
    faces<S, C, MODE>(
        dr, K, x, lane,
        [&](auto ic) {
          constexpr int ib = decltype(ic)::value + S::first(C), B = (C >> 1) == 0 ? 2 * ib : 2 * ib - 1;
          constexpr bool SIDE = B < 0 || B == D - 1;
          return table_entry((bits<B>() & (SIDE ? ln.mask[C] & 0x78u : ln.mask[C])) | (SIDE ? base_side : base), tbl,
                             kTable, err);
        },
        [&](auto ic, int32_t dE) {
          constexpr int ib = decltype(ic)::value + S::first(C), B = (C >> 1) == 0 ? 2 * ib : 2 * ib - 1;
          dsum += dE;
          flip<B>(ln.rows[C]);
        });
    if constexpr (C & 1) {
#pragma unroll
      for (int j = 0; j < NW; ++j) {
        const uint32_t dn = __shfl_down_sync(0xFFFFFFFFu, w[j], 1);
        w[j] = ((w[j] >> 2) & 0x33333333u) | ((dn << 2) & ln.m_dn);
      }
    }
    return dsum;
  }
};

// ---------------------------------------------------------------------------
// Planar lattice.  Lane k holds rows 2k (d qubits) and 2k+1 (d-1) of the grid,
// two bits per slot, one word each up to d = 15 and two above; it takes the faces
// of row 2k in colours 0 and 2 and of row 2k+1 in colours 1 and 3.  The faces of
// one lane and colour sit every second slot, the first at slot 0 or 1 (colours
// 0, 2) or -1 or 0 (colours 1, 3) in turn from lane to lane.  A phase shifts the
// centre row by that parity and packs the up and down slots of its faces
// beside each other into a second word, so that column t's four corners are the
// nibbles at bit 4t of two words, and writes the rows back after it: one
// shuffle to bring the neighbour's row in and one to hand its part back.
//
// Table order: 256 bulk signatures (left | right << 2 | up << 4 | down << 6);
// 256 of the top and bottom rows' faces (the missing corner's bits zero; both
// zero gives one entry); 256 of the left and right boundary's likewise.  Idle
// lanes use an entry none of them can reach.
// ---------------------------------------------------------------------------
template <int D>
struct PlanarLanes : LaneShape<D <= 4 ? 4 : D <= 8 ? 8 : D <= 16 ? 16 : 32, (D - 1) / 2, (D + 1) / 2, (D - 1) / 2,
                               (D + 1) / 2, 0> {
  using S = LaneShape<D <= 4 ? 4 : D <= 8 ? 8 : D <= 16 ? 16 : 32, (D - 1) / 2, (D + 1) / 2, (D - 1) / 2, (D + 1) / 2, 0>;
  using Row = typename std::conditional<(D > 15), uint64_t, uint32_t>::type;
  static constexpr int NS = (D - 1) / 2;
  static constexpr bool kByThree = D == 13 || D == 15;  // see sweeping_per_sm
  static constexpr int NR = sizeof(Row) / 4, NW = 2 * NR;
  static constexpr int kNQ = D * D + (D - 1) * (D - 1);
  static constexpr int kW = (kNQ + 31) / 32;
  static constexpr int kEntries = 768;
  static constexpr uint32_t kTable = kEntries * 8u;
  static constexpr uint32_t kEdgeAt = 256u * 8u, kSideAt = 512u * 8u, kIdleAt = (256u + 0x50u) * 8u;
  static constexpr Row M3 = (Row)0x3333333333333333ull;

  __device__ static int sig_source(int p) {
    const int e = p & 255, l = e & 3, r = (e >> 2) & 3, u = (e >> 4) & 3, d = e >> 6;
    if (p < 256) return planar_sig_base(kPBulk) + e;
    if (p < 512) {
      if (u == 0) return planar_sig_base(kPNoUp) + (l | (r << 2) | (d << 4));
      if (d == 0) return planar_sig_base(kPNoDown) + (l | (r << 2) | (u << 4));
      return -1;
    }
    if (l == 0) return planar_sig_base(kPNoLeft) + (r | (u << 2) | (d << 4));
    if (r == 0) return planar_sig_base(kPNoRight) + (l | (u << 2) | (d << 4));
    return -1;
  }

  uint32_t w[NW];  // row 2k, row 2k+1

  __device__ static Row row_of(const uint32_t (&v)[NW], int h) {
    if constexpr (NR == 1) return v[h];
    else return (uint64_t)v[2 * h] | ((uint64_t)v[2 * h + 1] << 32);
  }
  __device__ __forceinline__ void set_row(int h, Row v) {
    w[NR * h] = (uint32_t)v;
    if constexpr (NR == 2) w[2 * h + 1] = (uint32_t)(v >> 32);
  }
  // The same row of lane - 1 or lane + 1 (the warp's end lanes: their own).
  __device__ static Row shift_lane(Row v, bool up) {
    uint32_t lo = (uint32_t)v;
    lo = up ? __shfl_up_sync(0xFFFFFFFFu, lo, 1) : __shfl_down_sync(0xFFFFFFFFu, lo, 1);
    if constexpr (NR == 1) {
      return lo;
    } else {
      uint32_t hi = (uint32_t)(v >> 32);
      hi = up ? __shfl_up_sync(0xFFFFFFFFu, hi, 1) : __shfl_down_sync(0xFFFFFFFFu, hi, 1);
      return (uint64_t)lo | ((uint64_t)hi << 32);
    }
  }

  struct Lane {
    bool even_on, odd_on, edge;
    bool first;      // lane 0: no row above
    int par;         // k & 1
    Row odd_mask;    // slots of row 2k+1
    __device__ explicit Lane(int k)
        : even_on(k < D), odd_on(k < D - 1), edge(k == 0 || k == D - 1), first(k == 0), par(k & 1),
          odd_mask(k < D - 1 ? (Row)((1ull << (2 * (D - 1))) - 1ull) : (Row)0) {}
  };

  __device__ static int row_start(int r) { return (r >> 1) * (2 * D - 1) + ((r & 1) ? D : 0); }

  // Rows 2k and 2k+1 of R_i L_P (L_X: X on slot 0 of the even rows; L_Z: Z on
  // row 0).  Returns their energy.
  __device__ __forceinline__ int32_t load(const uint32_t* __restrict__ init, int P, int k, const int32_t (&W)[4]) {
    int32_t e = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = 2 * k + h, len = h ? D - 1 : D;
      uint64_t v = 0;
      if (r < 2 * D - 1) {
        v = core::spread2(core::plane_field(init + kW, kW, row_start(r), len)) |
            (core::spread2(core::plane_field(init, kW, row_start(r), len)) << 1);
        if ((P == 1 || P == 2) && h == 0) v ^= 2ull;
        if ((P == 2 || P == 3) && r == 0) v ^= 0x5555555555555555ull & ((1ull << (2 * D)) - 1ull);
        e += row_energy(v, W);
      }
      set_row(h, (Row)v);
    }
    return e;
  }
  __device__ static void place(const uint32_t (&v)[NW], uint32_t* stage, int k) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = 2 * k + h, len = h ? D - 1 : D;
      if (r < 2 * D - 1) {
        const uint64_t f = row_of(v, h);
        place_bits(stage, row_start(r), len, core::gather2(f >> 1));
        place_bits(stage + kW, row_start(r), len, core::gather2(f));
      }
    }
  }

  // The nibble at bit 4t of v, moved to bits [AT, AT + 4) (others undefined).
  template <int T, int AT>
  __device__ static uint32_t nibble(Row v) {
    const uint32_t x = T < 8 ? (uint32_t)v : (uint32_t)((uint64_t)v >> 32);
    constexpr int B = (4 * T) & 31;
    if constexpr (B >= AT) return x >> (B - AT);
    else return x << (AT - B);
  }

  template <int C, Draws MODE>
  __device__ __forceinline__ int32_t phase(const Lane& ln, uint32_t tbl, const core::SaDraws& dr, const PhiloxKeys& K,
                                           uint32_t* x, int lane, uint32_t* err) {
    const Row even = row_of(w, 0), odd = row_of(w, 1);
    Row A, U;
    int32_t dsum = 0;
    auto corners = [&](auto ic, uint32_t base, uint32_t mask) {
      constexpr int t = decltype(ic)::value;
      return table_entry((nibble<t, 3>(A) & 0x78u & mask) | ((nibble<t, 7>(U) & 0x780u & mask) | base), tbl, kTable, err);
    };
    auto move = [&](auto ic, int32_t dE) {  // X on left and right, Z on up and down
      constexpr int t = decltype(ic)::value;
      dsum += dE;
      A ^= (Row)0xAu << (4 * t);
      U ^= (Row)0x5u << (4 * t);
    };
    if constexpr ((C & 1) == 0) {
      const int p = 2 * (((C >> 1) + ln.par) & 1);  // 2 kl0
      const Row above = shift_lane(odd, true);
      A = even >> p;
      U = ((ln.first ? (Row)0 : above >> p) & M3) | (((odd >> p) & M3) << 2);
      const uint32_t base = tbl + (!ln.even_on ? kIdleAt : ln.edge ? kEdgeAt : 0u), mask = ln.even_on ? ~0u : 0u;
      const uint32_t mU = ln.edge ? (ln.first ? 0x600u : 0x180u) : ~0u;  // the corner that exists
      faces<S, C, MODE>(
          dr, K, x, lane,
          [&](auto ic) {
            constexpr int t = decltype(ic)::value;
            return table_entry((nibble<t, 3>(A) & 0x78u & mask) | ((nibble<t, 7>(U) & 0x780u & mU & mask) | base), tbl,
                               kTable, err);
          },
          move);
      const Row below = shift_lane(U, false);  // lane k+1's up slots, the other parity of row 2k+1
      set_row(0, (A << p) | (even & (p ? (Row)3 : (Row)0)));
      set_row(1, ((((U >> 2) & M3) << p) | ((below & M3) << (2 - p))) & ln.odd_mask);
    } else {
      const int n = ((C >> 1) + ln.par + 1) & 1;  // -kl0
      const Row below = shift_lane(even, false);
      A = odd << (2 * n);
      U = ((even >> (2 - 2 * n)) & M3) | (((below >> (2 - 2 * n)) & M3) << 2);
      const uint32_t bulk = tbl + (ln.odd_on ? 0u : kIdleAt), mask = ln.odd_on ? ~0u : 0u;
      const uint32_t first = tbl + (!ln.odd_on ? kIdleAt : n ? kSideAt : 0u), mask_last = ln.odd_on && n ? ~0u : 0u;
      const uint32_t last = tbl + (mask_last ? kSideAt : kIdleAt);
      faces<S, C, MODE>(
          dr, K, x, lane,
          [&](auto ic) {
            constexpr int t = decltype(ic)::value;
            return corners(ic, t == 0 ? first : t == NS ? last : bulk, t == NS ? mask_last : mask);
          },
          move);
      const Row above = shift_lane(U >> 2, true);  // lane k-1's down slots, the other parity of row 2k
      const Row rest = ln.first ? even >> (2 * n) : above;
      set_row(1, (A >> (2 * n)) & ln.odd_mask);
      set_row(0, ((U & M3) << (2 - 2 * n)) | ((rest & M3) << (2 * n)));
    }
    return dsum;
  }
};

// A launch form: NC warps that sweep and NP warps that produce for them, per
// CTA.  NP = 0: every warp sweeps, draws its own blocks where a vote finds a
// need, and the CTA rebuilds the tables of the next kSweeps sweeps together.
// NP > 0: the producing warps draw every block of the next kSweeps sweeps and
// write their tables while the sweeping warps run the current ones from shared
// memory (two sets of each).  PER: the CTAs that an SM holds at once, which the
// sweeps per set and the launch's register bound are chosen for.
constexpr size_t kSmShared = 228 * 1024, kCtaReserved = 1024;  // shared memory of an SM; taken by the system per CTA
template <class Geo, int NC, int NP, int PER>
struct Form {
  static constexpr int kThreads = 32 * (NC + NP), kPerSm = PER;
  static constexpr int kRegCtas = NP ? PER : 4;  // CTAs per SM of the register bound (sweeping warps need no more than 128)
  static constexpr int kCtaChains = NC * Geo::kChains;
  static constexpr int kSets = NP ? 2 : 1;
  static constexpr int draw_words(int sweeps) {
    return NP ? kSets * sweeps * NC * Geo::kBatches * kBatchWords : NC * 2 * kBatchWords;
  }
  // Dynamic shared memory: alignment slack, the tables, the list of entries
  // with a threshold, the draws, the output staging of each chain and, for NP =
  // 0, the raw thresholds of the next set's sweeps.
  static constexpr size_t bytes(int sweeps, int n_classes) {
    return 2048 + (size_t)kSets * sweeps * Geo::kTable + Geo::kEntries * sizeof(uint32_t) + 16 +
           (size_t)draw_words(sweeps) * 4 + (size_t)kCtaChains * 2 * Geo::kW * 4 +
           (NP ? 0 : (size_t)sweeps * n_classes * 4);
  }
  // PER CTAs fit on an SM (NP = 0: with schedules of up to 128 thresholds).
  static constexpr bool fits(int sweeps) { return PER * (bytes(sweeps, 128) + kCtaReserved) <= kSmShared; }
  static constexpr int kSweeps = fits(8) ? 8 : fits(4) ? 4 : fits(2) ? 2 : 1;
  static_assert(fits(kSweeps), "the CTAs that the launch rules count on do not fit");
  static constexpr int kDrawWords = draw_words(kSweeps);
  static constexpr size_t smem_bytes(int n_classes) { return bytes(kSweeps, n_classes); }
};

// What a producing warp does for one set of sweeps [t0, t0 + ns): the draws of
// every sweeping warp and the thresholds of the tables.
template <class Geo, int NC, int NP, int PER>
__device__ __forceinline__ void produce(int t0, int ns, const core::SaDraws (&base)[NC], const core::SweepTables& tab,
                                        const PhiloxKeys& K, uint32_t tables, const uint32_t* upd, int n_upd,
                                        uint32_t* draws, int pw, int lane) {
  const int k = lane & (Geo::G - 1);
  constexpr int kSweeps = Form<Geo, NC, NP, PER>::kSweeps;
  for (int j = pw * 32 + lane; j < n_upd; j += NP * 32) {
    const uint32_t v = upd[j], a = tables + 8u * (v >> 16) + 4u;
    const uint32_t* T = tab.T + (size_t)t0 * tab.n_classes + (v & 0xFFFFu);
    uint32_t A[kSweeps];
#pragma unroll
    for (int s = 0; s < kSweeps; ++s) A[s] = s < ns ? __ldg(&T[(size_t)s * tab.n_classes]) : 0u;
#pragma unroll
    for (int s = 0; s < kSweeps; ++s) core::sts_u32(a + (uint32_t)s * Geo::kTable, A[s]);
  }
#pragma unroll
  for (int w = 0; w < NC; ++w) {
    core::SaDraws dr = base[w];
    for (int s = 0; s < ns; ++s) {
      dr.sweep((uint32_t)(t0 + s), K);
      uint32_t* x = draws + (s * NC + w) * Geo::kBatches * kBatchWords;
#pragma unroll 2
      for (int j = (pw + s) % NP; j < Geo::kBatches; j += NP) {
        constexpr int B1 = Geo::start(1), B2 = Geo::start(2), B3 = Geo::start(3), F3 = Geo::first(3);
        const int C = j < B1 ? 0 : j < B2 ? 1 : j < B3 ? 2 : 3;
        const int j0 = j < B1 ? 0 : j < B2 ? B1 : j < B3 ? B2 : B3;
        draw_batch<Geo::Q>(batch_counter<Geo>((uint32_t)C, j < B3 ? 0u : (uint32_t)F3, (uint32_t)(j - j0), k), dr, K,
                           x + j * kBatchWords, lane);
      }
    }
  }
}

// Anneal the n_chains (1 to kCtaChains) chains of a segment from chain first by
// one CTA.  chain0, init0 and out0 are those of the segment's chain 0; groups
// past n_chains run a copy of the last chain and write nothing.  smem: Form::smem_bytes(tab.n_classes) bytes.
template <class Geo, int NC, int NP, int PER>
__device__ __forceinline__ void anneal_coop_cta(const uint32_t* __restrict__ init0, uint64_t chain0, int64_t first,
                                                int n_chains, const core::ChainOut& out0, const core::SweepTables& tab,
                                                const PhiloxKeys& K, uint8_t* smem) {
  using F = Form<Geo, NC, NP, PER>;
  constexpr int G = Geo::G, NW = Geo::NW, W = Geo::kW, kSweeps = F::kSweeps;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = lane & (G - 1);
  const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t pad = ((s0 + 2047u) & ~2047u) - s0, tables = s0 + pad;
  constexpr uint32_t kTable = Geo::kTable;
  constexpr int kEntries = Geo::kEntries;
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
  static_assert(kEntries % F::kThreads == 0, "whole warps in every pass");
  for (int e = tid; e < kEntries; e += F::kThreads) {
    const int src = Geo::sig_source(e);
    const int2 sg = src >= 0 ? __ldg(&tab.sig[src]) : make_int2(1, -1);
#pragma unroll
    for (int s = 0; s < F::kSets * kSweeps; ++s)
      core::sts_u2(tables + (uint32_t)s * Geo::kTable + 8u * (uint32_t)e, make_uint2((uint32_t)sg.x, 0u));
    core::append_entry(sg.y >= 0, ((uint32_t)e << 16) | (uint32_t)sg.y, upd, n_upd_s);
  }
  __syncthreads();
  const int n_upd = n_upd_s[0];

  if constexpr (NP > 0) if (warp >= NC) {  // a producing warp: one set ahead of the sweeping ones
    core::SaDraws base[NC];
#pragma unroll
    for (int w = 0; w < NC; ++w) {
      const uint64_t ch = chain0 + (uint64_t)(first + min(w * Geo::kChains + lane / G, n_chains - 1));
      base[w].init((uint32_t)ch, kTagSA | ((uint32_t)(ch >> 32) << 8), K);
    }
    for (int t0 = 0, set = 0; t0 < n_live; t0 += kSweeps, set ^= 1) {
      produce<Geo, NC, NP, PER>(t0, min(kSweeps, n_live - t0), base, tab, K, tables + (uint32_t)(set * kSweeps) * kTable, upd,
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

  Geo S;  // the lane's rows
  int32_t e_lane = S.load(init, P_coset, k, tab.W);
  const typename Geo::Lane ln(k);
  core::SaDraws dr;
  dr.init((uint32_t)chain, kTagSA | ((uint32_t)(chain >> 32) << 8), K);
  int32_t E_best = group_sum<G>(e_lane);
  uint32_t best[NW];
  copy_words(S.w, best);

  // One sweep; x: its draws (kStaged) or the warp's two areas (kVote).
  auto sweep = [&](auto mode, uint32_t tbl, uint32_t* x) {
    constexpr Draws M = decltype(mode)::value;
    constexpr int X1 = M == kStaged ? Geo::start(1) * kBatchWords : 0, X2 = M == kStaged ? Geo::start(2) * kBatchWords : 0,
                  X3 = M == kStaged ? Geo::start(3) * kBatchWords : 0;
    uint32_t w0[NW], w1[NW], w2[NW];  // the rows after colours 0, 1 and 2, for the minimum
    const int32_t d0 = S.template phase<0, M>(ln, tbl, dr, K, x, lane, tab.err);
    copy_words(S.w, w0);
    const int32_t d1 = S.template phase<1, M>(ln, tbl, dr, K, x + X1, lane, tab.err);
    copy_words(S.w, w1);
    const int32_t d2 = S.template phase<2, M>(ln, tbl, dr, K, x + X2, lane, tab.err);
    copy_words(S.w, w2);
    const int32_t d3 = S.template phase<3, M>(ln, tbl, dr, K, x + X3, lane, tab.err);
    if (__any_sync(0xFFFFFFFFu, (d0 < 0) | (d1 < 0) | (d2 < 0) | (d3 < 0))) {
      const int32_t e0 = e_lane + d0, e1 = e0 + d1, e2 = e1 + d2, e3 = e2 + d3;
      const int32_t E0 = group_sum<G>(e0), E1 = group_sum<G>(e1), E2 = group_sum<G>(e2), E3 = group_sum<G>(e3);
      if (min(min(E0, E1), min(E2, E3)) < E_best) {  // the earliest phase with the lowest energy
        if (E0 < E_best) E_best = E0, copy_words(w0, best);
        if (E1 < E_best) E_best = E1, copy_words(w1, best);
        if (E2 < E_best) E_best = E2, copy_words(w2, best);
        if (E3 < E_best) E_best = E3, copy_words(S.w, best);
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
      uint32_t* x = NP ? draws + set * (F::kDrawWords / 2) + (s * NC + warp) * Geo::kBatches * kBatchWords
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
    if ((i & (i + 1)) == 0) copy_words(S.w, saved);
    sweep(std::integral_constant<Draws, kFrozen>{}, tables, nullptr);
    if (may_stop) {
      uint32_t diff = 0;
#pragma unroll
      for (int j = 0; j < NW; ++j) diff |= S.w[j] ^ saved[j];
      const uint32_t same = __ballot_sync(0xFFFFFFFFu, diff == 0u) >> (lane & ~(G - 1));
      done |= (same & (0xFFFFFFFFu >> (32 - G))) == 0xFFFFFFFFu >> (32 - G);
      if (__all_sync(0xFFFFFFFFu, done)) break;
    }
  }

  const int32_t E_final = group_sum<G>(e_lane);
  if (active && k == 0) {
    *out.best_E = E_best;
    if (out.final_E) *out.final_E = E_final;
  }
  auto emit = [&](const uint32_t (&v)[NW], uint32_t* dst) {
    for (int i = k; i < 2 * W; i += G) stage[i] = 0u;
    __syncwarp();
    Geo::place(v, stage, k);
    __syncwarp();
    if (active)
      for (int i = k; i < 2 * W; i += G) dst[i] = stage[i];
    __syncwarp();
  };
  if (out.final_cfg) emit(S.w, out.final_cfg);
  if (out.best_cfg) emit(best, out.best_cfg);
}

}  // namespace coop
}  // namespace xzzx
