// Annealing in the literal forms of Alg. 2 and Alg. 3, on both lattices: random
// site per attempt (order 1) and/or the minimum after every attempt (emin 1).
//
// One chain per thread.  Its rows sit in shared memory as [row][thread], so that
// lanes on different rows still hit different banks: two bits per qubit, one
// word per lattice row (32 bits up to d = 15, 64 above), shifted up by one empty
// slot and with one empty row before the first and after the last, so that a
// corner outside the lattice reads as the identity.  A face is then the same
// few operations whatever its shape, driven by a 32-bit descriptor: where its
// first row is, the bit of its corners, the bits a move flips, and which of three
// 256-entry tables its signature indexes (bulk; top and bottom; left and right --
// the two shapes of a pair leave different bits empty and agree on the entry
// they share).  Rotated: corners TL, TR in row a and BL, BR in row a + 1.  Planar:
// left, right in row i, up and down in rows i - 1 and i + 1.
//
// Draws.  Random site: attempts 2j and 2j + 1 of sweep t take their site and
// acceptance draws from one Philox block, computed an iteration ahead of its
// use together with the two descriptors.  Stabilizer order: the face's draw is
// a lane of the colour sweep's block (the counter and lane from a second table),
// computed when a move can be accepted; a one-block cache serves the faces that
// share it.
//
// Acceptance table.  Two tables of (dE, A) per CTA, the next sweep's thresholds
// written while this one's are read: one barrier per sweep.
//
// What bounds it: issue slots and the dependent chain load row, load entry,
// compare, store row, hidden by the other warps (the best rows are kept only when
// asked for, which leaves room for 32 warps per SM at d = 9).  Against a branch
// per shape, a table per warp and 64-bit rows: planar d = 9, 500 shots x 100
// restarts x 100 sweeps 25.0 -> 9.5 ms, d = 31 11.1 -> 3.2 ms; rotated d = 7 5.7 ->
// 2.7 ms, d = 31 8.7 -> 3.0 ms.
#include "anneal_core.cuh"

namespace xzzx {
namespace {

constexpr int kThreads = 128;
constexpr int kRegion = 256, kEntries = 3 * kRegion;

struct LiteralArgs {
  PhiloxKeys keys;
  uint64_t chain0;
  int64_t n_chains;
  int d, m, W;  // distance, generators, words per plane
  int n_sweeps, n_classes;
  int32_t Wt[4];
  int colour_start[5];
  const int16_t* face_a;
  const int16_t* face_b;
  const uint32_t* T;
  const int2* sig;  // the schedule's full table
  const uint32_t* init;
  int32_t* best_E;
  uint32_t* best_cfg;
  int32_t* final_E;
  uint32_t* final_cfg;
  uint32_t* err;
};

__host__ __device__ inline int n_rows(bool planar, int d) { return planar ? 2 * d - 1 : d; }
__device__ __forceinline__ int row_start(bool planar, int d, int r) {
  return planar ? (r >> 1) * (2 * d - 1) + ((r & 1) ? d : 0) : r * d;
}
__device__ __forceinline__ int row_len(bool planar, int d, int r) { return planar && (r & 1) ? d - 1 : d; }

// Entry of the schedule's signature table for table index p, -1 for indices no
// face reaches.  Rotated signature TL | TR << 2 | BL << 4 | BR << 6; planar left |
// right << 2 | up << 4 | down << 6.
template <bool PLANAR>
__device__ __forceinline__ int sig_source(int p) {
  const int e = p & 255, c0 = e & 3, c1 = (e >> 2) & 3, c2 = (e >> 4) & 3, c3 = e >> 6;
  if (p < kRegion) return PLANAR ? planar_sig_base(kPBulk) + e : e;
  if (PLANAR) {
    if (p < 2 * kRegion) {
      if (c2 == 0) return planar_sig_base(kPNoUp) + (c0 | (c1 << 2) | (c3 << 4));
      if (c3 == 0) return planar_sig_base(kPNoDown) + (c0 | (c1 << 2) | (c2 << 4));
    } else {
      if (c0 == 0) return planar_sig_base(kPNoLeft) + (c1 | (c2 << 2) | (c3 << 4));
      if (c1 == 0) return planar_sig_base(kPNoRight) + (c0 | (c2 << 2) | (c3 << 4));
    }
  } else {
    if (p < 2 * kRegion) {
      if (c0 == 0 && c1 == 0) return sig_base(kTop) + (c2 | (c3 << 2));
      if (c2 == 0 && c3 == 0) return sig_base(kBottom) + (c0 | (c1 << 2));
    } else {
      if (c0 == 0 && c2 == 0) return sig_base(kLeft) + (c1 | (c3 << 2));
      if (c1 == 0 && c3 == 0) return sig_base(kRight) + (c0 | (c2 << 2));
    }
  }
  return -1;
}

// Descriptor of face (a, b): bits 0-15 byte offset of its first row (rotated: row
// a, planar: row i - 1), 16-21 the bit of its corners there (planar: of row i),
// 22-23 the table region, 24-27 the bits a move flips in row a (planar: row i),
// 28-31 in row a + 1 (planar: bit 28 up, 29 down, 30 odd i).
template <bool PLANAR, typename Row>
__device__ __forceinline__ uint32_t descriptor(int a, int b, int d) {
  constexpr uint32_t kRow = kThreads * sizeof(Row);
  if (PLANAR) {
    const int g = 2 * d - 1, kl = (b - 1 - (a & 1)) >> 1;
    const bool up = a > 0, down = a < g - 1, left = b > 0, right = b < g - 1;
    return (uint32_t)a * kRow | ((uint32_t)(2 * (kl + 1)) << 16) | ((!up || !down ? 1u : !left || !right ? 2u : 0u) << 22) |
           ((left ? 2u : 0u) | (right ? 8u : 0u)) << 24 | (uint32_t)up << 28 | (uint32_t)down << 29 |
           (uint32_t)(a & 1) << 30;
  }
  const bool top = a < 0, bottom = a == d - 1, left = b < 0, right = b == d - 1;
  const uint32_t cols = (left ? 0u : 3u) | (right ? 0u : 12u);
  return (uint32_t)(a + 1) * kRow | ((uint32_t)(2 * (b + 1)) << 16) | ((top || bottom ? 1u : left || right ? 2u : 0u) << 22) |
         (top ? 0u : 0x6u & cols) << 24 | (bottom ? 0u : 0x9u & cols) << 28;
}

// Colour-sweep draw of face (a, b): counter word | lane << 30.
template <bool PLANAR>
__device__ __forceinline__ uint32_t draw_place(int a, int b) {
  const uint32_t colour = PLANAR ? (uint32_t)((a & 1) | ((((a + b - 1) >> 1) & 1) << 1)) : (uint32_t)((a & 1) | ((b & 1) << 1));
  const uint32_t ia = (uint32_t)(PLANAR ? a >> 1 : (a + 1) >> 1), ib = (uint32_t)(PLANAR ? b >> 2 : (b + 1) >> 1);
  return (colour << 16) | (ib << 8) | (ia >> 2) | ((ia & 3u) << 30);
}

template <typename Row>
__device__ __forceinline__ Row lds_row(uint32_t a) {
  if constexpr (sizeof(Row) == 4) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
  } else {
    uint64_t v;
    asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(a));
    return v;
  }
}
template <typename Row>
__device__ __forceinline__ void sts_row(uint32_t a, Row v) {
  if constexpr (sizeof(Row) == 4) asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v));
  else asm volatile("st.shared.u64 [%0], %1;" ::"r"(a), "l"(v));
}

// One attempt on the face of descriptor fd; rows: shared address of the chain's
// first (empty) row, tbl: of the sweep's table.  draw() gives the acceptance draw
// when it can matter.  Returns the energy change.
template <bool PLANAR, typename Row, typename Draw>
__device__ __forceinline__ int32_t attempt(uint32_t fd, uint32_t rows, uint32_t tbl, uint32_t* err, Draw&& draw) {
  constexpr uint32_t kRow = kThreads * sizeof(Row);
  const uint32_t at = rows + (fd & 0xFFFFu), s = (fd >> 16) & 63u;
  uint32_t idx;
  Row v0, v1, v2 = 0;
  const uint32_t su = PLANAR ? s + ((fd >> 29) & 2u) : 0u;  // up and down: one slot on in odd rows
  if constexpr (PLANAR) {
    v0 = lds_row<Row>(at);
    v1 = lds_row<Row>(at + kRow);
    v2 = lds_row<Row>(at + 2 * kRow);
    idx = ((uint32_t)(v1 >> s) & 15u) | (((uint32_t)(v0 >> su) & 3u) << 4) | (((uint32_t)(v2 >> su) & 3u) << 6);
  } else {
    v0 = lds_row<Row>(at);
    v1 = lds_row<Row>(at + kRow);
    idx = ((uint32_t)(v0 >> s) & 15u) | (((uint32_t)(v1 >> s) & 15u) << 4);
  }
  idx |= (fd >> 14) & 0x300u;  // region * 256
  const uint2 e = XZZX_CHECK(err, idx < (uint32_t)kEntries && !injected(err, XZZX_DEVERR_BOUNDS))
                      ? core::lds_u2(tbl + 8u * idx)
                      : make_uint2(0u, 0u);
  const int32_t dE = (int32_t)e.x;
  bool acc = dE <= 0;
  if (draw(e.y, acc)) {
    if constexpr (PLANAR) {
      sts_row<Row>(at, v0 ^ ((Row)((fd >> 28) & 1u) << su));
      sts_row<Row>(at + kRow, v1 ^ ((Row)((fd >> 24) & 15u) << s));
      sts_row<Row>(at + 2 * kRow, v2 ^ ((Row)((fd >> 29) & 1u) << su));
    } else {
      sts_row<Row>(at, v0 ^ ((Row)((fd >> 24) & 15u) << s));
      sts_row<Row>(at + kRow, v1 ^ ((Row)(fd >> 28) << s));
    }
    return dE;
  }
  return 0;
}

struct Carve {
  uint32_t tables, faces, places, upd, n_upd, rows, best, total;
};
template <typename Row>
__host__ __device__ inline Carve carve(bool planar, int d, int m, int order, bool keep) {
  Carve c;
  uint32_t o = 0;
  auto take = [&](uint32_t bytes) {
    const uint32_t at = o;
    o = (o + bytes + 15u) & ~15u;
    return at;
  };
  const uint32_t rows = (uint32_t)(n_rows(planar, d) + 2) * kThreads * (uint32_t)sizeof(Row);
  c.tables = take(2 * kEntries * 8);
  c.faces = take(4 * (uint32_t)m);
  c.places = take(order == 0 ? 4 * (uint32_t)m : 0);
  c.upd = take(4 * kEntries);
  c.n_upd = take(4);
  c.rows = take(rows);
  c.best = keep ? take(rows) : c.rows;
  c.total = o;
  return c;
}

// Rows at shared address rows -> planar words (x plane then z plane).
template <bool PLANAR, typename Row>
__device__ void store_words(uint32_t rows, int d, int W, uint32_t* __restrict__ cfg) {
  constexpr uint32_t kRow = kThreads * sizeof(Row);
  const int g = n_rows(PLANAR, d), nq = row_start(PLANAR, d, g - 1) + row_len(PLANAR, d, g - 1);
  int r = 0;
  for (int j = 0; j < W; ++j) {
    uint32_t wx = 0u, wz = 0u;
    const int lo = 32 * j, hi = min(lo + 32, nq);
    while (r + 1 < g && row_start(PLANAR, d, r + 1) <= lo) ++r;
    for (int rr = r; rr < g && row_start(PLANAR, d, rr) < hi; ++rr) {
      const uint64_t v = (uint64_t)lds_row<Row>(rows + (uint32_t)(rr + 1) * kRow) >> 2;
      const uint32_t fz = core::gather2(v), fx = core::gather2(v >> 1);
      const int start = row_start(PLANAR, d, rr) - lo;
      wz |= start >= 0 ? fz << start : fz >> (-start);
      wx |= start >= 0 ? fx << start : fx >> (-start);
    }
    cfg[j] = wx;
    cfg[W + j] = wz;
  }
}

template <bool PLANAR, typename Row, int ORDER, bool EMIN>
__global__ void __launch_bounds__(kThreads) anneal_literal_kernel(const __grid_constant__ LiteralArgs A) {
  extern __shared__ __align__(16) uint8_t smem[];
  constexpr uint32_t kRow = kThreads * sizeof(Row);
  const bool keep = A.best_cfg != nullptr;
  const Carve c = carve<Row>(PLANAR, A.d, A.m, ORDER, keep);
  const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(smem);
  uint32_t* faces = reinterpret_cast<uint32_t*>(smem + c.faces);
  uint32_t* places = reinterpret_cast<uint32_t*>(smem + c.places);
  uint32_t* upd = reinterpret_cast<uint32_t*>(smem + c.upd);
  int* n_upd_s = reinterpret_cast<int*>(smem + c.n_upd);
  const int tid = threadIdx.x, d = A.d, m = A.m, g = n_rows(PLANAR, d);
  const uint32_t rows = s0 + c.rows + (uint32_t)(tid * sizeof(Row)), best = s0 + c.best + (uint32_t)(tid * sizeof(Row));

  const int64_t c_raw = (int64_t)blockIdx.x * kThreads + tid;
  const bool active = c_raw < A.n_chains;
  const int64_t ci = active ? c_raw : A.n_chains - 1;  // inactive threads shadow a real chain
  const uint64_t chain = A.chain0 + (uint64_t)ci;
  const int P = (int)(ci & 3);

  // Descriptors and the tables' energy changes; the thresholds that can change
  // are listed as index << 16 | class.
  if (tid == 0) *n_upd_s = 0;
  __syncthreads();
  for (int f = tid; f < m; f += kThreads) {
    faces[f] = descriptor<PLANAR, Row>(A.face_a[f], A.face_b[f], d);
    if (ORDER == 0) places[f] = draw_place<PLANAR>(A.face_a[f], A.face_b[f]);
  }
  static_assert(kEntries % kThreads == 0, "whole warps in every pass");
  for (int k = tid; k < kEntries; k += kThreads) {
    const int src = sig_source<PLANAR>(k);
    const int2 sg = src >= 0 ? __ldg(&A.sig[src]) : make_int2(1, -1);
#pragma unroll
    for (int b = 0; b < 2; ++b) core::sts_u2(s0 + c.tables + 8u * (uint32_t)(b * kEntries + k), make_uint2((uint32_t)sg.x, 0u));
    core::append_entry(sg.y >= 0, ((uint32_t)k << 16) | (uint32_t)sg.y, upd, n_upd_s);
  }
  __syncthreads();
  const int n_upd = *n_upd_s;
  auto fill = [&](int t) {  // thresholds of sweep t
    const uint32_t tbl = s0 + c.tables + (uint32_t)(t & 1) * kEntries * 8u;
    const uint32_t* T = A.T + (size_t)t * A.n_classes;
    for (int k = tid; k < n_upd; k += kThreads) {
      const uint32_t v = upd[k];
      core::sts_u32(tbl + 8u * (v >> 16) + 4u, __ldg(&T[v & 0xFFFFu]));
    }
  };
  if (A.n_sweeps > 0) fill(0);

  // R_i L_P.  Rotated: L_X is column 0 (X on even rows, Z on odd rows), L_Z row 0
  // (Z on even columns, X on odd columns).  Planar: L_X is X on slot 0 of the even
  // rows, L_Z is Z on row 0.
  const uint32_t* init = A.init + (size_t)(ci >> 2) * 2 * A.W;
  int32_t nx = 0, ny = 0, nz = 0;
  sts_row<Row>(rows, 0);
  sts_row<Row>(rows + (uint32_t)(g + 1) * kRow, 0);
  for (int r = 0; r < g; ++r) {
    const int at = row_start(PLANAR, d, r), len = row_len(PLANAR, d, r);
    const uint32_t x = core::plane_field(init, A.W, at, len), z = core::plane_field(init + A.W, A.W, at, len);
    uint64_t v = core::spread2(z) | (core::spread2(x) << 1);
    if (P == 1 || P == 2) {
      if (PLANAR) v ^= (r & 1) ? 0ull : 2ull;
      else v ^= (r & 1) ? 1ull : 2ull;
    }
    if ((P == 2 || P == 3) && r == 0)
      v ^= (PLANAR ? 0x5555555555555555ull : 0x9999999999999999ull) & ((1ull << (2 * d)) - 1ull);
    sts_row<Row>(rows + (uint32_t)(r + 1) * kRow, (Row)(v << 2));
    const uint64_t zz = v & 0x5555555555555555ull, xx = (v >> 1) & 0x5555555555555555ull;
    ny += __popcll(xx & zz);
    nx += __popcll(xx & ~zz);
    nz += __popcll(zz & ~xx);
  }
  int32_t E = nx * A.Wt[2] + ny * A.Wt[3] + nz * A.Wt[1];
  int32_t E_best = E;
  // Stabilizer order, whose first sweeps save often: eight loads ahead of their
  // stores, the last row again past the end (one at a time each store waits for
  // its load; rotated d = 31, 60 chains per SM x 20 sweeps 8.18 -> 6.92 ms).  In random
  // order the larger code costs more than it saves (planar d = 9 0.46 -> 0.50 ms).
  auto save = [&] {
    if constexpr (ORDER == 0) {
      for (int r = 1; r <= g; r += 8) {
        Row v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = lds_row<Row>(rows + (uint32_t)min(r + i, g) * kRow);
#pragma unroll
        for (int i = 0; i < 8; ++i) sts_row<Row>(best + (uint32_t)min(r + i, g) * kRow, v[i]);
      }
    } else {
      for (int r = 1; r <= g; ++r) sts_row<Row>(best + (uint32_t)r * kRow, lds_row<Row>(rows + (uint32_t)r * kRow));
    }
  };
  if (keep) save();
  auto settle = [&] {
    if (E < E_best) {
      E_best = E;
      if (keep) save();
    }
  };

  core::SaDraws dr;
  dr.init((uint32_t)chain, (ORDER == 1 ? kTagSite : kTagSA) | ((uint32_t)(chain >> 32) << 8), A.keys);
  for (int t = 0; t < A.n_sweeps; ++t) {
    __syncthreads();  // this sweep's thresholds are in, and the other table is free
    if (t + 1 < A.n_sweeps) fill(t + 1);
    const uint32_t tbl = s0 + c.tables + (uint32_t)(t & 1) * kEntries * 8u;
    dr.sweep((uint32_t)t, A.keys);
    if constexpr (ORDER == 1) {
      uint4 r = dr.block(0u, A.keys);
      uint32_t f0 = faces[__umulhi(r.x, (uint32_t)m)], f1 = faces[__umulhi(r.z, (uint32_t)m)];
#pragma unroll 1
      for (int k = 0; k < m; k += 2) {
        const uint32_t a0 = r.y, a1 = r.w, g0 = f0, g1 = f1;
        r = dr.block((uint32_t)(k >> 1) + 1u, A.keys);  // the next two attempts' (unused after the last)
        f0 = faces[__umulhi(r.x, (uint32_t)m)];
        f1 = faces[__umulhi(r.z, (uint32_t)m)];
        E += attempt<PLANAR, Row>(g0, rows, tbl, A.err, [&](uint32_t T, bool acc) { return acc | (a0 < T); });
        if (EMIN) settle();
        if (k + 1 < m) {
          E += attempt<PLANAR, Row>(g1, rows, tbl, A.err, [&](uint32_t T, bool acc) { return acc | (a1 < T); });
          if (EMIN) settle();
        }
      }
      settle();
    } else {
      uint32_t cached = 0xFFFFFFFFu;
      uint4 rc = make_uint4(0u, 0u, 0u, 0u);
      for (int colour = 0; colour < 4; ++colour) {
        for (int f = A.colour_start[colour]; f < A.colour_start[colour + 1]; ++f) {
          E += attempt<PLANAR, Row>(faces[f], rows, tbl, A.err, [&](uint32_t T, bool acc) {
            if (acc || T == 0u) return acc;
            const uint32_t at = places[f], c0 = at & 0x3FFFFFFFu;
            if (c0 != cached) {
              rc = dr.block(c0, A.keys);
              cached = c0;
            }
            return lane_of(rc, (int)(at >> 30)) < T;
          });
          if (EMIN) settle();
        }
        settle();
      }
    }
  }

  if (!active) return;
  A.best_E[ci] = E_best;
  if (A.final_E) A.final_E[ci] = E;
  if (A.final_cfg) store_words<PLANAR, Row>(rows, d, A.W, A.final_cfg + (size_t)ci * 2 * A.W);
  if (A.best_cfg) store_words<PLANAR, Row>(best, d, A.W, A.best_cfg + (size_t)ci * 2 * A.W);
}

template <bool PLANAR, typename Row, int ORDER, bool EMIN>
xzzx_status launch_form(const LiteralArgs& A, unsigned grid, cudaStream_t stream) {
  static DeviceOnce once;
  xzzx_status st = once.run([] { return allow_shared(anneal_literal_kernel<PLANAR, Row, ORDER, EMIN>); });
  if (st) return st;
  const Carve c = carve<Row>(PLANAR, A.d, A.m, ORDER, A.best_cfg != nullptr);
  anneal_literal_kernel<PLANAR, Row, ORDER, EMIN><<<grid, kThreads, c.total, stream>>>(A);
  XZZX_CUDA_TRY(cudaGetLastError());
  return XZZX_OK;
}
template <bool PLANAR, typename Row>
xzzx_status launch_rows(const LiteralArgs& A, int order, int emin, unsigned grid, cudaStream_t stream) {
  if (order == 0) return launch_form<PLANAR, Row, 0, true>(A, grid, stream);
  return emin ? launch_form<PLANAR, Row, 1, true>(A, grid, stream) : launch_form<PLANAR, Row, 1, false>(A, grid, stream);
}

}  // namespace

xzzx_status check_anneal_args(const xzzx_code* code, const xzzx_schedule* sched, int n_shots, int restarts);
xzzx_status launch_anneal(const xzzx_code* code, const xzzx_schedule* sched, uint64_t seed, uint64_t shot0, int n_shots,
                          int restarts, const uint32_t* init, int32_t* best_E, uint32_t* best_cfg, int32_t* final_E,
                          uint32_t* final_cfg, cudaStream_t stream);

}  // namespace xzzx

using namespace xzzx;

extern "C" xzzx_status xzzx_anneal_variant(const xzzx_code* code, const xzzx_schedule* sched, uint64_t seed,
                                           uint64_t shot0, int n_shots, int restarts, int order, int emin,
                                           const uint32_t* init, int32_t* best_E, uint32_t* best_cfg,
                                           int32_t* final_E, uint32_t* final_cfg, void* stream) {
  xzzx_status st = check_anneal_args(code, sched, n_shots, restarts);
  if (st) return st;
  if (order != 0 && order != 1) return fail(XZZX_EINVAL, "order must be 0 (colour sweep) or 1 (random site)");
  if (emin != 0 && emin != 1) return fail(XZZX_EINVAL, "emin must be 0 (per phase) or 1 (per attempt)");
  if (n_shots == 0) return XZZX_OK;
  if ((st = check_ptr(init, "init")) || (st = check_ptr(best_E, "best_E"))) return st;
  if (order == 0 && emin == 0)
    return launch_anneal(code, sched, seed, shot0, n_shots, restarts, init, best_E, best_cfg, final_E, final_cfg,
                         (cudaStream_t)stream);
  LiteralArgs A;
  A.keys = philox_keys(seed);
  A.chain0 = shot0 * (uint64_t)restarts * 4u;
  A.n_chains = (int64_t)n_shots * restarts * 4;
  A.d = code->d;
  A.m = code->ns;
  A.W = code->w;
  A.n_sweeps = sched->n_sweeps;
  A.n_classes = sched->n_classes;
  for (int k = 0; k < 4; ++k) A.Wt[k] = sched->noise.W[k];
  for (int k = 0; k < 5; ++k) A.colour_start[k] = code->colour_start[k];
  A.face_a = code->dev.face_a;
  A.face_b = code->dev.face_b;
  A.T = sched->d_T;
  A.sig = sched->d_sig;
  A.init = init;
  A.best_E = best_E;
  A.best_cfg = best_cfg;
  A.final_E = final_E;
  A.final_cfg = final_cfg;
  A.err = code->dev.err;
  const int64_t grid = (A.n_chains + kThreads - 1) / kThreads;
  if (grid > 0x7FFFFFFF) return fail(XZZX_EINVAL, "too many chains for one launch");
  const bool wide = code->d > 15;
  if (code->layout == kLayoutPlanar)
    return wide ? launch_rows<true, uint64_t>(A, order, emin, (unsigned)grid, (cudaStream_t)stream)
                : launch_rows<true, uint32_t>(A, order, emin, (unsigned)grid, (cudaStream_t)stream);
  return wide ? launch_rows<false, uint64_t>(A, order, emin, (unsigned)grid, (cudaStream_t)stream)
              : launch_rows<false, uint32_t>(A, order, emin, (unsigned)grid, (cudaStream_t)stream);
}
