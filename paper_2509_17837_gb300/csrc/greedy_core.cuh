// Randomised greedy matching (Algs. 5 and 6) on the GPU.
//
// One CTA per (shot, group of restarts); its warps take the group's restarts in
// turn.  The CTA first computes, in shared memory, each face's shortest distance
// to the open boundary of its decoding graph (w(u,b) of Eq.
// distance_u_boundary) by Bellman-Ford relaxation with the first step of its
// canonical walk there, and the defect list of each decoding-graph colour.  Then,
// colour by colour, every vertex's candidate list (below), which serves all the
// restarts of the CTA.  All of it depends on the shot only.
//
// Matching.  All candidate pairs are totally ordered by (w, key, u, v): w the
// pair weight of Eq. distance_u_v_def_new, key a Philox draw per pair (Alg. 6)
// or 0 (Alg. 5), u < v the stabilizer indices (0xFFFF for the virtual boundary
// vertex).  Scanning that order and keeping pairs whose ends are free gives
// the same matching as repeatedly matching every pair that is the best
// remaining pair of both its ends ("locally dominant" pairs), which is what
// the warp does, round by round, in parallel over vertices.  A vertex's best
// free partner is found from its candidate list: the other vertices sorted by
// (w, index), so the first free entry has the lowest weight and, among equal
// weights, the lowest (u, v); with random keys only the free entries tied with
// it at that weight are compared further.  Colours with more vertices than the
// CTA has list space for scan all candidates.
//
// Paths.  Every kept pair is joined by a canonical shortest path (a Z step
// toward the target whenever one is needed and possible, else an X step; to
// the boundary, the first of Z(+1,+1), Z(-1,-1), X(+1,-1), X(-1,+1) that lowers
// the boundary distance by its weight), added modulo two into the restart's
// configuration.  A walk that could not complete (never expected on a valid
// code) sets bit 7 of cbits and raises XZZX_DEVERR_GREEDY_WALK in the code's
// error area.
//
// What bounds it: dependent shared-memory loads of a few active lanes (walking
// lists, drawing tied keys), so occupancy; hence shared memory is carved to the
// code's own size, and one list buffer serves the two colours of a large code in
// turn.  Against lists for rotated d <= 17 only and a fixed carve for d = 31
// (identical references): 76 shots x 256 restarts at d = 31, p = 0.24 13.6 -> 2.85
// ms; 4000 x 100 planar d = 9 7.59 -> 2.35 ms; 100 x 100 planar d = 21 3.82 ->
// 1.05 ms; 4000 x 64 at d = 11 1.94 -> 1.69 ms; one shot x 32 at d = 25 0.58 -> 0.12
// ms.
#pragma once

#include <cmath>

#include "anneal_core.cuh"
#include "internal.h"
#include "philox.cuh"

namespace xzzx {
namespace greedy {

// Warps of a CTA (choose_warps): 8 for codes of up to 150 faces per
// decoding-graph colour (rotated d <= 17, planar d <= 11), 16 above, where the lists
// take long to build and most of the shared memory, 4 where there is too little
// for 8 to do.
constexpr int kFewWarps = 4, kSmallWarps = 8, kLargeWarps = 16, kSmallFaces = 150;
// A launch of at most one CTA per two SMs gives each restart two warps, one per colour.
inline bool few_ctas(int64_t n, int n_sm) { return 2 * n <= n_sm; }
// A launch takes the largest restarts-per-warp count (8, 4, 2 or 1) that still
// gives it enough CTAs: large launches then share each CTA's setup across more
// restarts, small ones keep their CTAs.  Lists of small codes cost little next
// to a restart, and several waves of CTAs (13 per SM) fill the launch's tail; the
// lists of larger codes cost about as much as one restart, so two CTAs per SM are
// enough.
constexpr int kMaxRestartsPerWarp = 8;
inline int64_t min_ctas(bool large, int n_sm) { return (int64_t)n_sm * (large ? 2 : 13); }
// CTAs of a shot's restarts at rpw restarts per warp.
inline int greedy_groups(int restarts, int warps, int rpw) { return (restarts + warps * rpw - 1) / (warps * rpw); }
// Reference modes: greedy matching with lexicographic ties (Alg. 5), with
// random ties (Alg. 6), or every defect joined to its nearer boundary.
constexpr int kInitGreedy = 0, kInitGreedyRandom = 1, kInitBoundary = 2;
constexpr int32_t kInf = 0x3FFFFFFF;

// Geometry of the rotated layout: faces (a, b), a, b in [-1, d-1]; qubit
// (r, c) = r*d + c.  The four edges of a face in walking order: Z(+1,+1),
// Z(-1,-1), X(+1,-1), X(-1,+1), crossing the qubit (max a, max b).
struct RotGeo {
  __device__ static int face(const int16_t* at, int d, int a, int b) {
    if (a < -1 || a > d - 1 || b < -1 || b > d - 1) return -1;
    return at[(a + 1) * (d + 1) + (b + 1)];
  }
  __device__ static int qubit(int d, int r, int c) { return (r >= 0 && r < d && c >= 0 && c < d) ? r * d + c : -1; }
  __device__ static void step(int a, int b, int e, int& na, int& nb, int& qr, int& qc) {
    na = a + ((e & 1) ? -1 : 1);
    nb = b + ((e == 1 || e == 2) ? -1 : 1);
    qr = max(a, na);
    qc = max(b, nb);
  }
  // Coordinates that a Z step (edge 0: +2) and an X step (edge 2: +2) move.
  __device__ static int zpos(int a, int b) { return a + b; }
  __device__ static int xpos(int a, int b) { return a - b; }
};

// Geometry of the planar layout: faces (i, j), i + j odd, of the (2d-1)^2
// grid; qubits on the sites with r + c even.  Edges in walking order: Z right
// and Z left (crossing (i, j+-1)), X down and X up (crossing (i+-1, j)).
struct PlanarGeo {
  __device__ static int face(const int16_t* at, int d, int a, int b) {
    const int g = 2 * d - 1;
    if (a < 0 || a >= g || b < 0 || b >= g) return -1;
    return at[a * g + b];
  }
  __device__ static int qubit(int d, int r, int c) {
    const int g = 2 * d - 1;
    if (r < 0 || r >= g || c < 0 || c >= g || ((r + c) & 1)) return -1;
    return planar_qubit(d, r, c);
  }
  __device__ static void step(int a, int b, int e, int& na, int& nb, int& qr, int& qc) {
    const int di = e < 2 ? 0 : (e == 2 ? 1 : -1);
    const int dj = e < 2 ? (e == 0 ? 1 : -1) : 0;
    na = a + 2 * di;
    nb = b + 2 * dj;
    qr = a + di;
    qc = b + dj;
  }
  __device__ static int zpos(int, int b) { return b; }
  __device__ static int xpos(int a, int) { return a; }
};

// Vertices a colour's candidate lists have room for: half of the colour's faces
// and a little (defect density stays below one half under independent noise),
// at least 64 and at most 256 (list entries are bytes).  None for colours of
// more than 800 faces (planar d >= 29), which mostly hold more than 256 defects:
// the lists' memory would only lower the occupancy of the scan that then runs
// (d = 31, p = 0.12: 4.96 against 4.26 ms, before three scanning CTAs fitted an SM).
__host__ __device__ inline int list_room(int faces_per_colour) {
  const int n = (faces_per_colour * 35 / 64 + 31) / 32 * 32;
  return faces_per_colour > 800 ? 0 : n < 64 ? 64 : n > 256 ? 256 : n;
}

inline bool is_large(const DevCode& C) { return C.ns / 2 > kSmallFaces && list_room(C.ns / 2) > 0; }

// Whether a launch scans every colour: without lists, or with so few restarts
// that the scan of a colour which has outgrown its list would leave most of a
// large CTA's warps idle, where the noise says that most colours will (1000 shots x
// 1, planar d = 27, p = 0.14: 8.6 -> 3.4 ms).
inline bool scans(const DevCode& C, const xzzx_noise& noise, int restarts) {
  const double a = 1.0 - 2.0 * (noise.px + noise.py), b = 1.0 - 2.0 * (noise.pz + noise.py);
  const double p = 0.5 * (1.0 - a * a * b * b), n = C.ns / 2 * p;  // defects of a colour of four-qubit faces
  const int room = list_room(C.ns / 2);
  return room == 0 || (restarts <= 4 && n + std::sqrt(n * (1.0 - p)) > room);
}

// Shared memory of a CTA: offsets in bytes; cols: colours whose lists are held at
// once (1 or 2), each in a buffer of list_bytes and tie_bytes; room: vertices a
// list has room for (0: every colour is scanned); matched: false for
// kInitBoundary, which has no pairs and needs none of that.  The boundary
// distances wb give way to the lists once they are in wd.
struct Carve {
  int wb, nb, fa, fb, step, syn, defects, pq, wd, lists, ties, cur, pairs, free_, cfg, misc, total;
  int list_stride, list_bytes, tie_stride, tie_bytes, vmax;
};
__host__ __device__ inline Carve carve(int ns, int sw, int w, int warps, int cols, int room, bool matched,
                                       int restarts_per_cta) {
  Carve c;
  int o = 0;
  auto take = [&](int bytes) {
    const int at = o;
    o = (o + bytes + 15) & ~15;
    return at;
  };
  const int half = ns / 2;      // faces per colour
  c.vmax = (half + 2 + 31) & ~31;  // vertices per colour, the virtual one too
  c.list_stride = room + 4;     // an odd number of words: lanes on different lists hit different banks
  c.tie_stride = room / 32 + 1;
  c.nb = take(4 * 2 * ns);
  c.fa = take(ns);
  c.fb = take(ns);
  c.step = take(ns);
  c.syn = take(4 * sw);
  c.defects = take(2 * 2 * c.vmax);
  c.pq = take(matched ? 2 * 4 * c.vmax : 0);
  c.wd = take(matched ? 2 * 4 * c.vmax : 0);
  // best and partner of each warp: beside the lists, or in their place when
  // the colour is scanned (without lists one area serves both colours: a warp
  // works on one at a time).
  const int scan = matched && c.vmax > room ? 4 * warps * c.vmax : 0, list = room * c.list_stride;
  c.list_bytes = room ? ((list > scan ? list : scan) + 15) & ~15 : 0;
  c.tie_bytes = (4 * room * c.tie_stride + 15) & ~15;
  const int lists = room ? cols * c.list_bytes : scan;
  c.wb = c.lists = take(lists > 4 * ns ? lists : 4 * ns);
  c.ties = take(cols * c.tie_bytes);
  c.cur = take(warps * room);
  c.pairs = take(4 * warps * room);
  c.free_ = take(matched ? 4 * warps * (c.vmax / 32) : 0);
  c.cfg = take(4 * restarts_per_cta * 2 * w);
  c.misc = take(4 * (4 + restarts_per_cta));  // n_def[2], usable[2], walk_error[]
  c.total = o;
  return c;
}

constexpr int kOut = -1, kNone = -2;

// A CTA's view of its shot.
template <class G>
struct Ctx {
  const int16_t* nb;    // [4][ns]: the face across edge e of a face; kOut: a boundary edge; kNone: no qubit there
  const int8_t *fa, *fb;
  const uint8_t* step;  // of a face: first edge of its walk to the boundary; 0xFF: none
  int d, w, nq, ns;
  uint32_t* err;        // the code's device error area
};

template <class G>
__device__ __forceinline__ void toggle(const Ctx<G>& X, uint32_t* cfg, int q, bool z_step) {
  if (!XZZX_CHECK(X.err, q >= 0 && q < X.nq)) return;
  atomicXor(&cfg[(z_step ? X.w : 0) + (q >> 5)], 1u << (q & 31));
}

// Toggles the qubit that edge e of face f crosses.
template <class G>
__device__ __forceinline__ void cross(const Ctx<G>& X, int f, int e, uint32_t* cfg) {
  int na, nb, qr, qc;
  G::step(X.fa[f], X.fb[f], e, na, nb, qr, qc);
  toggle(X, cfg, G::qubit(X.d, qr, qc), e < 2);
}

// Canonical internal walk: a Z step toward v whenever one is still needed and
// both the next face and the crossed qubit exist, else an X step.
template <class G>
__device__ bool walk_internal(const Ctx<G>& X, int u, int v, uint32_t* cfg) {
  int nz = G::zpos(X.fa[v], X.fb[v]) - G::zpos(X.fa[u], X.fb[u]);  // what is left, two a step
  int nx = G::xpos(X.fa[v], X.fb[v]) - G::xpos(X.fa[u], X.fb[u]);
  int cur = u;
  while (nz | nx) {
    int e = nz < 0 ? 1 : 0, next = nz ? X.nb[e * X.ns + cur] : kNone;
    if (next < 0 && nx) {
      e = nx < 0 ? 3 : 2;
      next = X.nb[e * X.ns + cur];
    }
    if (next < 0) return false;
    cross(X, cur, e, cfg);
    const int done = (e & 1) ? -2 : 2;
    if (e < 2) nz -= done;
    else nx -= done;
    cur = next;
  }
  return true;
}

// Walk to the open boundary: at each face the edge that the setup chose.
template <class G>
__device__ bool walk_boundary(const Ctx<G>& X, int u, uint32_t* cfg) {
  int cur = u;
  for (int guard = 0; guard < X.nq; ++guard) {
    const int e = X.step[cur];
    if (e == 0xFF) return false;
    cross(X, cur, e, cfg);
    cur = X.nb[e * X.ns + cur];
    if (cur < 0) return true;
  }
  return false;
}

// One colour of a shot: its defects as positions and boundary distances.
struct Vertices {
  const int16_t* D;   // face of vertex x < nd
  const int32_t* pq;  // zpos + 256 | (xpos + 256) << 16
  const int32_t* wd;  // w(u, b)
  int nd, nv;         // vertex nd (when nd is odd) is the virtual boundary vertex
};

__device__ __forceinline__ int32_t internal_weight(int32_t pu, int32_t pv, int32_t Wt_x, int32_t Wt_z) {
  return Wt_z * (abs((pu & 0xFFFF) - (pv & 0xFFFF)) >> 1) + Wt_x * (abs((pu >> 16) - (pv >> 16)) >> 1);
}
// Pair weight of vertices x != y.
__device__ __forceinline__ int32_t pair_weight(const Vertices& V, int x, int y, int32_t Wt_x, int32_t Wt_z) {
  if (x == V.nd) return V.wd[y];
  if (y == V.nd) return V.wd[x];
  return min(internal_weight(V.pq[x], V.pq[y], Wt_x, Wt_z), V.wd[x] + V.wd[y]);
}

// Ascending bitonic sort across the warp of 32 NK keys, element h * 32 + lane
// in key[h].
template <int NK>
__device__ __forceinline__ void warp_sort(uint32_t (&key)[NK], int lane) {
#pragma unroll
  for (int k = 2; k <= 32 * NK; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= 32) {
#pragma unroll
        for (int h = 0; h < NK; ++h) {
          const int o = h ^ (j >> 5);
          if (o < h) continue;
          const bool up = ((32 * h) & k) == 0;
          const uint32_t lo = min(key[h], key[o]), hi = max(key[h], key[o]);
          key[h] = up ? lo : hi;
          key[o] = up ? hi : lo;
        }
      } else {
        const bool lower = (lane & j) == 0;
#pragma unroll
        for (int h = 0; h < NK; ++h) {
          const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, key[h], j);
          const bool up = ((32 * h + lane) & k) == 0;
          key[h] = lower == up ? min(key[h], o) : max(key[h], o);
        }
      }
    }
  }
}

// Candidate list of vertex x, built by one warp: out[pos] the vertex, bit pos of
// ties set when its weight equals the previous entry's.  Returns false if a
// weight does not fit the 24 bits of the sort key.
template <int NK>
__device__ __forceinline__ bool build_list(const Vertices& V, int x, int32_t Wt_x, int32_t Wt_z, uint8_t* out,
                                           uint32_t* ties, int lane) {
  bool fits = true;
  uint32_t key[NK];
#pragma unroll
  for (int h = 0; h < NK; ++h) {
    const int y = lane + 32 * h;
    key[h] = 0xFFFFFFFFu;
    if (y < V.nv && y != x) {
      const int32_t w = pair_weight(V, x, y, Wt_x, Wt_z);
      fits = fits && w >= 0 && w < (1 << 24) - 1;  // keys stay below the 0xFFFFFFFF filler
      key[h] = ((uint32_t)w << 8) | (uint32_t)y;
    }
  }
  warp_sort<NK>(key, lane);
  uint32_t last = 0xFFFFFFFFu;  // the element before this block's first
#pragma unroll
  for (int h = 0; h < NK; ++h) {
    uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, key[h], 1);
    if (lane == 0) prev = last;
    last = __shfl_sync(0xFFFFFFFFu, key[h], 31);
    const int pos = 32 * h + lane;
    const bool on = pos < V.nv - 1;
    if (on) out[pos] = (uint8_t)(key[h] & 255u);
    const uint32_t t = __ballot_sync(0xFFFFFFFFu, on && pos > 0 && (key[h] >> 8) == (prev >> 8));
    if (lane == 0 && 32 * h < V.nv - 1) ties[h] = t;
  }
  return __all_sync(0xFFFFFFFFu, fits);
}

// The keys of Alg. 6: word 0 of Philox(seed; u | v << 16, restart, shot_lo, 2 |
// shot_hi << 8), the parts that depend on the shot or the restart taken once.
struct PairKeys {
  core::SaDraws dr;
  __device__ __forceinline__ PairKeys(uint64_t shot, const PhiloxKeys& K) {
    dr.init((uint32_t)shot, kTagGreedy | ((uint32_t)(shot >> 32) << 8), K);
  }
  __device__ __forceinline__ void restart(int i, const PhiloxKeys& K) { dr.sweep((uint32_t)i, K); }
  __device__ __forceinline__ uint32_t key(uint32_t u, uint32_t v, const PhiloxKeys& K) const {
    return dr.block(u | (v << 16), K).x;
  }
};

// Per-warp state of one matching.
struct Work {
  int16_t *best, *partner;
  uint32_t* free_;  // bit x: vertex x is free
  uint8_t* cur;     // first possibly-free entry of each list
};
__device__ __forceinline__ bool is_free(const Work& W, int x) { return (W.free_[x >> 5] >> (x & 31)) & 1u; }

// Greedy matching of one colour for one restart, by one warp: partner[].
// Returns false if a round could not complete (never expected).
template <bool LISTED>
__device__ __forceinline__ bool match(const Vertices& V, const Carve& c, const uint8_t* lists, const uint32_t* ties,
                                      const Work& W, bool random, const PairKeys& pk, const PhiloxKeys& K, int32_t Wt_x,
                                      int32_t Wt_z, uint32_t* err, int lane) {
  const int nd = V.nd, nv = V.nv;
  bool good = true;
  for (int x = lane; x < nv; x += 32) {
    W.partner[x] = -1;
    W.best[x] = -1;
    if (LISTED) W.cur[x] = 0;
  }
  for (int b = 0; b < nv; b += 32)
    if (lane == 0) W.free_[b >> 5] = nv - b >= 32 ? 0xFFFFFFFFu : (1u << (nv - b)) - 1u;
  __syncwarp();
  int unmatched = nv;
  while (unmatched > 0) {
    // A best partner that is still free stays the best (removing other vertices
    // cannot put one ahead of it), so only vertices whose best was matched in
    // the last round search again.
    for (int x = lane; x < nv; x += 32) {
      if (!is_free(W, x)) {
        W.best[x] = -1;
        continue;
      }
      const int bx = W.best[x];
      if (bx >= 0 && is_free(W, bx)) continue;
      const uint32_t sx = x == nd ? kBoundary : (uint32_t)V.D[x];
      int bestv = -1;
      if (LISTED) {
        // From the vertex's cursor to the first free entry: the lowest weight
        // among free vertices, and the lowest (u, v) at that weight.  Keys
        // order the free entries tied at that weight (Alg. 6).
        const uint8_t* Lx = lists + x * c.list_stride;
        const uint32_t* Tx = ties + x * c.tie_stride;
        int k = W.cur[x];
        while (k < nv - 1 && !is_free(W, Lx[k])) ++k;
        W.cur[x] = (uint8_t)k;
        if (k >= nv - 1) {  // no free vertex left for x: impossible with an even count
          W.best[x] = -1;
          good = false;
          continue;
        }
        bestv = Lx[k];
        if (random) {
          uint32_t bu = 0, bv = 0, bkey = 0;
          bool drawn = false;
          for (++k; k < nv - 1 && ((Tx[k >> 5] >> (k & 31)) & 1u); ++k) {
            const int y = Lx[k];
            if (!is_free(W, y)) continue;
            if (!drawn) {
              const uint32_t s0 = bestv == nd ? kBoundary : (uint32_t)V.D[bestv];
              bu = min(sx, s0);
              bv = max(sx, s0);
              bkey = pk.key(bu, bv, K);
              drawn = true;
            }
            const uint32_t sy = y == nd ? kBoundary : (uint32_t)V.D[y];
            const uint32_t u = min(sx, sy), v = max(sx, sy), key = pk.key(u, v, K);
            if (key < bkey || (key == bkey && (u < bu || (u == bu && v < bv)))) {
              bestv = y;
              bkey = key;
              bu = u;
              bv = v;
            }
          }
        }
      } else {
        // One pass over all candidates: a key is drawn only when a weight ties
        // the best so far.
        int32_t bw = kInf;
        uint32_t bkey = 0, bu = 0, bv = 0;
        bool drawn = false;
        for (int y = 0; y < nv; ++y) {
          if (y == x || !is_free(W, y)) continue;
          const int32_t w = pair_weight(V, x, y, Wt_x, Wt_z);
          if (w > bw) continue;
          const uint32_t sy = y == nd ? kBoundary : (uint32_t)V.D[y];
          const uint32_t u = min(sx, sy), v = max(sx, sy);
          uint32_t key = 0;
          if (w == bw) {
            if (random) {
              if (!drawn) {
                bkey = pk.key(bu, bv, K);
                drawn = true;
              }
              key = pk.key(u, v, K);
            }
            if (!(key < bkey || (key == bkey && (u < bu || (u == bu && v < bv))))) continue;
          } else {
            drawn = false;
          }
          bestv = y;
          bw = w;
          bkey = key;
          bu = u;
          bv = v;
        }
      }
      W.best[x] = (int16_t)bestv;
    }
    __syncwarp();
    // Matching phase: reads only best[], writes only partner[].
    for (int x = lane; x < nv; x += 32) {
      const int y = W.best[x];
      if (y > x && XZZX_CHECK(err, y < nv) && W.best[y] == x) {
        W.partner[x] = (int16_t)y;
        W.partner[y] = (int16_t)x;
      }
    }
    __syncwarp();
    int left = 0;
    for (int b = 0; b < nv; b += 32) {
      const uint32_t m = __ballot_sync(0xFFFFFFFFu, b + lane < nv && W.partner[b + lane] < 0);
      if (lane == 0) W.free_[b >> 5] = m;
      left += __popc(m);
    }
    __syncwarp();
    if (left == unmatched) {  // impossible for a strict total order; keep the warp from spinning
      good = false;
      break;
    }
    unmatched = left;
  }
  return good;
}

// One CTA: references of restarts [group * restarts / groups, (group + 1) *
// restarts / groups) of one shot.  syn: the shot's syndrome words; init / cbits:
// the shot's rows (restarts x 2w words, restarts bytes).  smem: carve().total
// bytes for at least that many restarts.
template <class G, int kWarps>
__device__ __forceinline__ void greedy_cta(const DevCode& C, const PhiloxKeys& K, uint64_t shot, int group, int groups,
                                           int cols, int room, int restarts, int mode, int32_t Wt_x, int32_t Wt_z,
                                           const uint32_t* __restrict__ syn, uint32_t* __restrict__ init,
                                           uint8_t* __restrict__ cbits, uint8_t* smem) {
  const int d = C.d, ns = C.ns, w = C.w;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int lo = (int)((int64_t)group * restarts / groups), hi = (int)((int64_t)(group + 1) * restarts / groups);
  const Carve c = carve(ns, C.sw, w, kWarps, cols, room, mode != kInitBoundary, hi - lo);
  int32_t* wb = reinterpret_cast<int32_t*>(smem + c.wb);
  int16_t* nb = reinterpret_cast<int16_t*>(smem + c.nb);            // [4][ns]
  int8_t* fa = reinterpret_cast<int8_t*>(smem + c.fa);
  int8_t* fb = reinterpret_cast<int8_t*>(smem + c.fb);
  uint8_t* step = smem + c.step;
  uint32_t* s_syn = reinterpret_cast<uint32_t*>(smem + c.syn);
  int16_t* defects = reinterpret_cast<int16_t*>(smem + c.defects);  // [2][vmax]
  int32_t* pq = reinterpret_cast<int32_t*>(smem + c.pq);            // [2][vmax]
  int32_t* wd = reinterpret_cast<int32_t*>(smem + c.wd);            // [2][vmax]
  uint32_t* cfgs = reinterpret_cast<uint32_t*>(smem + c.cfg);       // [hi - lo][2w]
  int* n_def = reinterpret_cast<int*>(smem + c.misc);               // [2]
  int* usable = n_def + 2;                                          // [2]
  int* walk_error = n_def + 4;                                      // [hi - lo]
  Work W;
  W.free_ = reinterpret_cast<uint32_t*>(smem + c.free_) + warp * (c.vmax / 32);
  W.cur = smem + c.cur + warp * room;

  // Faces, their neighbours, and distances over the boundary edges alone.
  for (int f = tid; f < ns; f += blockDim.x) {
    const int a = C.face_a[f], b = C.face_b[f];
    fa[f] = (int8_t)a;
    fb[f] = (int8_t)b;
    step[f] = C.face_c2[f];  // until the defects are listed
    int32_t best = kInf;
    for (int e = 0; e < 4; ++e) {
      int na, nb_, qr, qc;
      G::step(a, b, e, na, nb_, qr, qc);
      int to = kNone;
      if (G::qubit(d, qr, qc) >= 0) {
        to = G::face(C.face_at, d, na, nb_);
        if (to < 0) {
          to = kOut;
          best = min(best, e < 2 ? Wt_z : Wt_x);
        }
      }
      nb[e * ns + f] = (int16_t)to;
    }
    wb[f] = best;
  }
  for (int j = tid; j < C.sw; j += blockDim.x) s_syn[j] = syn[j];
  for (int j = tid; j < (hi - lo) * 2 * w; j += blockDim.x) cfgs[j] = 0u;
  for (int j = tid; j < hi - lo; j += blockDim.x) walk_error[j] = 0;
  __syncthreads();
  Ctx<G> X{nb, fa, fb, step, d, w, C.nq, ns, C.err};

  // Defect lists of both colours, in stabilizer-index order, a warp each.
  if (warp < 2) {
    int cnt = 0;
    for (int base = 0; base < ns; base += 32) {
      const int f = base + lane;
      const bool on = f < ns && ((s_syn[f >> 5] >> (f & 31)) & 1) && step[f] == warp;
      const uint32_t m = __ballot_sync(0xFFFFFFFFu, on);
      const int slot = cnt + __popc(m & ((1u << lane) - 1));
      if (on && XZZX_CHECK(C.err, slot < c.vmax)) defects[warp * c.vmax + slot] = (int16_t)f;
      cnt += __popc(m);
    }
    if (lane == 0) n_def[warp] = cnt;
  }
  // Boundary distances: relax until stable.
  for (int iter = 0; iter < ns + 1; ++iter) {
    int changed = 0;
    for (int f = tid; f < ns; f += blockDim.x) {
      const int32_t was = wb[f];
      int32_t cur = was;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int nf = nb[e * ns + f];
        if (nf >= 0) cur = min(cur, wb[nf] + (e < 2 ? Wt_z : Wt_x));
      }
      wb[f] = cur;
      changed |= cur != was;
    }
    if (!__syncthreads_or(changed)) break;
  }
  // The first edge, in walking order, that lowers the distance by its own weight.
  for (int f = tid; f < ns; f += blockDim.x) {
    int st = 0xFF;
#pragma unroll
    for (int e = 3; e >= 0; --e) {
      const int nf = nb[e * ns + f];
      const int32_t we = e < 2 ? Wt_z : Wt_x;
      if (nf == kOut ? we == wb[f] : nf >= 0 && wb[nf] + we == wb[f]) st = e;
    }
    step[f] = (uint8_t)st;
  }

  auto vertices = [&](int colour) {
    Vertices V;
    V.D = defects + colour * c.vmax;
    V.pq = pq + colour * c.vmax;
    V.wd = wd + colour * c.vmax;
    V.nd = n_def[colour];
    V.nv = V.nd + (V.nd & 1);
    return V;
  };
  if (mode == kInitBoundary) {
    __syncthreads();
    // Each defect joined to the nearer boundary of its decoding graph.
    for (int i = lo + warp; i < hi; i += kWarps)
      for (int colour = 0; colour < 2; ++colour) {
        const Vertices V = vertices(colour);
        for (int x = lane; x < V.nd; x += 32)
          if (!walk_boundary(X, V.D[x], cfgs + (i - lo) * 2 * w)) walk_error[i - lo] = 1;
      }
    __syncthreads();
  } else {
    for (int colour = 0; colour < 2; ++colour)
      for (int x = tid; x < n_def[colour]; x += blockDim.x) {
        const int f = defects[colour * c.vmax + x];
        pq[colour * c.vmax + x] = (G::zpos(fa[f], fb[f]) + 256) | ((G::xpos(fa[f], fb[f]) + 256) << 16);
        wd[colour * c.vmax + x] = wb[f];
      }
    if (tid < 2) usable[tid] = n_def[tid] + (n_def[tid] & 1) <= room;
    __syncthreads();
  }
  PairKeys pk(shot, K);
  for (int first = 0; first < 2 && mode != kInitBoundary; first += cols) {
    for (int slot = 0; slot < cols; ++slot) {  // candidate lists, every warp of the CTA building some
      const Vertices V = vertices(first + slot);
      if (V.nv <= 2 || V.nv > room) continue;  // two vertices match each other
      bool fits = true;
      for (int x = warp; x < V.nv; x += kWarps) {
        uint8_t* Lx = smem + c.lists + slot * c.list_bytes + x * c.list_stride;
        uint32_t* Tx = reinterpret_cast<uint32_t*>(smem + c.ties + slot * c.tie_bytes) + x * c.tie_stride;
        fits = (V.nv <= 32   ? build_list<1>(V, x, Wt_x, Wt_z, Lx, Tx, lane)
                : V.nv <= 64 ? build_list<2>(V, x, Wt_x, Wt_z, Lx, Tx, lane)
                : V.nv <= 128 ? build_list<4>(V, x, Wt_x, Wt_z, Lx, Tx, lane)
                              : build_list<8>(V, x, Wt_x, Wt_z, Lx, Tx, lane)) && fits;
      }
      if (lane == 0 && !fits) usable[first + slot] = 0;
    }
    __syncthreads();
    for (int it = warp; it < cols * (hi - lo); it += kWarps) {  // both colours of a warp's restarts, not one of more
      const int slot = it >= hi - lo, i = lo + it - slot * (hi - lo);
      const Vertices V = vertices(first + slot);
      if (V.nv == 0) continue;
      const bool listed = usable[first + slot] != 0;
      const uint8_t* lists = smem + c.lists + slot * c.list_bytes;
      const uint32_t* ties = reinterpret_cast<const uint32_t*>(smem + c.ties + slot * c.tie_bytes);
      const int len = listed ? room : c.vmax;  // per warp: best, then partner
      W.best = reinterpret_cast<int16_t*>(smem + (listed ? c.pairs : c.lists + slot * c.list_bytes)) + warp * 2 * len;
      W.partner = W.best + len;
      __syncwarp();  // the warp's previous matching is walked
      if (mode == kInitGreedyRandom) pk.restart(i, K);
      bool good = true;
      if (V.nv == 2) {
        if (lane < 2) W.partner[lane] = (int16_t)(1 - lane);
        __syncwarp();
      } else {
        good = listed ? match<true>(V, c, lists, ties, W, mode == kInitGreedyRandom, pk, K, Wt_x, Wt_z, C.err, lane)
                      : match<false>(V, c, lists, ties, W, mode == kInitGreedyRandom, pk, K, Wt_x, Wt_z, C.err, lane);
      }
      uint32_t* cfg = cfgs + (i - lo) * 2 * w;
      bool ok = good;
      // Join every kept pair.
      for (int x = lane; x < V.nd; x += 32) {
        const int y = W.partner[x];
        if (y <= x) continue;
        const int fx = V.D[x];
        if (y == V.nd) {
          ok = walk_boundary(X, fx, cfg) && ok;
        } else {
          const int fy = V.D[y];
          if (internal_weight(V.pq[x], V.pq[y], Wt_x, Wt_z) <= V.wd[x] + V.wd[y]) ok = walk_internal(X, fx, fy, cfg) && ok;
          else ok = walk_boundary(X, fx, cfg) && walk_boundary(X, fy, cfg) && ok;
        }
      }
      if (!ok) walk_error[i - lo] = 1;
    }
    __syncthreads();  // the lists are free for the other colour, the configurations complete
  }

  // Output R_i and its commutation bits with L_Z (bit 0) and L_X (bit 1).
  const uint32_t* LX = C.logical;
  const uint32_t* LZ = C.logical + 2 * w;
  for (int i = lo + warp; i < hi; i += kWarps) {
    const uint32_t* cfg = cfgs + (i - lo) * 2 * w;
    uint32_t* out = init + (size_t)i * 2 * w;
    uint32_t par = 0;  // bit 0: with L_Z, bit 1: with L_X
    for (int j = lane; j < w; j += 32) {
      const uint32_t ex = cfg[j], ez = cfg[w + j];
      out[j] = ex;
      out[w + j] = ez;
      par ^= (uint32_t)(__popc((ex & LZ[w + j]) ^ (ez & LZ[j])) & 1) |
             ((uint32_t)(__popc((ex & LX[w + j]) ^ (ez & LX[j])) & 1) << 1);
    }
    par = __reduce_xor_sync(0xFFFFFFFFu, par);
    if (lane == 0) {
      // A walk that could not complete is recorded in the code's error area
      // (XZZX_DEVERR_GREEDY_WALK) and in bit 7 of the restart's class byte.
      const bool bad = walk_error[i - lo] != 0 || (i == 0 && injected(C.err, XZZX_DEVERR_GREEDY_WALK));
      if (bad) raise_device_error(C.err, XZZX_DEVERR_GREEDY_WALK);
      cbits[i] = (uint8_t)(par | (bad ? 0x80 : 0));
    }
  }
}

// How the shots of one code are cut at rpw restarts per warp: CTAs per shot,
// colours held at once, room of the lists, shared memory.
struct Cut {
  int groups = 1, cols = 2, room = 0;
  size_t smem = 0;
};
inline Cut cut_of(const DevCode& C, int warps, int restarts, int mode, int rpw, bool few, bool scan) {
  Cut k;
  const bool matched = mode != kInitBoundary;
  k.room = matched && !scan ? list_room(C.ns / 2) : 0;
  k.groups = few ? (restarts + warps / 2 - 1) / (warps / 2) : greedy_groups(restarts, warps, rpw);
  k.cols = C.ns / 2 > kSmallFaces && k.room && !few ? 1 : 2;
  k.smem = (size_t)carve(C.ns, C.sw, C.w, warps, k.cols, k.room, matched, (restarts + k.groups - 1) / k.groups).total;
  return k;
}

// Warps per CTA of a launch.
inline int choose_warps(const DevCode& C, int64_t n_shots, int restarts, int mode, bool scan, int n_sm) {
  const int half = C.ns / 2;
  // Past one wave of eight-warp CTAs, where a shot has not enough to keep them
  // busy, narrow ones hold twice the shots on an SM (p = 0.14, us, 8 warps / 4: 1000
  // shots x 1 restart d = 3 13.8 / 8.5, d = 9 28.5 / 20.8, d = 17 91 / 87; 1000 x 3 d = 5
  // 19.1 / 17.3, d = 17 98 / 114; 300 x 64 d = 3 34.7 / 30.2, with lists for two
  // vertices too; without them 1000 x 8 at d = 3 19.0 -> 16.1).
  if (half <= kSmallFaces && !scan && n_shots * greedy_groups(restarts, kSmallWarps, 1) > 4 * n_sm &&
      (half <= 6 || restarts <= 2 || (restarts == 3 && (half <= 12 || mode == kInitBoundary))))
    return kFewWarps;
  if (!is_large(C) || scan) return kSmallWarps;
  // Boundary references of a large code build no lists: its wide CTAs only pay
  // while all of them are resident (1000 shots x 1, us, 16 warps with the lists'
  // memory / 8 without: rotated d = 21 54 / 32, d = 31 182 / 67).
  return mode == kInitBoundary && n_shots * greedy_groups(restarts, kLargeWarps, 1) > min_ctas(true, n_sm) ? kSmallWarps
                                                                                                     : kLargeWarps;
}

}  // namespace greedy
}  // namespace xzzx
