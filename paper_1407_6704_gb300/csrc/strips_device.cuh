// Ordered spreading by strips, 3D: the sum of A_p g w over the stencils that reach each
// lattice cell, in a fixed order and without atomics.
#pragma once

#include "pibm_internal.cuh"

namespace pibm {

namespace {

// A warp owns a strip of 128 cells: one z plane of a busy tile; the strips of a tile
// share a CTA, and so the records in its L1.
template <int W, int R>
struct StripShape {
  using TD = TileDims<3>;
  static constexpr int SX = TD::TX, SY = TD::TY;
  static constexpr int CELLS = SX * SY;
  static constexpr int PER_TILE = TD::TC / CELLS;
  static constexpr int QUEUE = 64;
  static constexpr int WARPS = 4;  // strips per CTA
  static constexpr int ROWS = (SY + 2 * R) * (2 * R + 1);
  static constexpr int SEGS = ROWS * (2 * R + 1);  // R single cells, the strip's run, R cells
};

// The cells around a strip have to be distinct: a periodic axis at least as long as
// the strip and its two margins.
template <int W, int R>
bool strips_fit(const Geometry& g) {
  using S = StripShape<W, R>;
  const int span[3] = {S::SX + 2 * R, S::SY + 2 * R, 2 * R + 1};
  for (int k = 0; k < 3; ++k)
    if (g.periodic[k] && g.n[k] < span[k]) return false;
  return true;
}

// Where the weight wz of a term A_p g wx wy wz goes in the ordered sums. FP32 multiplies
// the weights first, ((wx wy) wz) A_p g, as the atomic spreading does: 16-bit storage
// turns another rounding into other stored values. FP64 multiplies A_p g once per particle
// and plane instead of the weights once per node: slice of 64^3 with 62,500 particles,
// 10 steps: 3.88 ms against 3.97.
template <typename FT>
constexpr bool PLANE_WITH_AMP = sizeof(FT) == 8;
// Values queued per particle: A_p g, and wz where it goes with the weights.
template <typename FT>
constexpr int QUEUED = PLANE_WITH_AMP<FT> ? 3 : 4;

// Where a strip lies; valid is false past the end of the list or of the lattice.
struct Strip {
  int x0, y0, z0;
  bool valid;
};

template <int W, int R>
__device__ __forceinline__ Strip strip_of(const Geometry& g, const BinMap& bm,
                                          const int* __restrict__ tbusy, unsigned nbusy,
                                          unsigned strip) {
  using S = StripShape<W, R>;
  using TD = TileDims<3>;
  Strip p = {0, 0, 0, false};
  const unsigned ti = strip / S::PER_TILE;
  if (ti >= nbusy) return p;
  const int t = tbusy[ti], row = t / bm.nt[0], part = (int)(strip % S::PER_TILE);
  p.x0 = (t - row * bm.nt[0]) * TD::TX;
  p.y0 = (row % bm.nt[1]) * TD::TY;
  p.z0 = (row / bm.nt[1]) * TD::TZ + part;
  p.valid = p.y0 < g.n[1] && p.z0 < g.n[2];
  return p;
}

// acc[k][cell] = component k of the sum over the cells of the calling warp's strip. A
// particle is met once, in the order of the neighbour cells by ascending z, y, x offset
// and of the slots inside a cell, so every cell receives its terms in that order; one
// lane takes one stencil node of the plane and one component (in turns). The particles
// are found first (32 slots tested at a time, the hits queued in order), so that the
// reads of their records do not wait for the sums. R: reach in cells of a stencil
// around its particle's bin. tf, tr: first node, and weights and A_p g, by slot.
template <int W, int R, typename FT>
__device__ __forceinline__ void strip_sums(const Geometry& g, const BinMap& bm, long long np,
                                           const Strip& st, const int4* __restrict__ tf,
                                           const FT* __restrict__ tr,
                                           const unsigned* __restrict__ start, unsigned* err,
                                           FT (&acc)[3][StripShape<W, R>::CELLS],
                                           int2 (&queue)[StripShape<W, R>::QUEUE],
                                           FT (&qv)[StripShape<W, R>::QUEUE][QUEUED<FT>]) {
  using S = StripShape<W, R>;
  constexpr int NODES = W * W, CPL = 32 / NODES;  // components side by side in a warp
  constexpr int NC = 3, TURNS = (NC + CPL - 1) / CPL;
  const int lane = threadIdx.x & 31;
  const int xend = min(st.x0 + S::SX, g.n[0]);
#pragma unroll
  for (int k = 0; k < NC; ++k)
    for (int i = lane; i < S::CELLS; i += 32) acc[k][i] = FT(0);
  const int ni = lane % W, nj = (lane / W) % W, comp = lane / NODES;
  int queued = 0;
  auto drain = [&]() {
    __syncwarp();
#pragma unroll 1
    for (int i0 = 0; i0 < queued; i0 += 4) {
      // four records' values at once, then their adds in order
      FT wt[4], v[4][TURNS];
      int c[4];
      bool in[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        in[u] = false;
        wt[u] = FT(0);
        c[u] = 0;
#pragma unroll
        for (int t = 0; t < TURNS; ++t) v[u][t] = FT(0);
        if (i0 + u >= queued) continue;
        const int2 e = queue[i0 + u];
        const FT* r = tr + (long long)e.x * TAP_RECORD;
        const int rx = (e.y & 0xff) - 8 + ni, ry = ((e.y >> 8) & 0xff) - 8 + nj;
        in[u] = rx >= 0 && rx < S::SX && ry >= 0 && ry < S::SY;
        c[u] = ry * S::SX + rx;
        wt[u] = r[ni] * r[4 + nj];
        if constexpr (!PLANE_WITH_AMP<FT>) wt[u] *= qv[i0 + u][3];
#pragma unroll
        for (int t = 0; t < TURNS; ++t)
          if (comp + t * CPL < NC) v[u][t] = qv[i0 + u][comp + t * CPL];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (in[u]) {
#pragma unroll
          for (int t = 0; t < TURNS; ++t)
            if (comp + t * CPL < NC) {
              FT& a = acc[comp + t * CPL][c[u]];
              a = fma(v[u][t], wt[u], a);
            }
        }
        __syncwarp();
      }
    }
    queued = 0;
  };
#pragma unroll 1
  for (int s0 = 0; s0 < S::SEGS; s0 += 32) {  // 32 segments of bins at a time
    unsigned lo = 0, hi = 0;
    const int sg = s0 + lane;
    if (sg < S::SEGS) {
      const int rr = sg / (2 * R + 1), i = sg - rr * (2 * R + 1);
      int cy = st.y0 - R + rr % (S::SY + 2 * R);
      int cz = st.z0 - R + rr / (S::SY + 2 * R);
      // R cells before the strip's run, the run, R cells after it
      int cx = i < R ? st.x0 - R + i : (i == R ? st.x0 : xend + i - R - 1);
      if (lattice_coord(cx, g.n[0], g.periodic[0]) && lattice_coord(cy, g.n[1], g.periodic[1]) &&
          lattice_coord(cz, g.n[2], g.periodic[2])) {
        const unsigned b = bin_index<3>(bm, cx, cy, cz);
        lo = start[b];
        hi = start[i == R ? b + (unsigned)(xend - st.x0) : b + 1];
      }
    }
    if (hi > (unsigned)np || lo > hi) {
      atomicOr(err, ERR_INDEX);
      hi = lo = 0;
    }
    // the particles of the 32 segments in order, 32 at a time: lane l of a turn takes
    // particle base + l, in the segment whose range of running counts holds it
    unsigned incl = hi - lo;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    const unsigned total = __shfl_sync(0xffffffffu, incl, 31);
    const unsigned before = lo - (incl - (hi - lo));  // slot = before + running index
    for (unsigned base = 0; base < total; base += 32) {
      const unsigned idx = base + lane;
      int seg = 0;  // segments whose particles all come before idx
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned u = __shfl_sync(0xffffffffu, incl, seg + o - 1);
        if (u <= idx) seg += o;
      }
      const unsigned sl = __shfl_sync(0xffffffffu, before, seg & 31) + idx;
      bool hit = false;
      int word = 0;
      FT v[QUEUED<FT>] = {};
      if (idx < total) {
        const int4 f = tf[sl];
        // first node relative to the strip, in the image that can reach it
        int dx = f.x - st.x0, dy = f.y - st.y0, dz = st.z0 - f.z;
        if (g.periodic[0]) {
          if (dx <= S::SX - g.n[0]) dx += g.n[0];
          else if (dx >= g.n[0] - W) dx -= g.n[0];
        }
        if (g.periodic[1]) {
          if (dy <= S::SY - g.n[1]) dy += g.n[1];
          else if (dy >= g.n[1] - W) dy -= g.n[1];
        }
        if (g.periodic[2]) {
          if (dz < 0) dz += g.n[2];
          else if (dz >= g.n[2]) dz -= g.n[2];
        }
        hit = dx > -W && dx < S::SX && dy > -W && dy < S::SY && dz >= 0 && dz < W;
        if (hit) {
          // A_p g and the weight of the strip's plane, once per particle
          word = (dx + 8) | (dy + 8) << 8;
          const FT* r = tr + (long long)sl * TAP_RECORD;
          const FT wz = r[8 + dz];
#pragma unroll
          for (int k = 0; k < 3; ++k) v[k] = PLANE_WITH_AMP<FT> ? r[12 + k] * wz : r[12 + k];
          if constexpr (!PLANE_WITH_AMP<FT>) v[3] = wz;
        }
      }
      const unsigned hits = __ballot_sync(0xffffffffu, hit);
      if (queued + __popc(hits) > S::QUEUE) drain();
      if (hit) {
        const int i = queued + __popc(hits & ((1u << lane) - 1u));
        queue[i] = make_int2((int)sl, word);
#pragma unroll
        for (int k = 0; k < QUEUED<FT>; ++k) qv[i][k] = v[k];
      }
      queued += __popc(hits);
    }
  }
  drain();
  __syncwarp();
}

}  // namespace

}  // namespace pibm
