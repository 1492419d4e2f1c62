// Discrete adjoint of the coupled step, FP64: the exact gradient of the mean
// settling velocity (the particles' mean velocity along the last axis after the
// last step) with respect to tau, each particle's density ratio and each initial
// position.
//
// The forward run is the library's own step in deterministic mode, so a replayed
// stretch of steps reproduces the trajectory bit for bit. Every K steps the whole
// workspace is kept as a checkpoint; the reverse sweep replays each stretch from
// its checkpoint (the last one is taped by the forward sweep itself), keeping a tape
// of the workspace as it stands before each collision (stored populations of the step start, the spread force, the moment
// field, the particle state of both buffers and the cell list), then runs the
// adjoint of each step backwards:
//   1. streaming and collision (Eqs. 2, 3, 8) per cell: the pull of the forward
//      step becomes a pull in the opposite direction (each stored population feeds
//      exactly one post-stream one); then the adjoint of the post-stream
//      populations, of the force field, and the tau sensitivity;
//   2. spreading (Eq. 9) and the particle update (Eqs. 6-7, 13) per particle;
//   3. contacts (linear spring-dashpot) and interpolation (Eq. 4) per particle,
//      the latter spreading the adjoint of (rho_l, j_l) into a cell field;
//   4. that field into the adjoint of the post-stream populations.
#include <math.h>

#include <algorithm>
#include <vector>

#include "pibm_internal.cuh"

namespace pibm {

namespace {

// Delta-kernel taps with their derivatives d w / d X along one axis, FP64, the
// same nodes, weights and wall renormalisation as the forward interpolation.
template <int W>
struct TapsD {
  int idx[W];
  double w[W];
  double dw[W];
};

template <int W>
__device__ __forceinline__ void axis_taps_d(double X, int n, int periodic, TapsD<W>& t) {
  const int b = (int)floor(X - 0.5);
  const int first = (W == 2) ? b : b - 1;
  const double r0 = (double)first + 0.5 - X;  // d r0 / d X = -1
  if constexpr (W == 2) {
    t.w[0] = 1.0 + r0;
    t.dw[0] = -1.0;
    t.w[1] = -r0;
    t.dw[1] = 1.0;
  } else {
    // w = 1/4 (1 + cos th), 1/4 (1 - sin th), 1/4 (1 - cos th), 1/4 (1 + sin th),
    // th = pi r0 / 2, d th / d X = -pi / 2
    double sn, cs;
    sincospi(0.5 * r0, &sn, &cs);
    const double c = 0.125 * 3.14159265358979323846;
    t.w[0] = 0.25 * (1.0 + cs);
    t.dw[0] = c * sn;
    t.w[1] = 0.25 * (1.0 - sn);
    t.dw[1] = c * cs;
    t.w[2] = 0.25 * (1.0 - cs);
    t.dw[2] = -c * sn;
    t.w[3] = 0.25 * (1.0 + sn);
    t.dw[3] = -c * cs;
  }
  if (periodic) {
#pragma unroll
    for (int i = 0; i < W; ++i) {
      int k = (first + i) % n;
      t.idx[i] = k < 0 ? k + n : k;
    }
  } else {
    double s = 0.0, ds = 0.0;
#pragma unroll
    for (int i = 0; i < W; ++i) {
      const int k = first + i;
      const bool in = (k >= 0 && k < n);
      t.idx[i] = in ? k : (k < 0 ? 0 : n - 1);
      if (!in) {
        t.w[i] = 0.0;
        t.dw[i] = 0.0;
      }
      s += t.w[i];
      ds += t.dw[i];
    }
#pragma unroll
    for (int i = 0; i < W; ++i) {
      t.w[i] /= s;
      t.dw[i] = (t.dw[i] - t.w[i] * ds) / s;
    }
  }
}

// The same from the record the forward step kept (first node and weights), for a
// stencil that no wall clips: the four cosine weights are 1/4 (1 + c), 1/4 (1 - s),
// 1/4 (1 - c), 1/4 (1 + s), so the first two give the sine and cosine of the derivatives
// without evaluating them again.
template <int W>
__device__ __forceinline__ void axis_taps_kept(int first, const double* __restrict__ w, int n,
                                               TapsD<W>& t) {
#pragma unroll
  for (int i = 0; i < W; ++i) {
    t.w[i] = w[i];
    int k = first + i;
    if (k < 0 || k >= n) {
      k %= n;
      k = k < 0 ? k + n : k;
    }
    t.idx[i] = k;
  }
  if constexpr (W == 2) {
    t.dw[0] = -1.0;
    t.dw[1] = 1.0;
  } else {
    const double c = 0.125 * 3.14159265358979323846;
    t.dw[0] = fma(-4.0 * c, t.w[1], c);
    t.dw[1] = fma(4.0 * c, t.w[0], -c);
    t.dw[2] = -t.dw[0];
    t.dw[3] = -t.dw[1];
  }
}

// Neighbour of (x, y, z) in the direction sgn * e_a, wrapped on periodic axes;
// false when it lies beyond a wall (the link then bounces back).
template <int Q>
__device__ __forceinline__ bool adj_neighbour(const Geometry& g, int x, int y, int z, int a,
                                              int sgn, long long& c) {
  using L = Lattice<Q>;
  int t[3] = {x + sgn * L::e(a, 0), y + sgn * L::e(a, 1), z + sgn * L::e(a, 2)};
  bool in = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (L::e(a, k) == 0) continue;
    if (t[k] < 0 || t[k] >= g.n[k]) {
      if (g.periodic[k]) t[k] = t[k] < 0 ? t[k] + g.n[k] : t[k] - g.n[k];
      else in = false;
    }
  }
  c = t[0] + (long long)g.n[0] * (t[1] + (long long)g.n[1] * t[2]);
  return in;
}

constexpr int ADJ_THREADS = 256;
// Threads per CTA of the cell kernel: small CTAs, so that a few thousand cells
// already spread over every SM (its FP64 work is the bound at any size).
constexpr int ADJ_CELLS = 64;

// Moments of one value per velocity, weighted: m0 = sum w v, m1 = sum w e v,
// m2 = sum w e e v (diagonal, then xy, xz, yz). Opposite velocities share their
// weight, so an even sum and an odd difference per pair carry everything; the two
// weight classes (axis links, the rest) are summed before they are weighted.
template <int Q>
__device__ __forceinline__ void weighted_moments(const double (&v)[Q], double& m0,
                                                 double (&m1)[3], double (&m2)[6]) {
  using L = Lattice<Q>;
  constexpr int D = L::D;
  constexpr double w1 = L::w(1), w2 = L::w(Q - 1);
  double ax = 0.0, d0 = 0.0, dd[3] = {0.0, 0.0, 0.0}, od[3] = {0.0, 0.0, 0.0};
  double off[3] = {0.0, 0.0, 0.0}, pk[3] = {0.0, 0.0, 0.0}, mk[3] = {0.0, 0.0, 0.0};
  bool hd[3] = {false, false, false}, ho[3] = {false, false, false};  // sums begun
#pragma unroll
  for (int a = 1; a < Q; a += 2) {
    const double p = v[a] + v[a + 1], m = v[a] - v[a + 1];
    if (a < 2 * D) {  // the link along axis (a - 1) / 2
      pk[(a - 1) / 2] = p;
      mk[(a - 1) / 2] = m;
      ax = a == 1 ? p : ax + p;
      continue;
    }
    const bool first = a == 2 * D + 1;
    d0 = first ? p : d0 + p;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      if (L::e(a, k) == 0) continue;
      const double q = L::e(a, k) > 0 ? m : -m;
      dd[k] = hd[k] ? dd[k] + p : p;
      od[k] = hd[k] ? od[k] + q : q;
      hd[k] = true;
    }
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
      for (int l = k + 1; l < D; ++l) {
        const int s = L::e(a, k) * L::e(a, l), i = k + l - 1;
        if (s == 0) continue;
        const double q = s > 0 ? p : -p;
        off[i] = ho[i] ? off[i] + q : q;
        ho[i] = true;
      }
  }
  m0 = L::w(0) * v[0] + (w1 * ax + w2 * d0);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    m1[k] = k < D ? w1 * mk[k] + w2 * od[k] : 0.0;
    m2[k] = k < D ? w1 * pk[k] + w2 * dd[k] : 0.0;
    m2[3 + k] = w2 * off[k];
  }
}

// 1. Stream and collision adjoint per cell. Forward, with T_a = f*_a - (1 - om) f_a:
//   T_a = w_a [om rho (1 + 3 eu + 4.5 eu^2 - 1.5 uu) + cF (3 eF - 3 uF + 9 eu eF)],
//   u = (j + F/2) / rho, cF = 1 - om/2.
// The adjoint gb of f* is pulled from fnext, the adjoint of the post-stream
// populations of the following step: the stored population (x, a) reaches exactly
// one of them, (x + e_a, a) when that cell is in the lattice (wrapped on periodic
// axes), else (x, opp a) by bounce-back. Writes fb = adjoint of this step's
// post-stream populations (without the interpolation's moment terms), Fb = adjoint
// of the force, and adds this block's d L / d om to om_part[block].
// Everything the collision adjoint needs of gb are its weighted moments up to
// second order, M0 = sum w gb, M1 = sum w e gb, M2 = sum w e e gb:
//   V  = 3 M1 + 9 M2 u - 3 u M0,         ub = om rho V + cF (9 M2 F - 3 F M0),
//   jb = ub / rho, Fb = cF V + jb / 2,   rhob = om sum w gb poly - jb.u,
//   fb = (1 - om) gb + rhob + e.jb.
// FP64-bound: on a 96^3 D3Q19 lattice the form that summed every term per
// velocity took 1,996 us with a separate stream pass of 371 us; now 445 us with the pull
// included (and 48 us for the moment terms, which the stream pass used to add).
template <int Q>
__global__ void __launch_bounds__(ADJ_CELLS) k_adj_collide(Geometry g, double om, double cF,
                                                           const double* __restrict__ fin,
                                                           const double* __restrict__ F,
                                                           const double* __restrict__ fnext,
                                                           double* __restrict__ fbar,
                                                           double* __restrict__ Fbar,
                                                           double* __restrict__ om_part) {
  using L = Lattice<Q>;
  constexpr int D = L::D;
  constexpr int FS = FieldStride<D>::F;
  static_assert(StoreF64::S == 1, "stored values are f - w");
  __shared__ double red[ADJ_CELLS / 32];
  const unsigned cu = blockIdx.x * (unsigned)ADJ_CELLS + threadIdx.x;  // at most 2^26 cells
  double omb = 0.0;
  if (cu < (unsigned)g.ncell) {
    const long long c = cu;
    const unsigned n0 = (unsigned)g.n[0], n1 = (unsigned)g.n[1];
    const unsigned row = cu / n0;
    const int x = (int)(cu - row * n0);
    const int z = D == 3 ? (int)(row / n1) : 0;
    const int y = (int)(row - (unsigned)z * n1);
    const long long P = g.pitch;
    double f[Q], gb[Q];
    const bool inner = x >= 1 && x <= g.n[0] - 2 && y >= 1 && y <= g.n[1] - 2 &&
                       (D == 2 || (z >= 1 && z <= g.n[2] - 2));
    if (inner) {
      const int s0 = g.n[0], s01 = g.n[0] * g.n[1];
#pragma unroll
      for (int a = 0; a < Q; ++a) {
        const int o = L::e(a, 0) + s0 * L::e(a, 1) + s01 * L::e(a, 2);
        f[a] = fin[a * P + c - o];
        gb[a] = fnext[a * P + c + o];
      }
    } else {
#pragma unroll
      for (int a = 0; a < Q; ++a) {
        long long t;
        f[a] = adj_neighbour<Q>(g, x, y, z, a, -1, t) ? fin[a * P + t] : fin[opp(a) * P + c];
        gb[a] = adj_neighbour<Q>(g, x, y, z, a, 1, t) ? fnext[a * P + t] : fnext[opp(a) * P + c];
      }
    }
    double Fv[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < D; ++k) Fv[k] = F[FS * c + k];
    // moments of the populations (stored as f - w) and sum gb s
    double dev = f[0], gs = gb[0] * f[0], j[3] = {0.0, 0.0, 0.0};
    bool hj[3] = {false, false, false};
#pragma unroll
    for (int a = 1; a < Q; a += 2) {
      dev += f[a] + f[a + 1];
      gs += gb[a] * f[a];
      gs += gb[a + 1] * f[a + 1];
      const double m = f[a] - f[a + 1];
#pragma unroll
      for (int k = 0; k < D; ++k) {
        if (L::e(a, k) == 0) continue;
        const double q = L::e(a, k) > 0 ? m : -m;
        j[k] = hj[k] ? j[k] + q : q;
        hj[k] = true;
      }
    }
    const double rho = 1.0 + dev, inv = rcp_series(rho);
    double M0, M1[3], M2[6];
    weighted_moments<Q>(gb, M0, M1, M2);
    double u[3] = {0.0, 0.0, 0.0}, uu = 0.0, uF = 0.0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      u[k] = (j[k] + 0.5 * Fv[k]) * inv;
      uu += u[k] * u[k];
      uF += u[k] * Fv[k];
    }
    double M2u[3] = {0.0, 0.0, 0.0}, M2F[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
      for (int l = 0; l < D; ++l) {
        const double q = k == l ? M2[k] : M2[2 + k + l];
        M2u[k] += q * u[l];
        M2F[k] += q * Fv[l];
      }
    double M1u = 0.0, M1F = 0.0, uM2u = 0.0, uM2F = 0.0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      M1u += M1[k] * u[k];
      M1F += M1[k] * Fv[k];
      uM2u += u[k] * M2u[k];
      uM2F += u[k] * M2F[k];
    }
    const double poly1 = 3.0 * M1u + 4.5 * uM2u - 1.5 * uu * M0;  // sum w gb (poly - 1)
    const double guo = 3.0 * M1F - 3.0 * uF * M0 + 9.0 * uM2F;
    // sum gb f = gs + M0, whose M0 cancels against that of rho poly
    omb = dev * M0 - gs + rho * poly1 - 0.5 * guo;
    const double omrho = om * rho;
    double jb[3] = {0.0, 0.0, 0.0}, rhob = om * (M0 + poly1);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const double V = 3.0 * M1[k] + 9.0 * M2u[k] - 3.0 * u[k] * M0;
      jb[k] = (omrho * V + cF * (9.0 * M2F[k] - 3.0 * Fv[k] * M0)) * inv;
      Fbar[FS * c + k] = cF * V + 0.5 * jb[k];
      rhob -= jb[k] * u[k];
    }
    const double om1 = 1.0 - om;
    fbar[c] = om1 * gb[0] + rhob;
#pragma unroll
    for (int a = 1; a < Q; a += 2) {
      double ej = 0.0;
      bool first = true;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        if (L::e(a, k) == 0) continue;
        const double v = L::e(a, k) > 0 ? jb[k] : -jb[k];
        ej = first ? v : ej + v;
        first = false;
      }
      fbar[a * P + c] = om1 * gb[a] + (rhob + ej);
      fbar[(a + 1) * P + c] = om1 * gb[a + 1] + (rhob - ej);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) omb += __shfl_xor_sync(0xffffffffu, omb, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = omb;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < ADJ_CELLS / 32; ++w) omb += red[w];
    om_part[blockIdx.x] += omb;
  }
}

struct AdjArgs {
  Geometry g;
  Physics ph;
  BinMap bm;
  long long np;
  int cur;              // buffer of the step-start particle state in the tape
  // tape of the step (pointers into the tape copy of the workspace)
  const double* X;      // step-start state by storage position
  const double* U;
  const double* Un;     // U' by slot
  const double* gin;    // g by slot
  const double* mass;   // by storage position
  const double* Ap;
  const double* buoy;
  const double* rad;
  const double* gw;
  const unsigned* pid;
  const int4* cs;
  const unsigned* start;
  const int4* tf;       // stencil records of the step's ordered spreading, by slot
  const double* tr;
  const double* mom;    // moment field of the post-stream state [pitch][4]
  // adjoint state
  const double* Fbar;   // [pitch][FS]
  const double* Xb_in;  // adjoint of X' by slot
  const double* Ub_in;
  double* Xb_tmp;       // by slot
  double* Ub_tmp;
  double* Fcb;          // adjoint of F_c by slot
  double* rlb;          // adjoint of rho_l by slot
  double* jlb;          // adjoint of j_l by slot
  double* mb_tmp;       // adjoint of the density ratio from the update, by slot
  double* rjbar;        // adjoint of the moment field [pitch][4] (accumulated)
  double* Xb_out;       // adjoint of X by storage position
  double* Ub_out;
  double* drho;         // user order, accumulated over steps
  unsigned* err;
};

// The particle kernels give each particle ROWS = W^(d-1) lanes, one per stencil
// row of W cells along x, and keep PPB particles per CTA: tens of thousands of
// particles fill the GPU, and the FP64 taps, row sums and scalar updates each run
// on full warps. One thread per particle left most SMs with a single warp walking
// 64 taps one after another: on 20,000 particles of a 96^3 lattice the two kernels
// took 105 and 352 us, now 74 and 153 us.
template <int D, int W>
struct AdjShape {
  static constexpr int WZ = D == 3 ? W : 1;
  static constexpr int ROWS = W * WZ;
  static constexpr int THREADS = 128;
  static constexpr int PPB = THREADS / ROWS;
};

template <int D, int W>
struct AdjTapsShared {
  TapsD<W> t[AdjShape<D, W>::PPB][D];
};

// Taps of the CTA's particles, one thread per particle and axis; p[i] is the storage
// position of particle i (np: none).
template <int D, int W>
__device__ __forceinline__ void adj_block_taps(const AdjArgs& A, const unsigned* p,
                                               AdjTapsShared<D, W>& sh) {
  using S = AdjShape<D, W>;
  for (int i = threadIdx.x; i < S::PPB * D; i += S::THREADS) {
    const int q = i % S::PPB, k = i / S::PPB;
    if (p[q] >= (unsigned)A.np) continue;
    const long long sl = blockIdx.x * (long long)S::PPB + q;
    const int4 f = A.tf[sl];
    const int first = k == 0 ? f.x : (k == 1 ? f.y : f.z);
    if (A.g.periodic[k] || (first >= 0 && first <= A.g.n[k] - W))
      axis_taps_kept<W>(first, A.tr + sl * TAP_RECORD + 4 * k, A.g.n[k], sh.t[q][k]);
    else
      axis_taps_d<W>(A.X[k * A.np + p[q]], A.g.n[k], 0, sh.t[q][k]);
  }
}

// Storage positions of the CTA's particles into p (np when the slot is past the
// end or its record is out of range).
template <int D, int W>
__device__ __forceinline__ void adj_block_particles(const AdjArgs& A, unsigned* p) {
  using S = AdjShape<D, W>;
  if (threadIdx.x < S::PPB) {
    const long long sl = blockIdx.x * (long long)S::PPB + threadIdx.x;
    unsigned v = (unsigned)A.np;
    if (sl < A.np) {
      v = (unsigned)A.cs[sl].w;
      if (v >= (unsigned)A.np) {
        atomicOr(A.err, ERR_INDEX);
        v = (unsigned)A.np;
      }
    }
    p[threadIdx.x] = v;
  }
}

// Sum over the ROWS lanes of a particle (a power of two up to 16, aligned).
template <int ROWS>
__device__ __forceinline__ double row_sum(double v) {
#pragma unroll
  for (int o = ROWS / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 2. Spreading and particle update adjoint, per slot (implicit drag):
//   U' = N / den, N = m U + 2 A_p j_l + b G + F_c, den = m + 2 A_p rho_l,
//   X' = X + U', g = 2 (rho_l U' - j_l), F += A_p g w(X).
template <int D, int W>
__global__ void __launch_bounds__(AdjShape<D, W>::THREADS) k_adj_update(AdjArgs A) {
  using S = AdjShape<D, W>;
  __shared__ AdjTapsShared<D, W> sh;
  __shared__ unsigned sp[S::PPB];
  __shared__ double sums[S::PPB][1 + 2 * D];  // rho_l - S, sum w Fb, sum dw (Fb.g)
  const long long np = A.np;
  const Geometry& g = A.g;
  constexpr int FS = FieldStride<D>::F;
  adj_block_particles<D, W>(A, sp);
  __syncthreads();
  adj_block_taps<D, W>(A, sp, sh);
  __syncthreads();
  const int q = threadIdx.x / S::ROWS, row = threadIdx.x % S::ROWS;
  const long long slq = blockIdx.x * (long long)S::PPB + q;
  double rl = 0.0, gb[3] = {0.0, 0.0, 0.0}, xs[3] = {0.0, 0.0, 0.0};
  if (sp[q] < (unsigned)np) {
    const TapsD<W>(&t)[D] = sh.t[q];
    const int iy = row % W, iz = row / W;
    double gg[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < D; ++k) gg[k] = A.gin[k * np + slq];
    const double wy = t[1].w[iy], dwy = t[1].dw[iy];
    const double wz = D == 3 ? t[D - 1].w[iz] : 1.0, dwz = D == 3 ? t[D - 1].dw[iz] : 0.0;
    const long long r0 =
        (long long)g.n[0] * (t[1].idx[iy] + (long long)g.n[1] * (D == 3 ? t[D - 1].idx[iz] : 0));
    double R = 0.0, G[3] = {0.0, 0.0, 0.0}, H = 0.0;
#pragma unroll
    for (int ix = 0; ix < W; ++ix) {
      const long long c = r0 + t[0].idx[ix];
      const double w = t[0].w[ix];
      R += w * A.mom[4 * c];
      double Fg = 0.0;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const double Fb = A.Fbar[FS * c + k];
        G[k] += w * Fb;
        Fg += Fb * gg[k];
      }
      H += t[0].dw[ix] * Fg;
    }
    const double wyz = wy * wz;
    double Sg = 0.0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      Sg += G[k] * gg[k];
      gb[k] = wyz * G[k];
    }
    rl = wyz * R;
    xs[0] = wyz * H;
    xs[1] = dwy * wz * Sg;
    xs[2] = wy * dwz * Sg;
  }
  rl = row_sum<S::ROWS>(rl);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    gb[k] = row_sum<S::ROWS>(gb[k]);
    xs[k] = row_sum<S::ROWS>(xs[k]);
  }
  if (row == 0) {
    sums[q][0] = rl;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      sums[q][1 + k] = gb[k];
      sums[q][1 + D + k] = xs[k];
    }
  }
  __syncthreads();
  // --- the particle's scalars, one thread each ---
  if (threadIdx.x >= S::PPB || sp[threadIdx.x] >= (unsigned)np) return;
  const unsigned p = sp[threadIdx.x];
  const long long sl = blockIdx.x * (long long)S::PPB + threadIdx.x;
  const double m = A.mass[p], Ap = A.Ap[p], bu = A.buoy[p];
  // the moment field holds rho - S, as in the forward step
  const double rho_l = sums[threadIdx.x][0] + StoreF64::S;
  const double den = m + 2.0 * Ap * rho_l, iden = 1.0 / den;
  double rlb = 0.0, denb = 0.0, mb = 0.0, bb = 0.0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const double gbk = Ap * sums[threadIdx.x][1 + k], xsk = Ap * sums[threadIdx.x][1 + D + k];
    const double U = A.U[k * np + p], Un = A.Un[k * np + sl], Xb = A.Xb_in[k * np + sl];
    const double Ubt = A.Ub_in[k * np + sl] + Xb + 2.0 * rho_l * gbk;
    const double Nb = Ubt * iden;
    denb -= Nb * Un;
    rlb += 2.0 * gbk * Un;
    A.Ub_tmp[k * np + sl] = m * Nb;
    A.jlb[k * np + sl] = 2.0 * Ap * Nb - 2.0 * gbk;
    A.Fcb[k * np + sl] = Nb;
    mb += Nb * U;
    bb += Nb * A.ph.gravity[k];
    A.Xb_tmp[k * np + sl] = Xb + xsk;
  }
  mb += denb;
  A.rlb[sl] = rlb + 2.0 * Ap * denb;
  // m = rho_r V, b = m (1 - 1/rho_r) = V (rho_r - 1), V = m - b
  A.mb_tmp[sl] = (m - bu) * (mb + bb);
}

// 3. Contact and interpolation adjoint, per slot. Pair force f_ij = (k_n delta -
// gamma v_n) n with n = s / |s|, s = X_i - X_j, delta = r_i + r_j - |s|,
// v_n = (U_i - U_j).n, gamma = 2 beta sqrt(m_eff k_n); it enters F_c,i with + and
// F_c,j with -, so particle i takes the transposed Jacobian of f_ij applied to
// (Fcb_i - Fcb_j). Walls: F_k += -(+/-) ... as in the forward kernel.
// Interpolation rho_l = sum w rho(c), j_l = sum w j(c): the adjoint moments are
// spread into rjbar with the same weights, and the weight derivatives add to X.
// A particle's lanes share the neighbour rows of the contact search, then its
// stencil rows.
template <int D, int W>
__global__ void __launch_bounds__(AdjShape<D, W>::THREADS) k_adj_contact_interp(AdjArgs A) {
  using S = AdjShape<D, W>;
  __shared__ AdjTapsShared<D, W> sh;
  __shared__ unsigned sp[S::PPB];
  __shared__ double sums[S::PPB][2 * D + 1];  // X, U and mass adjoints
  const long long np = A.np;
  const Geometry& g = A.g;
  const BinMap& bm = A.bm;
  adj_block_particles<D, W>(A, sp);
  __syncthreads();
  adj_block_taps<D, W>(A, sp, sh);
  __syncthreads();
  const int qi = threadIdx.x / S::ROWS, row = threadIdx.x % S::ROWS;
  const long long slq = blockIdx.x * (long long)S::PPB + qi;
  const unsigned pq = sp[qi];
  double Xb[3] = {0.0, 0.0, 0.0}, Ub[3] = {0.0, 0.0, 0.0}, mb = 0.0;
  if (pq < (unsigned)np) {
    const int4 mc = A.cs[slq];
    const int bc[3] = {mc.x, mc.y, mc.z};
    const double r = A.rad[pq];
    constexpr int NR = D == 3 ? 9 : 3;  // neighbour rows of three cells along x
    for (int nr = row; nr < NR; nr += S::ROWS) {
      int cy = bc[1] + nr % 3 - 1, cz = D == 3 ? bc[2] + nr / 3 - 1 : 0;
      if (!lattice_coord(cy, g.n[1], g.periodic[1])) continue;
      if (D == 3 && !lattice_coord(cz, g.n[2], g.periodic[2])) continue;
      for (int ox = -1; ox <= 1; ++ox) {
        int cx = bc[0] + ox;
        if (!lattice_coord(cx, g.n[0], g.periodic[0])) continue;
        const unsigned b = bin_index<D>(bm, cx, cy, cz);
        const unsigned lo = A.start[b], hi = A.start[b + 1];
        if (hi > (unsigned)np || lo > hi) {
          atomicOr(A.err, ERR_INDEX);
          continue;
        }
        for (unsigned s2 = lo; s2 < hi; ++s2) {
          if (s2 == (unsigned)slq) continue;
          const unsigned q = (unsigned)A.cs[s2].w;
          if (q >= (unsigned)np) {
            atomicOr(A.err, ERR_INDEX);
            continue;
          }
          double s[3] = {0.0, 0.0, 0.0}, d2 = 0.0;
#pragma unroll
          for (int k = 0; k < D; ++k) {
            s[k] = min_image(A.X[k * np + pq] - A.X[k * np + q], g.n[k], g.periodic[k]);
            d2 += s[k] * s[k];
          }
          const double rs = r + A.rad[q];
          if (d2 > rs * rs * (1.0 + 1e-12)) continue;  // clear of each other: no square root
          const double dist = sqrt(d2);
          const double delta = rs - dist;
          if (!(delta > 0.0) || !(dist > 0.0)) continue;
          const double kn = A.ph.kn, beta = A.ph.beta;
          const double m = A.mass[pq], mq = A.mass[q];
          const double meff = m * mq / (m + mq);
          const double gam = 2.0 * beta * sqrt(meff * kn);
          double n[3] = {0.0, 0.0, 0.0}, dU[3] = {0.0, 0.0, 0.0}, vn = 0.0, an = 0.0;
          double av[3] = {0.0, 0.0, 0.0};
#pragma unroll
          for (int k = 0; k < D; ++k) {
            n[k] = s[k] / dist;
            dU[k] = A.U[k * np + pq] - A.U[k * np + q];
            vn += dU[k] * n[k];
            av[k] = A.Fcb[k * np + slq] - A.Fcb[k * np + s2];
            an += av[k] * n[k];
          }
          const double mag = kn * delta - gam * vn;
#pragma unroll
          for (int k = 0; k < D; ++k) {
            const double dmag = -kn * n[k] - gam * (dU[k] - vn * n[k]) / dist;
            Xb[k] += an * dmag + mag * (av[k] - an * n[k]) / dist;
            Ub[k] -= an * gam * n[k];
          }
          const double mqs = mq / (m + mq);
          mb -= an * vn * gam / (2.0 * meff) * mqs * mqs;
        }
      }
    }
    // interpolation adjoint of this lane's stencil row
    const TapsD<W>(&t)[D] = sh.t[qi];
    const int iy = row % W, iz = row / W;
    const double wy = t[1].w[iy], dwy = t[1].dw[iy];
    const double wz = D == 3 ? t[D - 1].w[iz] : 1.0, dwz = D == 3 ? t[D - 1].dw[iz] : 0.0;
    const long long r0 =
        (long long)g.n[0] * (t[1].idx[iy] + (long long)g.n[1] * (D == 3 ? t[D - 1].idx[iz] : 0));
    const double rlb = A.rlb[slq], wyz = wy * wz;
    double jlb[3] = {0.0, 0.0, 0.0}, amp[4] = {rlb * wyz, 0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < D; ++k) {
      jlb[k] = A.jlb[k * np + slq];
      amp[1 + k] = jlb[k] * wyz;
    }
    double V = 0.0, DV = 0.0;
#pragma unroll
    for (int ix = 0; ix < W; ++ix) {
      const long long c = r0 + t[0].idx[ix];
      const double* mcell = A.mom + 4 * c;
      double val = rlb * mcell[0];
#pragma unroll
      for (int k = 0; k < D; ++k) val += jlb[k] * mcell[1 + k];
      const double w = t[0].w[ix];
      V += w * val;
      DV += t[0].dw[ix] * val;
      if (w * wyz != 0.0) {
#pragma unroll
        for (int k = 0; k <= D; ++k) atomicAdd(A.rjbar + 4 * c + k, amp[k] * w);
      }
    }
    Xb[0] += wyz * DV;
    Xb[1] += dwy * wz * V;
    if constexpr (D == 3) Xb[2] += wy * dwz * V;
  }
  mb = row_sum<S::ROWS>(mb);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    Xb[k] = row_sum<S::ROWS>(Xb[k]);
    Ub[k] = row_sum<S::ROWS>(Ub[k]);
  }
  if (row == 0) {
    sums[qi][2 * D] = mb;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      sums[qi][k] = Xb[k];
      sums[qi][D + k] = Ub[k];
    }
  }
  __syncthreads();
  // --- walls and the sums, one thread per particle ---
  if (threadIdx.x >= S::PPB || sp[threadIdx.x] >= (unsigned)np) return;
  const unsigned p = sp[threadIdx.x];
  const long long sl = blockIdx.x * (long long)S::PPB + threadIdx.x;
  const double m = A.mass[p], r = A.rad[p], kn = A.ph.kn, gw = A.gw[p];
  mb = sums[threadIdx.x][2 * D];
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const double X = A.X[k * np + p], U = A.U[k * np + p], ai = A.Fcb[k * np + sl];
    double xb = A.Xb_tmp[k * np + sl] + sums[threadIdx.x][k];
    double ub = A.Ub_tmp[k * np + sl] + sums[threadIdx.x][D + k];
    if (!g.periodic[k]) {
      // wall at 0: F_k += k_n (r - X_k) - gw U_k; wall at n: F_k -= k_n (r - n + X_k) + gw U_k
      const bool lo = r - X > 0.0, hi = r - ((double)g.n[k] - X) > 0.0;
      const int cnt = (lo ? 1 : 0) + (hi ? 1 : 0);
      if (cnt) {
        xb -= cnt * kn * ai;
        ub -= cnt * gw * ai;
        mb -= cnt * ai * U * gw / (2.0 * m);
      }
    }
    A.Xb_out[k * np + p] = xb;
    A.Ub_out[k * np + p] = ub;
  }
  const unsigned user = A.pid[p];
  if (user >= (unsigned)np) {
    atomicOr(A.err, ERR_INDEX);
    return;
  }
  A.drho[user] += (m - A.buoy[p]) * mb + A.mb_tmp[sl];
}

// 4. The interpolation's moment adjoint: fb_a += rho_bar + e_a.j_bar at the cells a
// stencil reached (all in busy tiles), clearing the field for the next step.
template <int Q>
__global__ void __launch_bounds__(256) k_adj_moments(Geometry g, BinMap bm,
                                                     const int* __restrict__ tbusy,
                                                     const unsigned* __restrict__ tn,
                                                     double* __restrict__ rjbar,
                                                     double* __restrict__ fbar) {
  using L = Lattice<Q>;
  constexpr int D = L::D;
  using TD = TileDims<D>;
  constexpr int PER = TD::TC / 256;  // CTAs per tile
  const unsigned i = blockIdx.x / PER;
  if (i >= tn[0]) return;
  const int lin = (int)(blockIdx.x % PER) * 256 + (int)threadIdx.x;
  const int t = tbusy[i], r = t / bm.nt[0];
  const int x = (t - r * bm.nt[0]) * TD::TX + lin % TD::TX;
  const int y = (r % bm.nt[1]) * TD::TY + (lin / TD::TX) % TD::TY;
  const int z = (r / bm.nt[1]) * TD::TZ + lin / (TD::TX * TD::TY);
  if (x >= g.n[0] || y >= g.n[1] || z >= g.n[2]) return;
  const long long c = x + (long long)g.n[0] * (y + (long long)g.n[1] * z);
  double2* rj = reinterpret_cast<double2*>(rjbar) + 2 * c;
  const double2 lo = rj[0], hi = rj[1];
  const double rho = lo.x, j[3] = {lo.y, hi.x, hi.y};
  if (rho == 0.0 && j[0] == 0.0 && j[1] == 0.0 && j[2] == 0.0) return;
  rj[0] = make_double2(0.0, 0.0);
  rj[1] = make_double2(0.0, 0.0);
  const long long P = g.pitch;
  fbar[c] += rho;
#pragma unroll
  for (int a = 1; a < Q; a += 2) {
    double ej = 0.0;
    bool first = true;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      if (L::e(a, k) == 0) continue;
      const double v = L::e(a, k) > 0 ? j[k] : -j[k];
      ej = first ? v : ej + v;
      first = false;
    }
    fbar[a * P + c] += rho + ej;
    fbar[(a + 1) * P + c] += rho - ej;
  }
}

__global__ void k_adj_seed(long long np, int d, double* __restrict__ Ub) {
  const long long i = blockIdx.x * (long long)ADJ_THREADS + threadIdx.x;
  if (i < np) Ub[(long long)(d - 1) * np + i] = 1.0 / (double)np;
}

__global__ void k_mean_last(long long np, int d, const double* __restrict__ U,
                            double* __restrict__ out) {
  __shared__ double red[ADJ_THREADS];
  double s = 0.0;
  for (long long i = threadIdx.x; i < np; i += ADJ_THREADS) s += U[(long long)(d - 1) * np + i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int k = ADJ_THREADS / 2; k > 0; k >>= 1) {
    if ((int)threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = red[0] / (double)np;
}

__global__ void k_sum_blocks(long long n, const double* __restrict__ in, double* __restrict__ out) {
  __shared__ double red[ADJ_THREADS];
  double s = 0.0;
  for (long long i = threadIdx.x; i < n; i += ADJ_THREADS) s += in[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int k = ADJ_THREADS / 2; k > 0; k >>= 1) {
    if ((int)threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = red[0];
}

unsigned cell_blocks(long long n) { return (unsigned)((n + ADJ_CELLS - 1) / ADJ_CELLS); }

unsigned nblk(long long n) { return (unsigned)((n + ADJ_THREADS - 1) / ADJ_THREADS); }

template <typename T>
T* rebase(T* p, const char* from, char* to) {
  return p ? (T*)(to + ((const char*)p - from)) : nullptr;
}

// A copy of the state whose pointers address the tape copy of the workspace.
State rebase_state(const State& s, const void* ws, void* tape) {
  const char* a = (const char*)ws;
  char* b = (char*)tape;
  State t = s;
  for (int i = 0; i < 2; ++i) t.f[i] = rebase((char*)s.f[i], a, b);
  t.F = rebase((char*)s.F, a, b);
  t.mom = rebase((char*)s.mom, a, b);
  t.red = rebase(s.red, a, b);
  t.err = rebase(s.err, a, b);
  Particles& P = t.p;
  const Particles& Q = s.p;
  for (int i = 0; i < 2; ++i) {
    P.X[i] = rebase(Q.X[i], a, b);
    P.U[i] = rebase(Q.U[i], a, b);
    P.rad[i] = rebase(Q.rad[i], a, b);
    P.mass[i] = rebase(Q.mass[i], a, b);
    P.Ap[i] = rebase(Q.Ap[i], a, b);
    P.buoy[i] = rebase(Q.buoy[i], a, b);
    P.gw[i] = rebase(Q.gw[i], a, b);
    P.cf[i] = rebase(Q.cf[i], a, b);
    P.pid[i] = rebase(Q.pid[i], a, b);
  }
  P.xr = rebase(Q.xr, a, b);
  P.cr = rebase(Q.cr, a, b);
  for (int i = 0; i < 2; ++i) {
    P.xs[i] = rebase(Q.xs[i], a, b);
    P.cs[i] = rebase(Q.cs[i], a, b);
  }
  P.g = rebase(Q.g, a, b);
  P.Fc = rebase(Q.Fc, a, b);
  P.rl = rebase(Q.rl, a, b);
  P.jl = rebase(Q.jl, a, b);
  P.Fs = rebase(Q.Fs, a, b);
  P.key = rebase(Q.key, a, b);
  P.rank = rebase(Q.rank, a, b);
  P.bin_cnt = rebase(Q.bin_cnt, a, b);
  P.perm = rebase(Q.perm, a, b);
  P.block_sums = rebase(Q.block_sums, a, b);
  P.tf = rebase(Q.tf, a, b);
  P.tr = rebase((char*)Q.tr, a, b);
  P.tbusy = rebase(Q.tbusy, a, b);
  P.tn = rebase(Q.tn, a, b);
  return t;
}

// The adjoint of one step: fnext (adjoint of the post-stream populations of the
// step after it) -> fbar (of this step's); rjbar is zero on entry and on return.
template <int Q, int W>
cudaError_t adjoint_step(const State& T, AdjArgs A, const double* fnext, double* fbar,
                         double* Fbar, double* om_part, cudaStream_t st) {
  constexpr int D = Lattice<Q>::D;
  using S = AdjShape<D, W>;
  const Geometry& g = T.geo;
  const int cur = T.cur, nxt = 1 - T.cur;
  A.X = T.p.X[cur];
  A.U = T.p.U[cur];
  A.Un = T.p.U[nxt];
  A.gin = T.p.g;
  A.mass = T.p.mass[cur];
  A.Ap = T.p.Ap[cur];
  A.buoy = T.p.buoy[cur];
  A.rad = T.p.rad[cur];
  A.gw = T.p.gw[cur];
  A.pid = T.p.pid[cur];
  A.cs = T.p.cs[cur];
  A.start = T.p.bin_cnt;
  A.tf = T.p.tf;
  A.tr = (const double*)T.p.tr;
  A.mom = (const double*)T.mom;
  k_adj_collide<Q><<<cell_blocks(g.ncell), ADJ_CELLS, 0, st>>>(
      g, T.phy.omega, T.phy.cF, (const double*)T.f[cur], (const double*)T.F, fnext, fbar, Fbar,
      om_part);
  const unsigned pb = (unsigned)((A.np + S::PPB - 1) / S::PPB);
  k_adj_update<D, W><<<pb, S::THREADS, 0, st>>>(A);
  k_adj_contact_interp<D, W><<<pb, S::THREADS, 0, st>>>(A);
  k_adj_moments<Q><<<(unsigned)(T.p.ntiles * (TileDims<D>::TC / 256)), 256, 0, st>>>(
      g, A.bm, T.p.tbusy, T.p.tn, A.rjbar, fbar);
  return cudaGetLastError();
}

template <int Q>
cudaError_t adjoint_step_w(const State& T, const AdjArgs& A, const double* fnext, double* fbar,
                           double* Fbar, double* om_part, cudaStream_t st) {
  return T.phy.width == 2 ? adjoint_step<Q, 2>(T, A, fnext, fbar, Fbar, om_part, st)
                          : adjoint_step<Q, 4>(T, A, fnext, fbar, Fbar, om_part, st);
}

// One device allocation for everything a gradient run needs, laid out by walking the
// same list of arrays twice: once to add up the bytes, once for the pointers.
struct Arena {
  char* base = nullptr;
  size_t bytes = 0;
  bool counting = true;
  ~Arena() {
    if (base) cudaFree(base);
  }
  template <typename T>
  T* take(size_t n) {
    T* p = counting ? nullptr : (T*)(base + bytes);
    bytes += (n + 255) / 256 * 256;
    return p;
  }
  bool allocate() {
    if (cudaMalloc(&base, bytes ? bytes : 256) != cudaSuccess) {
      cudaGetLastError();
      base = nullptr;
      return false;
    }
    counting = false;
    bytes = 0;
    return true;
  }
};

// CUDA graphs of the recurring stretches (forward, replay, reverse), by the parity they
// start from.
struct StretchGraphs {
  cudaStream_t cap = nullptr;
  cudaGraphExec_t exec[3][2] = {};
  ~StretchGraphs() {
    for (auto& k : exec)
      for (cudaGraphExec_t e : k)
        if (e) cudaGraphExecDestroy(e);
    if (cap) cudaStreamDestroy(cap);
  }
};

struct HandleGuard {
  pibm_t* h = nullptr;
  ~HandleGuard() {
    if (h) pibm_destroy(h);
  }
};

}  // namespace

int settling_gradient(const pibm_config* cfg_in, int64_t nsteps, int64_t K, void* stream,
                      double* loss, double* dtau, double* drho, double* dx0) {
  if (!cfg_in || nsteps < 1 || K < 1 || !loss) return PIBM_EINVAL;
  if (cfg_in->n_particles < 1) return PIBM_EINVAL;
  if (cfg_in->precision != PIBM_FP64 || cfg_in->coupling != PIBM_IMPLICIT ||
      cfg_in->interp != PIBM_INTERP_DELTA || cfg_in->dem_model != PIBM_DEM_LINEAR ||
      cfg_in->dem_substeps > 1 || cfg_in->rebin_every > 1)
    return PIBM_ENOTSUP;
  pibm_config cfg = *cfg_in;
  cfg.deterministic = 1;  // replayed stretches reproduce the forward run bit for bit
  cudaStream_t st = (cudaStream_t)stream;
  size_t wsb = 0;
  int rc = pibm_workspace_bytes(&cfg, &wsb);
  if (rc != PIBM_OK) return rc;
  const bool grads = dtau || drho || dx0;
  const int d = cfg.lattice == PIBM_D2Q9 ? 2 : 3, q = cfg.lattice, FS = d == 2 ? 2 : 4;
  const long long np = cfg.n_particles, ncell = cfg.n[0] * cfg.n[1] * cfg.n[2];
  const long long P = (ncell + 63) / 64 * 64;  // the plane pitch
  const long long nseg = (nsteps + K - 1) / K;
  const size_t D8 = sizeof(double);

  Arena al;
  char *ws, *ckpt = nullptr, *tape = nullptr;
  double *scal, *fb[2], *Fbar, *rjbar, *om_part, *pb[2][2], *Xb_tmp, *Ub_tmp, *Fcb, *rlb, *jlb,
      *mb_tmp, *drho_d;
  for (int pass = 0; pass < 2; ++pass) {
    ws = al.take<char>(wsb);
    scal = al.take<double>(D8 * 4);
    if (grads) {
      // checkpoints, the tape of one stretch, and the adjoint state: of the post-stream
      // populations (of the step after and of this one), the force, the moment field
      // and the particles
      ckpt = al.take<char>(wsb * (size_t)(nseg - 1));
      tape = al.take<char>(wsb * (size_t)std::min<int64_t>(K, nsteps));
      for (int i = 0; i < 2; ++i) {
        fb[i] = al.take<double>(D8 * q * P);
        for (int j = 0; j < 2; ++j) pb[i][j] = al.take<double>(D8 * d * np);
      }
      Fbar = al.take<double>(D8 * FS * P);
      rjbar = al.take<double>(D8 * 4 * P);
      om_part = al.take<double>(D8 * cell_blocks(ncell));
      Xb_tmp = al.take<double>(D8 * d * np);
      Ub_tmp = al.take<double>(D8 * d * np);
      Fcb = al.take<double>(D8 * d * np);
      rlb = al.take<double>(D8 * np);
      jlb = al.take<double>(D8 * d * np);
      mb_tmp = al.take<double>(D8 * np);
      drho_d = al.take<double>(D8 * np);
    }
    if (pass == 0 && !al.allocate()) return PIBM_ENOMEM;
  }
  HandleGuard hg;  // destroyed before the arena
  rc = pibm_create(&cfg, ws, wsb, stream, &hg.h);
  if (rc != PIBM_OK) return rc;
  HandleView v = handle_view(hg.h);
  State& s = *v.s;

  // A copy of the workspace without the partner population buffer, which holds nothing
  // between steps and is not read by a step's adjoint. The two buffers open the
  // workspace, so the rest is one range behind the second.
  auto copy_state = [&](char* to, const char* from, cudaStream_t st) -> cudaError_t {
    const char* ws = (const char*)v.ws;
    const size_t f0 = (const char*)s.f[0] - ws, f1 = (const char*)s.f[1] - ws;
    const size_t rest = (const char*)s.F - ws;
    const size_t lo = s.cur == 0 ? f0 : f1, hi = s.cur == 0 ? f1 : wsb;
    cudaError_t e = cudaMemcpyAsync(to + lo, from + lo, hi - lo, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess && s.cur == 0)
      e = cudaMemcpyAsync(to + rest, from + rest, wsb - rest, cudaMemcpyDeviceToDevice, st);
    return e;
  };
  auto fwd_step = [&](char* tape_slot, cudaStream_t st) -> cudaError_t {
    cudaError_t e;
    if ((e = launch_bin(s, st, nullptr)) != cudaSuccess) return e;
    if ((e = launch_contacts(s, st, nullptr)) != cudaSuccess) return e;
    if ((e = launch_couple(s, st, nullptr)) != cudaSuccess) return e;
    if (tape_slot && (e = copy_state(tape_slot, (const char*)v.ws, st)) != cudaSuccess) return e;
    if ((e = launch_collide_stream(s, st, true)) != cudaSuccess) return e;
    s.cur ^= 1;
    return cudaSuccess;
  };
  int io = 0;  // pb[io], fb[io] = adjoint of the state being reversed into
  // n forward steps, taped or not
  auto forward = [&](long long n, bool taped, cudaStream_t st) -> cudaError_t {
    for (long long i = 0; i < n; ++i) {
      const cudaError_t e = fwd_step(taped ? tape + wsb * i : nullptr, st);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  };
  AdjArgs A{};
  // the adjoint of the n steps on the tape, whose first started from buffer par
  auto reverse = [&](long long n, int par, cudaStream_t st) -> cudaError_t {
    for (long long i = n - 1; i >= 0; --i) {
      State T = rebase_state(s, v.ws, tape + wsb * i);
      T.cur = par ^ (int)(i & 1);
      A.Xb_in = pb[io][0];
      A.Ub_in = pb[io][1];
      A.Xb_out = pb[1 - io][0];
      A.Ub_out = pb[1 - io][1];
      cudaError_t e = cudaErrorInvalidValue;
      if (q == 9) e = adjoint_step_w<9>(T, A, fb[io], fb[1 - io], Fbar, om_part, st);
      else if (q == 15) e = adjoint_step_w<15>(T, A, fb[io], fb[1 - io], Fbar, om_part, st);
      else if (q == 19) e = adjoint_step_w<19>(T, A, fb[io], fb[1 - io], Fbar, om_part, st);
      if (e != cudaSuccess) return e;
      io = 1 - io;
    }
    return cudaSuccess;
  };
  // Full stretches recur with the same arguments (up to the buffer parity they start
  // from), so in runs of four stretches or more they are captured once and replayed: a
  // step of a small lattice is 13 launches of a few microseconds each, and launching them
  // one by one took longer than running them (72 x 60, 120 steps: 23.3 ms for 14.9 ms of
  // kernels).
  StretchGraphs graphs;
  bool replayed = grads && nseg >= 4 && K <= 64 &&
                  make_capture_stream(&graphs.cap);
  // body(stream) enqueues stretch kind kd of K steps starting from parity key; the host
  // state it advances is s.cur (forward kinds) or io (reverse)
  auto stretch = [&](int kd, int key, auto&& body) -> cudaError_t {
    if (!replayed) return body(st);
    int& moved = kd == 2 ? io : s.cur;
    const int before = moved;
    cudaGraphExec_t& ex = graphs.exec[kd][key];
    if (!ex) {
      cudaGraph_t gr = nullptr;
      cudaError_t e = cudaStreamBeginCapture(graphs.cap, cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) {
        e = body(graphs.cap);
        const cudaError_t ee = cudaStreamEndCapture(graphs.cap, &gr);
        if (e == cudaSuccess) e = ee;
      }
      if (e == cudaSuccess) e = cudaGraphInstantiate(&ex, gr, 0);
      if (gr) cudaGraphDestroy(gr);
      moved = before;
      if (e != cudaSuccess) {  // not capturable here: launch directly from now on
        cudaGetLastError();
        ex = nullptr;
        replayed = false;
        return body(st);
      }
    }
    moved = before ^ (int)(K & 1);
    return cudaGraphLaunch(ex, st);
  };

  // forward sweep with checkpoints; the last stretch, which the reverse sweep starts
  // with, keeps its tape at once
  std::vector<int> par(nseg);
  for (long long sg = 0; sg < nseg; ++sg) {
    par[sg] = s.cur;
    const bool last = sg == nseg - 1;
    const long long n = last ? nsteps - sg * K : K;
    cudaError_t e;
    if (last) {
      e = forward(n, grads, st);
    } else {
      e = grads ? copy_state(ckpt + wsb * sg, (const char*)v.ws, st) : cudaSuccess;
      if (e == cudaSuccess)
        e = stretch(0, s.cur, [&](cudaStream_t to) { return forward(n, false, to); });
    }
    if (e != cudaSuccess) return PIBM_ECUDA;
  }
  k_mean_last<<<1, ADJ_THREADS, 0, st>>>(np, d, s.p.U[s.cur], scal);
  if (cudaMemcpyAsync(loss, scal, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return PIBM_ECUDA;
  rc = pibm_status(hg.h);
  if (rc != PIBM_OK || !grads) return rc;

  // adjoint of the final state: d loss / d U_last = 1 / np
  if (cudaMemsetAsync(fb[io], 0, sizeof(double) * q * P, st) != cudaSuccess ||
      cudaMemsetAsync(rjbar, 0, sizeof(double) * 4 * P, st) != cudaSuccess ||
      cudaMemsetAsync(pb[io][0], 0, sizeof(double) * d * np, st) != cudaSuccess ||
      cudaMemsetAsync(pb[io][1], 0, sizeof(double) * d * np, st) != cudaSuccess ||
      cudaMemsetAsync(om_part, 0, sizeof(double) * cell_blocks(ncell), st) != cudaSuccess ||
      cudaMemsetAsync(drho_d, 0, sizeof(double) * np, st) != cudaSuccess)
    return PIBM_ECUDA;
  k_adj_seed<<<nblk(np), ADJ_THREADS, 0, st>>>(np, d, pb[io][1]);

  A.g = s.geo;
  A.ph = s.phy;
  A.bm = s.p.bm;
  A.np = np;
  A.Fbar = Fbar;
  A.Xb_tmp = Xb_tmp;
  A.Ub_tmp = Ub_tmp;
  A.Fcb = Fcb;
  A.rlb = rlb;
  A.jlb = jlb;
  A.mb_tmp = mb_tmp;
  A.rjbar = rjbar;
  A.drho = drho_d;
  A.err = s.err;
  for (long long sg = nseg - 1; sg >= 0; --sg) {
    const bool last = sg == nseg - 1;
    const long long n = last ? nsteps - sg * K : K;
    cudaError_t e = cudaSuccess;
    if (!last) {
      // replay the stretch from its checkpoint, keeping the tape
      s.cur = par[sg];
      e = copy_state((char*)v.ws, ckpt + wsb * sg, st);
      if (e == cudaSuccess)
        e = stretch(1, par[sg], [&](cudaStream_t to) { return forward(n, true, to); });
    }
    // the adjoint buffers alternate with the tape's parity (both flip with every step
    // from the last one back), so that parity is the whole key of a reverse stretch
    if (e == cudaSuccess) {
      if (n == K) e = stretch(2, par[sg], [&](cudaStream_t to) { return reverse(n, par[sg], to); });
      else e = reverse(n, par[sg], st);
    }
    if (e != cudaSuccess) return PIBM_ECUDA;
  }
  k_sum_blocks<<<1, ADJ_THREADS, 0, st>>>(cell_blocks(ncell), om_part, scal + 1);
  double omb = 0.0;
  if (cudaMemcpyAsync(&omb, scal + 1, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return PIBM_ECUDA;
  // the initial storage order is the user order
  std::vector<double> xb((size_t)d * np);
  if (dx0 && cudaMemcpyAsync(xb.data(), pb[io][0], sizeof(double) * d * np,
                             cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return PIBM_ECUDA;
  if (drho && cudaMemcpyAsync(drho, drho_d, sizeof(double) * np, cudaMemcpyDeviceToHost, st) !=
                  cudaSuccess)
    return PIBM_ECUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return PIBM_ECUDA;
  if (dx0)
    for (long long i = 0; i < np; ++i)
      for (int k = 0; k < d; ++k) dx0[i * d + k] = xb[(size_t)k * np + i];
  // om = 1 / tau
  if (dtau) *dtau = -omb / (cfg.tau * cfg.tau);
  return pibm_status(hg.h);
}

}  // namespace pibm

extern "C" int pibm_settling_gradient(const pibm_config* cfg, int64_t nsteps,
                                      int64_t checkpoint_every, void* stream, double* loss,
                                      double* dtau, double* drho, double* dx0) {
  return pibm::settling_gradient(cfg, nsteps, checkpoint_every, stream, loss, dtau, drho, dx0);
}
