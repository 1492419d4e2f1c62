// Ordered spreading in 3D: the strips against the per-cell form, bit for bit, and both
// against the sum over the particles in FP64 on the host, on synthetic stencil records.
// Lattices whose strips wrap in x, y and z, end at walls, or meet partial tiles.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "particles_device.cuh"

using namespace pibm;

namespace {

unsigned long long seed_ = 1;
double uniform() {  // splitmix64
  unsigned long long x = (seed_ += 0x9e3779b97f4a7c15ull);
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return (double)((x ^ (x >> 31)) >> 11) * 0x1p-53;
}

void check(cudaError_t e) {
  if (e != cudaSuccess) {
    printf("%s\n", cudaGetErrorString(e));
    exit(2);
  }
}

template <typename T>
struct Dev {
  T* p = nullptr;
  explicit Dev(const std::vector<T>& v) {
    check(cudaMalloc(&p, sizeof(T) * v.size()));
    check(cudaMemcpy(p, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice));
  }
  ~Dev() { cudaFree(p); }
};

// W nodes, search reach RE cells (one more than the stencil's with a kept cell list, whose
// particles lie within half a cell of their bin).
template <int W, int RE, typename FT>
int run(const int (&n)[3], int wrap) {
  using TD = TileDims<3>;
  using S = StripShape<W, RE>;
  Geometry g{};
  g.q = 19;
  g.d = 3;
  g.ncell = 1;
  BinMap bm{};
  const int T[3] = {TD::TX, TD::TY, TD::TZ};
  for (int k = 0; k < 3; ++k) {
    g.n[k] = n[k];
    g.periodic[k] = wrap >> k & 1;
    g.ncell *= n[k];
    bm.T[k] = T[k];
    bm.nt[k] = (n[k] + T[k] - 1) / T[k];
  }
  bm.tc = TD::TC;
  g.pitch = (g.ncell + 63) / 64 * 64;
  if (!strips_fit<W, RE>(g)) return 0;
  const int ntiles = bm.nt[0] * bm.nt[1] * bm.nt[2], nbin = ntiles * bm.tc;
  const bool kept = RE > W / 2;
  const long long np = g.ncell * 3 / 5 + 1;
  struct P {
    int bin;
    int4 first;
    FT r[TAP_RECORD];
  };
  std::vector<P> ps(np);
  std::vector<double> want(g.ncell * 3, 0.0);
  for (P& p : ps) {
    int c[3], f[3];
    for (int i = 0; i < TAP_RECORD; ++i) p.r[i] = FT(0);
    for (int k = 0; k < 3; ++k) {
      c[k] = (int)(uniform() * n[k]);
      double x = c[k] + (kept ? 2.0 * uniform() - 0.5 : uniform());
      if (!g.periodic[k]) x = std::fmin(std::fmax(x, 0.0), n[k] - 1e-9);
      // FP64 takes the taps of the wrapped position, FP32 those beside the bin
      else if (sizeof(FT) == 8) x -= n[k] * std::floor(x / n[k]);
      f[k] = (int)std::floor(x - 0.5) - (W / 2 - 1);
      for (int i = 0; i < W; ++i) {
        const bool out = f[k] + i < 0 || f[k] + i >= n[k];
        p.r[4 * k + i] = out && !g.periodic[k] ? FT(0) : FT(0.05 + uniform());
      }
      p.r[12 + k] = FT(uniform() - 0.5);
    }
    const int t = c[0] / T[0] + bm.nt[0] * (c[1] / T[1] + bm.nt[1] * (c[2] / T[2]));
    p.bin = t * bm.tc + c[0] % T[0] + T[0] * (c[1] % T[1] + T[1] * (c[2] % T[2]));
    p.first = make_int4(f[0], f[1], f[2], 0);
    for (int i = 0; i < W * W * W; ++i) {
      const int o[3] = {i % W, i / W % W, i / (W * W)};
      long long cell = 0;
      double w = 1.0;
      for (int k = 2; k >= 0; --k) {
        cell = cell * n[k] + ((f[k] + o[k]) % n[k] + n[k]) % n[k];
        w *= (double)p.r[4 * k + o[k]];
      }
      if (w != 0.0)
        for (int k = 0; k < 3; ++k) want[3 * cell + k] += w * (double)p.r[12 + k];
    }
  }
  std::vector<unsigned> start(nbin + 1, 0u);
  for (const P& p : ps) ++start[p.bin + 1];
  for (int b = 0; b < nbin; ++b) start[b + 1] += start[b];
  std::vector<unsigned> at(start.begin(), start.end() - 1);
  std::vector<int4> tf(np);
  std::vector<FT> tr(np * TAP_RECORD);
  for (const P& p : ps) {
    const unsigned sl = at[p.bin]++;
    tf[sl] = p.first;
    memcpy(&tr[(size_t)sl * TAP_RECORD], p.r, sizeof(p.r));
  }
  std::vector<int> tbusy(ntiles);
  for (int t = 0; t < ntiles; ++t) tbusy[t] = ntiles - 1 - t;
  const std::vector<unsigned> tn = {(unsigned)ntiles, 0u}, none = {0u};
  const size_t stride = FieldStride<3>::F;
  const std::vector<FT> zero(g.pitch * stride, FT(0));
  Dev<unsigned> dstart(start), dtn(tn), err(none);
  Dev<int> dtbusy(tbusy);
  Dev<int4> dtf(tf);
  Dev<FT> dtr(tr), strips(zero), cells(zero);
  k_spread_strips<W, RE, FT><<<ntiles * (S::PER_TILE / S::WARPS), S::WARPS * 32>>>(
      g, bm, np, dtbusy.p, dtn.p, dtf.p, dtr.p, dstart.p, strips.p, err.p);
  check(cudaGetLastError());
  k_spread_gather<3, W, RE, FT>
      <<<ntiles, TD::TC>>>(g, bm, dtbusy.p, dtn.p, dtf.p, dtr.p, dstart.p, cells.p);
  check(cudaGetLastError());
  check(cudaDeviceSynchronize());
  std::vector<FT> a(zero), b(zero);
  unsigned e = 0;
  check(cudaMemcpy(a.data(), strips.p, sizeof(FT) * a.size(), cudaMemcpyDeviceToHost));
  check(cudaMemcpy(b.data(), cells.p, sizeof(FT) * b.size(), cudaMemcpyDeviceToHost));
  check(cudaMemcpy(&e, err.p, sizeof(e), cudaMemcpyDeviceToHost));
  double off = 0.0, top = 0.0;
  for (long long c = 0; c < g.ncell; ++c)
    for (int k = 0; k < 3; ++k) {
      off = std::fmax(off, std::fabs((double)b[stride * c + k] - want[3 * c + k]));
      top = std::fmax(top, std::fabs(want[3 * c + k]));
    }
  const bool same = memcmp(a.data(), b.data(), sizeof(FT) * a.size()) == 0;
  // at most about 100 terms a cell, each at most about the largest sum and in as many
  // rounded additions
  const bool near = off <= 10000 * (sizeof(FT) == 8 ? 0x1p-53 : 0x1p-24) * top && top > 0.0;
  if (!same || !near || e)
    printf("W %d reach %d %s %d x %d x %d periodic %d: %s, off %.2g, err %u\n", W, RE,
           sizeof(FT) == 8 ? "FP64" : "FP32", n[0], n[1], n[2], wrap,
           same ? "equal" : "NOT EQUAL", off / top, e);
  return same && near && !e ? 1 : -1000000;
}

}  // namespace

int main() {
  const int sizes[][3] = {{22, 14, 7}, {23, 15, 9}, {37, 17, 7}, {32, 16, 8}, {33, 31, 10},
                          {16, 8, 4},  {17, 9, 5},  {5, 3, 2},   {1, 40, 1}};
  int ran = 0;
  for (const auto& n : sizes)
    for (int wrap = 0; wrap < 8; ++wrap) {
      ran += run<2, 1, double>(n, wrap) + run<2, 2, double>(n, wrap);
      ran += run<4, 2, double>(n, wrap) + run<4, 3, double>(n, wrap);
      ran += run<2, 1, float>(n, wrap) + run<2, 2, float>(n, wrap);
      ran += run<4, 2, float>(n, wrap) + run<4, 3, float>(n, wrap);
    }
  printf("%d lattices\n", ran);
  return ran > 0 ? 0 : 1;
}
