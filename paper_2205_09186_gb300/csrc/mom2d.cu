// Launchers of the D2Q9 moment steps (mom2d.cuh) for single lattices.
#include <algorithm>

#include "launch.cuh"
#include "mom2d.cuh"

namespace lbmd {

namespace {

template <int S, bool FINAL>
__global__ void __launch_bounds__(T2NT, T2_CTAS) k_mom2(const KParams p, const Mom2Geo g, const float* rin, const float* jin,
                                                  float* rout, float* jout, float* fout, unsigned long long* bad,
                                                  long long t) {
  extern __shared__ __align__(16) float sm_mom2[];
  const int x0 = blockIdx.x * g.TW, y0 = blockIdx.y * g.TH;
  pdl_wait();
  mom2_tile<S, FINAL>(p, g.LX, g.P, rin, jin, rout, jout, fout, bad, t, x0, y0, min(g.TW, p.nx - x0),
                      min(g.TH, p.ny - y0), sm_mom2);
}

// a warp gathers one row of a tile
__global__ void __launch_bounds__(256) k_mom2_gather(const KParams p, const Mom2Geo g, const float* f, const float* rho,
                                                     float* rout, float* jout, unsigned long long* bad, long long t) {
  const int y = blockIdx.y * 8 + (threadIdx.x >> 5);
  if (y >= p.ny) return;
  const int x0 = blockIdx.x * g.TW;
  mom2_gather(p, g.LX, g.P, f, rho, rout, jout, bad, t, x0, min(g.TW, p.nx - x0), y, y + 1);
}

template <int S>
cudaError_t steps(const Launch& c, long long n) {
  const KParams& kp = c.kp;
  const Mom2Geo g = mom2_geo(kp, device_sms());
  if (cudaError_t e = ensure_smem(k_mom2<S, false>, T2_SMEM); e != cudaSuccess) return e;
  if (cudaError_t e = ensure_smem(k_mom2<S, true>, T2_SMEM); e != cudaSuccess) return e;
  float* s = static_cast<float*>(c.fout);  // scratch: rho x 2, j x 2
  float* r[2] = {s, s + g.P};
  float* j[2] = {s + 2 * g.P, s + 4 * g.P};
  float* f = const_cast<float*>(static_cast<const float*>(c.fin));
  float* rho = const_cast<float*>(static_cast<const float*>(c.rin));
  k_mom2_gather<<<dim3(g.nt, (kp.ny + 7) / 8), 256, 0, c.stream>>>(kp, g, f, rho, r[0], j[0], c.aux.bad_step, c.aux.t);
  const dim3 grid(g.nt, g.nr);
  for (long long k = 0; k < n; ++k) {
    const int a = int(k & 1);
    const cudaError_t e =
        k + 1 < n ? launch_pdl(k_mom2<S, false>, grid, T2NT, T2_SMEM, c.stream, kp, g, r[a], j[a], r[a ^ 1], j[a ^ 1], nullptr,
                               c.aux.bad_step, c.aux.t + k)
                  : launch_pdl(k_mom2<S, true>, grid, T2NT, T2_SMEM, c.stream, kp, g, r[a], j[a], rho, nullptr, f,
                               c.aux.bad_step, c.aux.t + k);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace

// Tiles evenly cut: the fewest across, and as many rows as make the tiles of an
// SM end together: a tile costs its rows and eight more; an SM with one tile takes
// twice, with two 1.3 times what the arithmetic alone would (three run at a time
// and cover each other's waits).  512^2 EFDS6, us a step by rows: 8 7.7, 12 6.8, 15
// 7.6, 20 8.4, 29 10.4.
Mom2Geo mom2_geo(const KParams& kp, int sms) {
  Mom2Geo g{};
  g.LX = (kp.nx + 3) / 4 * 4 + 16;
  g.P = (g.LX * kp.ny + 3) / 4 * 4;
  const int nt = (kp.nx + T2W - 1) / T2W;
  g.TW = ((kp.nx + nt - 1) / nt + 3) / 4 * 4;
  g.nt = (kp.nx + g.TW - 1) / g.TW;
  double best = 1e300;
  // (each height once, the tallest first: a call of two steps on a long lattice is not
  // to wait for the search)
  for (int most = std::min(T2H, kp.ny); most > 0; --most) {
    const int nr = (kp.ny + most - 1) / most, th = (kp.ny + nr - 1) / nr, rows = (kp.ny + th - 1) / th;
    if (th < 8 && best < 1e300) break;
    const long long tiles = (long long)g.nt * rows;
    const long long k = (tiles + sms - 1) / sms;
    const double cost = double(k) * (k == 1 ? 2.0 : (k == 2 ? 1.3 : 1.0)) * (th + 8);
    if (cost < best - 1e-9) { best = cost; g.TH = th; g.nr = rows; }
  }
  return g;
}

bool mom2d_ok(const KParams& kp, int scheme, int prec, bool mrt) {
  if (prec != 1 || mrt || kp.omega != 1.0) return false;
  if (scheme != S_EFDS2 && scheme != S_EFDS4 && scheme != S_EFDS6 && scheme != S_E4 && scheme != S_E8) return false;
  const long long LX = (kp.nx + 3) / 4 * 4 + 16, P = (LX * kp.ny + 3) / 4 * 4;
  return 6 * P <= 9 * kp.n && 9 * kp.n < (1LL << 31) && kp.ny <= 8LL * 65535;
}

cudaError_t mom2d_steps(const Launch& c, int scheme, long long n) {
  switch (scheme) {
    case S_EFDS2: return steps<S_EFDS2>(c, n);
    case S_EFDS4: return steps<S_EFDS4>(c, n);
    case S_EFDS6: return steps<S_EFDS6>(c, n);
    case S_E4: return steps<S_E4>(c, n);
    case S_E8: return steps<S_E8>(c, n);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace lbmd
