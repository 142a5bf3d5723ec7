// Launchers of the moment steps (mom3d.cuh): D3Q19, FP32 deviations, tau = 1,
// explicit line schemes and (with the accelerations of iir.cuh) compact ones.
#include <algorithm>

#include "iir.cuh"
#include "launch.cuh"
#include "mom3d.cuh"

namespace lbmd {

namespace {

constexpr int MW3 = 16;  // warps of a CTA, one CTA per SM

// columns per tile: the fewest tiles of at most 64 columns, evenly cut, none
// narrower than four columns (a row's two edge nodes then lie in two lanes)
MomGeo mom_geo(const KParams& kp) {
  MomGeo g{};
  g.LX = (kp.nx + 3) / 4 * 4 + 8;
  g.PL = g.LX * kp.ny;
  g.P = (g.PL * kp.nz + 63) / 64 * 64;
  const int nt = (kp.nx + 63) / 64;
  g.TW = ((kp.nx + nt - 1) / nt + 3) / 4 * 4;
  while (kp.nx % g.TW != 0 && kp.nx % g.TW < 4) g.TW -= 4;
  g.nt = (kp.nx + g.TW - 1) / g.TW;
  return g;
}

// rows per band and planes per chunk together (the chunk of lbm_set_zchunk belongs to
// the collision pass on the populations, another kernel): the waves
// of CTAs (one per SM) times a CTA's planes (two collided beyond the chunk,
// the prologue worth two more) times the time of a plane, which grows with
// the rows held (the band, one beyond either side, the edge warp, and about
// four rows' worth of barrier and latency)
void mom_cut(const KParams& kp, MomGeo* g, int* zc) {
  const long long slots = device_sms();
  double best = 1e300;
  // (each height of a band and each chunk once, the largest first)
  for (int most = std::min(MW3 - 3, kp.ny); most > 0; --most) {
    const int nb = (kp.ny + most - 1) / most, rb = (kp.ny + nb - 1) / nb, bands = (kp.ny + rb - 1) / rb;
    if (2 * rb < MW3 - 3 && best < 1e300) break;
    for (int n = 1, c; n <= kp.nz; n = (kp.nz + c - 2) / (c - 1)) {
      c = (kp.nz + n - 1) / n;
      if (c < 2 && n > 1) break;
      const long long ctas = (long long)g->nt * bands * ((kp.nz + c - 1) / c);
      const double cost = double((ctas + slots - 1) / slots) * (c + 4) * (rb + 7);
      if (cost < best - 1e-9) { best = cost; *zc = c; g->RB = rb; g->nb = bands; }
      if (ctas > 8 * slots || c < 2) break;
    }
  }
}

template <int S>
MomConst mom_const() {
  auto two = [](double v) { return float2{float(v), float(v)}; };
  MomConst k{};
  for (int m = 1; m <= Sch<S>::R && !Sch<S>::GF; ++m) {
    k.g[m - 1] = two(Sch<S>::g(m));
    k.h[m - 1] = two(Sch<S>::g(m) / 3.0);
  }
  k.m1 = two(-1.0); k.c45 = two(4.5); k.m15 = two(-1.5); k.m12 = two(-12.0);
  k.w0 = two(1.0 / 3); k.w1 = two(1.0 / 18); k.w2 = two(1.0 / 36);
  k.t1 = two(3.0 / 18); k.t2 = two(3.0 / 36); k.n1 = two(-3.0 / 18); k.n2 = two(-3.0 / 36);
  return k;
}

// S: the scheme, SL: the one whose Laplacian the mu pass takes (S itself unless
// compact, S == S_CFDS4, whose solves are those of `scheme`)
template <int S, int SL, bool M64>
cudaError_t steps(const Launch& c, int scheme, long long n) {
  constexpr bool GF = Sch<S>::GF;
  const KParams& kp = c.kp;
  MomGeo g = mom_geo(kp);
  int zc = 0;
  mom_cut(kp, &g, &zc);
  const float *fin = static_cast<const float*>(c.fin), *rin = static_cast<const float*>(c.rin);
  float* s = static_cast<float*>(c.fout);  // scratch: rho x 2, j x 2, mu, compact: F / rho
  float* r[2] = {s, s + g.P};
  float* j[2] = {s + 2 * g.P, s + 5 * g.P};
  float *mu = s + 8 * g.P, *acc = s + 9 * g.P;
  const int elems = g.PL * kp.nz;
  k_mom_gather<<<(elems + 255) / 256, 256, 0, c.stream>>>(kp, g, fin, rin, r[0], j[0], r[1], mu, j[1],
                                                          GF ? acc : nullptr, c.aux.bad_step, c.aux.t);
  // mu pass: about eight CTAs per SM; at least eight planes each, down to two
  // where that leaves SMs without a CTA (a plane is a round trip to L2)
  const int gm = ((kp.nx + 3) / 4 * kp.ny + 255) / 256;
  const int least = std::max(2, std::min(8, int((long long)gm * kp.nz / (2 * device_sms()))));
  const int nzm = std::max(1, std::min((8 * device_sms() + gm - 1) / gm, (kp.nz + least - 1) / least));
  const int zm = (kp.nz + nzm - 1) / nzm;
  const dim3 gridm(gm, (kp.nz + zm - 1) / zm);
  const dim3 grid(g.nt, g.nb, (kp.nz + zc - 1) / zc);
  const IirGeo ig{kp.nx, kp.ny, kp.nz, g.LX, g.PL, 4, g.P};
  for (long long k = 0; k < n; ++k) {
    const int a = int(k & 1);
    if (c.ev_mu) cudaEventRecord(c.ev_mu[2 * k], c.stream);
    cudaError_t e = launch_pdl(k_mom_mu<SL, M64>, gridm, 256, 0, c.stream, kp, g, r[a], mu, zm);
    if (c.ev_mu) cudaEventRecord(c.ev_mu[2 * k + 1], c.stream);
    if constexpr (GF) {
      constexpr size_t smem = size_t(2) * (MomCell<MW3>::XB + MomCell<MW3>::EB) * 4;
      if (e == cudaSuccess) e = iir_acc(ig, scheme, r[a], mu, acc, float(kp.rho_ref), c.stream);
      if (e == cudaSuccess) e = ensure_smem(k_mom3d_acc<MW3>, smem);
      if (e == cudaSuccess)
        e = launch_pdl(k_mom3d_acc<MW3>, grid, 32 * MW3, smem, c.stream, kp, g, r[a], acc, j[a], r[a ^ 1], j[a ^ 1],
                       c.aux.bad_step, c.aux.t + k, zc, mom_const<S>());
    } else {
      using Sh = MomShape<S, MW3>;
      static_assert(Sh::bytes <= size_t(227) * 1024, "shared memory of one CTA");
      if (e == cudaSuccess) e = ensure_smem(k_mom3d<S, MW3>, Sh::bytes);
      if (e == cudaSuccess)
        e = launch_pdl(k_mom3d<S, MW3>, grid, Sh::NT, Sh::bytes, c.stream, kp, g, r[a], mu, j[a], r[a ^ 1], j[a ^ 1],
                       c.aux.bad_step, c.aux.t + k, zc, mom_const<S>());
    }
    if (e != cudaSuccess) return e;
  }
  const int a = int((n - 1) & 1);
  k_mom_expand<S><<<int((kp.n + 255) / 256), 256, 0, c.stream>>>(kp, g, r[a], GF ? acc : mu, j[a], r[a ^ 1],
                                                                 const_cast<float*>(fin), const_cast<float*>(rin));
  return cudaGetLastError();
}

}  // namespace

bool mom3d_ok(const KParams& kp, int scheme, int prec) {
  if ((prec != 1 && prec != 2) || kp.omega != 1.0) return false;
  const bool compact = scheme >= S_CFDS4 && scheme <= S_OCFDS4;
  if (!compact && scheme != S_EFDS2 && scheme != S_EFDS4 && scheme != S_EFDS6) return false;
  if (compact && (prec != 1 || !iir_ok(kp))) return false;
  const long long LX = (kp.nx + 3) / 4 * 4 + 8, P = (LX * kp.ny * kp.nz + 63) / 64 * 64;
  return (compact ? 12 : 9) * P <= 19 * kp.n && 19 * kp.n < (1LL << 31);
}

// A call's gather and expansion cost as much as two of its steps on the moments, so
// two steps pay only where a step on the populations is dear.  Not where rows are
// whole 16-byte chunks beyond the node-parallel passes' sizes and the stencil is wide
// or the populations are partly in the L2, nor where the compact schemes' lines are
// solved in registers (multiples of 32; CFDS8's mu pass is dearer).  Measured, us a
// step of single steps, two and three a call: 160^3 EFDS2 143, 158, 134, EFDS6 159,
// 187, 159; 256^3 EFDS2 566, 524, 430, EFDS4 580, 564, 466, EFDS6 610, 619, 516; 192^3
// EFDS6 281, 270, 224, 224^3 417, 440, 367; 129^3 EFDS6 134, 111.  CFDS4 128 x 128 x 64
// 84, 68; 128^3 115, 128, 114; 160^3 202, 236, 210; 224^3 550, 589, 522; 256^3 847, 795;
// CFDS8 160^3 283, 245.
int mom3d_least(const KParams& kp, int scheme) {
  if (scheme == S_EFDS2 || scheme == S_EFDS4 || scheme == S_EFDS6)
    return kp.nx % 4 == 0 && kp.n > 1200000 && (scheme == S_EFDS6 || kp.n < 6000000) ? 3 : 2;
  const bool regs = kp.nx % 32 == 0 && kp.ny % 32 == 0 && kp.nz % 32 == 0;
  if (!regs || scheme == S_CFDS8 || kp.n < 1500000 || kp.n > 14000000) return 2;
  return scheme == S_CFDS4 && kp.n > 3000000 && kp.n < 6000000 ? 4 : 3;
}

cudaError_t mom3d_steps(const Launch& c, int scheme, int prec, long long n) {
  switch (scheme) {
    case S_EFDS2:
      return prec == 2 ? steps<S_EFDS2, S_EFDS2, true>(c, scheme, n) : steps<S_EFDS2, S_EFDS2, false>(c, scheme, n);
    case S_EFDS4:
      return prec == 2 ? steps<S_EFDS4, S_EFDS4, true>(c, scheme, n) : steps<S_EFDS4, S_EFDS4, false>(c, scheme, n);
    case S_EFDS6:
      return prec == 2 ? steps<S_EFDS6, S_EFDS6, true>(c, scheme, n) : steps<S_EFDS6, S_EFDS6, false>(c, scheme, n);
    // compact schemes: the Laplacian of their order (Sec. 2.3)
    case S_CFDS4:
    case S_OCFDS4: return steps<S_CFDS4, S_EFDS4, false>(c, scheme, n);
    case S_CFDS6: return steps<S_CFDS4, S_EFDS6, false>(c, scheme, n);
    case S_CFDS8: return steps<S_CFDS4, S_LAP8, false>(c, scheme, n);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace lbmd
