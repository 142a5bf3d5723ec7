// D2Q9 FP32-deviation step as three node-parallel passes, for lattices that are
// done in a few microseconds:
//
//  k_node2_mu    mu = k^2 psi'(rho) - kappa lap rho (Eq. 16)
//  k_node2_coll  F, collision (single relaxation or MRT), push streaming
//  k_node2_rho   the next density, the sum of the populations pushed into a node
//
// On such a lattice a launch is a chain of latencies: the tiled passes stage their
// halo, wait, collide the ring of each tile as well and wait again for the
// exchange (5.5 and 10.8 us at 512^2); a node per thread reads its neighbours
// through the caches, and the launches overlap their starts. Beyond the ranges of
// node2_rule (k2d.cu) reading the populations back costs more than it saves.
#pragma once
#include "launch.cuh"
#include "mrt.cuh"
#include "step2d.cuh"

namespace lbmd {

constexpr int NODE2_T = 128;  // threads per block

// a node's coordinates and its neighbours' indices; mx: ceil(2^32 / nx), a
// quotient at most one too large
struct Node2 {
  int n, x, y, nx, ny;
  __device__ __forceinline__ Node2(const KParams& p, int n_, unsigned mx) : n(n_), nx(p.nx), ny(p.ny) {
    y = int(__umulhi(unsigned(n), mx));
    if (y * nx > n) --y;
    x = n - y * nx;
  }
  __device__ __forceinline__ int dx(int d) const { return d + (x + d < 0 ? nx : (x + d >= nx ? -nx : 0)); }
  __device__ __forceinline__ int dy(int d) const { return (d + (y + d < 0 ? ny : (y + d >= ny ? -ny : 0))) * nx; }
};

template <int S>
__global__ void __launch_bounds__(NODE2_T) k_node2_mu(const KParams p, const unsigned mx, const float* rin,
                                                      float* __restrict__ mu) {
  pdl_wait();
  using Sc = Sch<S>;
  constexpr int R = Sc::R;
  const int n = blockIdx.x * NODE2_T + threadIdx.x;
  if (n >= int(p.n)) return;
  const Node2 c(p, n, mx);
  const float* q = rin + n;
  const float d = q[0];
  float lap;
  if constexpr (Sc::ISO) {
    lap = 0.f;
#pragma unroll
    for (int j = -R; j <= R; ++j)
#pragma unroll
      for (int i = -R; i <= R; ++i)
        if (const double w = Sc::w2d(i, j); w != 0.0 && (i != 0 || j != 0)) lap += float(2.0 * w) * (q[c.dx(i) + c.dy(j)] - d);
  } else {
    lap = float(2.0 * Sc::l(0)) * d;
#pragma unroll
    for (int m = 1; m <= R; ++m) lap += float(Sc::l(m)) * ((q[c.dx(m)] + q[c.dx(-m)]) + (q[c.dy(m)] + q[c.dy(-m)]));
  }
  mu[n] = float(p.k2) * eos_mu_f(float(p.rho_ref) + d, eos_f(p)) - float(p.kappa) * lap;
}

// COLL: 0 single relaxation at tau = 1, 1 at any tau, 2 MRT
template <int S, int COLL>
__global__ void __launch_bounds__(NODE2_T) k_node2_coll(const KParams p, const unsigned mx, const float* fin,
                                                        float* __restrict__ fout, const float* rin,
                                                        const float* mu, unsigned long long* bad,
                                                        const long long t, const Mrt mrt) {
  pdl_wait();
  using L = Lattice<0>;
  using Sc = Sch<S>;
  constexpr int Q = 9, R = Sc::R;
  const int n = blockIdx.x * NODE2_T + threadIdx.x, N = int(p.n);
  if (n >= N) return;
  float f[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) f[i] = fin[i * N + n];
  const Node2 c(p, n, mx);
  const float d = rin[n], rc = float(p.rho_ref) + d;
  float grx = 0.f, gry = 0.f, gmx = 0.f, gmy = 0.f;
  if constexpr (Sc::ISO) {
    // half the offsets, each with its opposite (the weights are even)
#pragma unroll
    for (int j = 0; j <= R; ++j)
#pragma unroll
      for (int i = -R; i <= R; ++i)
        if (const double w = Sc::w2d(i, j); w != 0.0 && (j > 0 || i > 0)) {
          const int a = n + c.dx(i) + c.dy(j), b = n + c.dx(-i) + c.dy(-j);
          const float r = rin[a] - rin[b], m = mu[a] - mu[b];
          if (i != 0) {
            grx += float(w * i) * r;
            gmx += float(w * i) * m;
          }
          if (j != 0) {
            gry += float(w * j) * r;
            gmy += float(w * j) * m;
          }
        }
  } else {
#pragma unroll
    for (int m = 1; m <= R; ++m) {
      const float g = float(Sc::g(m));
      const int xp = n + c.dx(m), xm = n + c.dx(-m), yp = n + c.dy(m), ym = n + c.dy(-m);
      grx += g * (rin[xp] - rin[xm]);
      gry += g * (rin[yp] - rin[ym]);
      gmx += g * (mu[xp] - mu[xm]);
      gmy += g * (mu[yp] - mu[ym]);
    }
  }
  float jx = 0.f, jy = 0.f;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    if (L::ex(i) != 0) jx = L::ex(i) > 0 ? jx + f[i] : jx - f[i];
    if (L::ey(i) != 0) jy = L::ey(i) > 0 ? jy + f[i] : jy - f[i];
  }
  if (!(rc > 0.f)) atomicMin(bad, (unsigned long long)t);
  // v = u + F / rho, F = -rho grad mu + grad rho / 3 (Eq. 12)
  const float ir = __fdividef(1.f, rc), om = float(p.omega), o1 = 1.f - om;
  const float ux = jx * ir, uy = jy * ir;
  const float vx = fmaf(fmaf(-rc, gmx, grx * (1.f / 3.f)), ir, ux), vy = fmaf(fmaf(-rc, gmy, gry * (1.f / 3.f)), ir, uy);
  const int ox[3] = {c.dx(-1), 0, c.dx(1)}, oy[3] = {c.dy(-1), 0, c.dy(1)};
  auto put = [&](int i, float v) { fout[i * N + n + ox[L::ex(i) + 1] + oy[L::ey(i) + 1]] = v; };
  if constexpr (COLL == 2) {
    float post[Q];
    mrt_post9<float>(f, d, rc, ux, uy, vx, vy, mrt, post);
#pragma unroll
    for (int i = 0; i < Q; ++i) put(i, post[i]);
  } else {
    const float vv = 1.5f * (vx * vx + vy * vy), uu = 1.5f * (ux * ux + uy * uy);
    // the rest population carries the density less the others' shares (rounded
    // weights; w5 = w1 / 4 exactly)
    const float wd1 = float(L::w(1)) * d, wd2 = float(L::w(5)) * d, wd0 = fmaf(-5.f, wd1, d);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const float wd = i == 0 ? wd0 : (i < 5 ? wd1 : wd2);
      const float wr = float(L::w(i)) * rc;
      const float ev = edot<L>(i, vx, vy, 0.f), Av = i == 0 ? -vv : ev * (3.f + 4.5f * ev) - vv;
      if constexpr (COLL == 0) {
        put(i, wd + wr * Av);
      } else {
        const float eu = edot<L>(i, ux, uy, 0.f), Au = i == 0 ? -uu : eu * (3.f + 4.5f * eu) - uu;
        put(i, o1 * f[i] + om * wd + wr * (om * Au + Av - Au));
      }
    }
  }
}

__global__ void __launch_bounds__(NODE2_T) k_node2_rho(const KParams p, const float* f,
                                                       float* __restrict__ rho, unsigned long long* bad, const long long t1) {
  pdl_wait();
  const int n = blockIdx.x * NODE2_T + threadIdx.x, N = int(p.n);
  if (n >= N) return;
  float v[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) v[i] = f[i * N + n];
  const float d = v[0] + (((v[1] + v[2]) + (v[3] + v[4])) + ((v[5] + v[6]) + (v[7] + v[8])));
  rho[n] = d;
  if (!(float(p.rho_ref) + d > 0.f)) atomicMin(bad, (unsigned long long)t1);
}

}  // namespace lbmd
