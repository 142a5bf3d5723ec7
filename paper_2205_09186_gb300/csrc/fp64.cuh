// The FP64 step as three node-parallel passes:
//
//  k64_mu    mu = k^2 psi'(rho) - kappa lap rho (Eq. 16), once per node
//  k64_coll  F, collision, push streaming, one thread per node
//  k64_rho   the next density, the sum of the populations pushed into a node
//
// The FP64 pipe sets the time of such a step (about two operations per clock
// and SM, 1/64 of FP32), not the 330 (D3Q19) bytes a node moves: everything
// here serves to issue few FP64 instructions.  mu is not evaluated on halos
// (the tiled kernels evaluate it 2.2 times per node in 2D and more in 3D),
// nothing is collided twice for the sake of the next density (read back
// instead), one reciprocal replaces the divisions by rho and by 3, and opposite
// directions share their even and odd parts.  Blocks are small on small
// lattices, whose nodes are too few to fill 152 SMs: 32 nodes per block.
#pragma once
#include "lbm_device.cuh"
#include "mrt.cuh"
#include "step2d.cuh"

namespace lbmd {

// coordinates of node n and its neighbours' indices
template <int LAT>
struct Node64 {
  int n, x, y, z, nx, ny, nz, nxy;
  __device__ __forceinline__ Node64(const KParams& p, int n_) : n(n_), nx(p.nx), ny(p.ny), nz(p.nz), nxy(p.nx * p.ny) {
    const int r = n / nx;
    x = n - r * nx;
    z = LAT == 0 ? 0 : r / ny;
    y = LAT == 0 ? r : r - z * ny;
  }
  __device__ __forceinline__ int at(int dx, int dy, int dz) const {
    int o = n;
    if (dx != 0) o += dx + (x + dx < 0 ? nx : (x + dx >= nx ? -nx : 0));
    if (dy != 0) o += (dy + (y + dy < 0 ? ny : (y + dy >= ny ? -ny : 0))) * nx;
    if (dz != 0) o += (dz + (z + dz < 0 ? nz : (z + dz >= nz ? -nz : 0))) * nxy;
    return o;
  }
};

template <int S, int LAT>
__device__ __forceinline__ double lap64(const double* q, const Node64<LAT>& c, double v) {
  using Sc = Sch<S>;
  constexpr int R = Sc::R, D = LAT == 0 ? 2 : 3;
  double a;
  if constexpr (Sc::ISO) {
    a = 0.0;
#pragma unroll
    for (int dz = (D == 3 ? -R : 0); dz <= (D == 3 ? R : 0); ++dz)
#pragma unroll
      for (int dy = -R; dy <= R; ++dy)
#pragma unroll
        for (int dx = -R; dx <= R; ++dx) {
          const double w = D == 2 ? Sc::w2d(dx, dy) : Sc::w3d(dx, dy, dz);
          if (w != 0.0) a += (2.0 * w) * (q[c.at(dx, dy, dz)] - v);
        }
  } else {
    a = double(D) * Sc::l(0) * v;
#pragma unroll
    for (int m = 1; m <= R; ++m) {
      double s = (q[c.at(m, 0, 0)] + q[c.at(-m, 0, 0)]) + (q[c.at(0, m, 0)] + q[c.at(0, -m, 0)]);
      if constexpr (D == 3) s += q[c.at(0, 0, m)] + q[c.at(0, 0, -m)];
      a += Sc::l(m) * s;
    }
  }
  return a;
}

template <int S, int LAT>
__device__ __forceinline__ void grad64(const double* q, const Node64<LAT>& c, double* g) {
  using Sc = Sch<S>;
  constexpr int R = Sc::R, D = LAT == 0 ? 2 : 3;
  g[0] = g[1] = g[2] = 0.0;
  if constexpr (Sc::ISO) {
#pragma unroll
    for (int dz = (D == 3 ? -R : 0); dz <= (D == 3 ? R : 0); ++dz)
#pragma unroll
      for (int dy = -R; dy <= R; ++dy)
#pragma unroll
        for (int dx = -R; dx <= R; ++dx) {
          const double w = D == 2 ? Sc::w2d(dx, dy) : Sc::w3d(dx, dy, dz);
          if (w != 0.0 && (dx != 0 || dy != 0 || dz != 0)) {
            const double v = q[c.at(dx, dy, dz)];
            if (dx != 0) g[0] += (w * dx) * v;
            if (dy != 0) g[1] += (w * dy) * v;
            if (dz != 0) g[2] += (w * dz) * v;
          }
        }
  } else {
#pragma unroll
    for (int m = 1; m <= R; ++m) {
      g[0] += Sc::g(m) * (q[c.at(m, 0, 0)] - q[c.at(-m, 0, 0)]);
      g[1] += Sc::g(m) * (q[c.at(0, m, 0)] - q[c.at(0, -m, 0)]);
      if constexpr (D == 3) g[2] += Sc::g(m) * (q[c.at(0, 0, m)] - q[c.at(0, 0, -m)]);
    }
  }
}

template <int S, int LAT>
__global__ void k64_mu(const KParams p, const double* __restrict__ rho, double* __restrict__ mu) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= int(p.n)) return;
  const Node64<LAT> c(p, n);
  const double r = rho[n];
  mu[n] = p.k2 * eos_mu<double>(r, p) - p.kappa * lap64<S, LAT>(rho, c, r);
}

// e_i . (x, y, z) of a direction's first nonzero components, no multiplication
template <class L>
__device__ __forceinline__ double edot64(int i, double x, double y, double z) {
  double s = 0.0;
  bool any = false;
  const int e[3] = {L::ex(i), L::ey(i), L::ez(i)};
  const double v[3] = {x, y, z};
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if (e[a] != 0) {
      s = any ? (e[a] > 0 ? s + v[a] : s - v[a]) : (e[a] > 0 ? v[a] : -v[a]);
      any = true;
    }
  return s;
}

// index of the direction opposite to i (constant after unrolling)
template <class L>
__device__ constexpr int opp64(int i) {
  for (int j = 0; j < L::Q; ++j)
    if (L::ex(j) == -L::ex(i) && L::ey(j) == -L::ey(i) && L::ez(j) == -L::ez(i)) return j;
  return i;
}

// COLL: 0 single relaxation at tau = 1, 1 at any tau, 2 the D2Q9 MRT operator.
// A compact scheme (GF) reads grad mu and grad rho from gi, the others take
// them from rho and mu.
template <int S, int LAT, int COLL>
__global__ void k64_coll(const KParams p, const double* __restrict__ fin, double* __restrict__ fout,
                         const double* __restrict__ rho, const double* __restrict__ mu, const GradIn gi,
                         const StepAux aux, const Mrt mrt) {
  using L = Lattice<LAT>;
  constexpr int Q = L::Q, D = L::D;
  const int n = blockIdx.x * blockDim.x + threadIdx.x, N = int(p.n);
  if (n >= N) return;
  const Node64<LAT> c(p, n);
  double f[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) f[i] = fin[i * N + n];
  const double r = rho[n];
  double gm[3], gr[3];
  if constexpr (Sch<S>::GF) {
    const double *a = static_cast<const double*>(gi.gmu), *b = static_cast<const double*>(gi.grho);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      gm[k] = k < D ? a[k * N + n] : 0.0;
      gr[k] = k < D ? b[k * N + n] : 0.0;
    }
  } else {
    grad64<S, LAT>(mu, c, gm);
    grad64<S, LAT>(rho, c, gr);
  }
  if (!(r > 0.0)) atomicMin(aux.bad_step, (unsigned long long)aux.t);
  double jx = 0.0, jy = 0.0, jz = 0.0;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const int o = opp64<L>(i);
    if (o < i) continue;
    const double d = f[i] - f[o];
    if (L::ex(i) != 0) jx = L::ex(i) > 0 ? jx + d : jx - d;
    if (L::ey(i) != 0) jy = L::ey(i) > 0 ? jy + d : jy - d;
    if (L::ez(i) != 0) jz = L::ez(i) > 0 ? jz + d : jz - d;
  }
  const double ir = 1.0 / r;
  const double ux = jx * ir, uy = jy * ir, uz = D == 3 ? jz * ir : 0.0;
  // v = u + F / rho, F = -rho grad mu + grad rho / 3 (Eq. 12)
  const double ir3 = ir * (1.0 / 3.0);
  const double vx = ux + (gr[0] * ir3 - gm[0]), vy = uy + (gr[1] * ir3 - gm[1]),
               vz = D == 3 ? uz + (gr[2] * ir3 - gm[2]) : 0.0;
  auto push = [&](int i, double v) { fout[i * N + c.at(L::ex(i), L::ey(i), L::ez(i))] = v; };
  if constexpr (COLL == 2) {
    double post[Q];
    mrt_post9<double>(f, r, r, ux, uy, vx, vy, mrt, post);
#pragma unroll
    for (int i = 0; i < Q; ++i) push(i, post[i]);
  } else {
    // w rho (1 - 1.5 v.v + 4.5 (e.v)^2 +- 3 e.v) at tau = 1; else the same with
    // omega for 1 and the u terms times omega - 1 added, plus (1 - omega) f_i
    const double om = p.omega, o1 = om - 1.0;
    double ev = 1.0 - 1.5 * (vx * vx + vy * vy + (D == 3 ? vz * vz : 0.0));
    double sx = vx, sy = vy, sz = vz;
    if constexpr (COLL == 1) {
      ev += o1 - (1.5 * o1) * (ux * ux + uy * uy + (D == 3 ? uz * uz : 0.0));
      sx += o1 * ux;
      sy += o1 * uy;
      sz += o1 * uz;
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int o = opp64<L>(i);
      if (o < i) continue;
      const double w = L::w(i);
      const double wr = w * r;
      if (i == 0) {
        push(0, COLL == 1 ? wr * ev - o1 * f[0] : wr * ev);
        continue;
      }
      const double E = edot64<L>(i, vx, vy, vz);
      double even = 4.5 * (E * E) + ev, odd = E;
      if constexpr (COLL == 1) {
        const double U = edot64<L>(i, ux, uy, uz);
        even += (4.5 * o1) * (U * U);
        odd = edot64<L>(i, sx, sy, sz);
      }
      const double a = wr * even, b = (3.0 * wr) * odd;
      push(i, COLL == 1 ? (a + b) - o1 * f[i] : a + b);
      push(o, COLL == 1 ? (a - b) - o1 * f[o] : a - b);
    }
  }
}

template <int Q>
__global__ void k64_rho(const KParams p, const double* __restrict__ f, double* __restrict__ rho,
                        unsigned long long* bad, long long t1) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x, N = int(p.n);
  if (n >= N) return;
  double a = 0.0;
#pragma unroll
  for (int i = 0; i < Q; ++i) a += f[i * N + n];
  rho[n] = a;
  if (!(a > 0.0)) atomicMin(bad, (unsigned long long)t1);
}

}  // namespace lbmd
