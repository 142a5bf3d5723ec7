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
#include "launch.cuh"
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
__global__ void k64_mu(const KParams p, const double* rho, double* __restrict__ mu) {
  pdl_wait();
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

// Post-collision populations of one node from its populations f, density r and
// the gradients of mu and rho, handed to put(i, value).  COLL: 0 single
// relaxation at tau = 1, 1 at any tau, 2 the D2Q9 MRT operator.
template <int LAT, int COLL, class Put>
__device__ __forceinline__ void post64(const KParams& p, const Mrt& mrt, const double* f, double r, const double* gm,
                                       const double* gr, Put put) {
  using L = Lattice<LAT>;
  constexpr int Q = L::Q, D = L::D;
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
  // v = u + F / rho, F = -rho grad mu + grad rho / 3 (Eq. 12)
  const double ir = rcp64(r), ir3 = ir * (1.0 / 3.0);
  const double vx = fma(gr[0], ir3, fma(jx, ir, -gm[0])), vy = fma(gr[1], ir3, fma(jy, ir, -gm[1])),
               vz = D == 3 ? fma(gr[2], ir3, fma(jz, ir, -gm[2])) : 0.0;
  const double ux = COLL ? jx * ir : 0.0, uy = COLL ? jy * ir : 0.0, uz = COLL && D == 3 ? jz * ir : 0.0;
  if constexpr (COLL == 2) {
    double post[Q];
    mrt_post9<double>(f, r, r, ux, uy, vx, vy, mrt, post);
#pragma unroll
    for (int i = 0; i < Q; ++i) put(i, post[i]);
  } else {
    // w rho (1 - 1.5 v.v + 4.5 (e.v)^2 +- 3 e.v) at tau = 1; else the same with
    // omega for 1 and the u terms times omega - 1 added, plus (1 - omega) f_i
    const double o1 = p.omega - 1.0;
    double vv = vx * vx + vy * vy;
    if constexpr (D == 3) vv = fma(vz, vz, vv);
    double ev = fma(-1.5, vv, 1.0), sx = vx, sy = vy, sz = vz;
    if constexpr (COLL == 1) {
      double uu = ux * ux + uy * uy;
      if constexpr (D == 3) uu = fma(uz, uz, uu);
      ev = fma(o1, fma(-1.5, uu, 1.0), ev);
      sx = fma(o1, ux, sx);
      sy = fma(o1, uy, sy);
      sz = fma(o1, uz, sz);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int o = opp64<L>(i);
      if (o < i) continue;
      const double wr = L::w(i) * r;
      if (i == 0) {
        put(0, COLL == 1 ? fma(wr, ev, -o1 * f[0]) : wr * ev);
        continue;
      }
      const double E = edot64<L>(i, vx, vy, vz), t = (3.0 * L::w(i)) * r;
      double even = fma(4.5, E * E, ev), odd = E;
      if constexpr (COLL == 1) {
        const double U = edot64<L>(i, ux, uy, uz);
        even = fma(4.5 * o1, U * U, even);
        odd = edot64<L>(i, sx, sy, sz);
      }
      const double a = wr * even;
      put(i, COLL == 1 ? fma(-o1, f[i], fma(t, odd, a)) : fma(t, odd, a));
      put(o, COLL == 1 ? fma(-o1, f[o], fma(-t, odd, a)) : fma(-t, odd, a));
    }
  }
}

// A compact scheme (GF) reads grad mu and grad rho from gi, or F / rho from gi.gmu
// where gi.grho is null; the others take them from rho and mu.
template <int S, int LAT, int COLL>
__global__ void k64_coll(const KParams p, const double* fin, double* __restrict__ fout,
                         const double* rho, const double* mu, const GradIn gi,
                         const StepAux aux, const Mrt mrt) {
  pdl_wait();
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
      gm[k] = k < D ? (b ? a[k * N + n] : -a[k * N + n]) : 0.0;
      gr[k] = k < D && b ? b[k * N + n] : 0.0;
    }
  } else {
    grad64<S, LAT>(mu, c, gm);
    grad64<S, LAT>(rho, c, gr);
  }
  if (!(r > 0.0)) atomicMin(aux.bad_step, (unsigned long long)aux.t);
  post64<LAT, COLL>(p, mrt, f, r, gm, gr,
                    [&](int i, double v) { fout[i * N + c.at(L::ex(i), L::ey(i), L::ez(i))] = v; });
}

// The whole D2Q9 step of an 8 x 4 tile by one CTA of four warps (one per
// scheduler, each with its own FP64 pipe): density of the tile and its halo in
// shared memory, mu on the tile and R + 1 beyond, collision of the tile and a
// ring, next density from the ring's and the tile's populations.  For lattices
// whose tiles find an SM each: the redundant nodes run on pipes that would idle,
// and one launch takes the place of three.  64^2 EFDS2 takes 8.2 us a step (16.4
// on the three passes; 6.0 with each launch overlapping the step before); with two tiles per SM the pipes are shared and the passes
// (16.4 us at 96^2 EFDS6) are level with it.
constexpr int T64X = 8, T64Y = 4, T64N = 128;

template <int S, int COLL>
__global__ void __launch_bounds__(T64N) k64_tile(const KParams p, const double* fin,
                                                 double* __restrict__ fout, const double* rin,
                                                 double* __restrict__ rout, const StepAux aux, const Mrt mrt) {
  pdl_wait();
  using L = Lattice<0>;
  constexpr int Q = 9, R = Sch<S>::R, H = 2 * R + 1;
  constexpr int RW = T64X + 2 * H, RH = T64Y + 2 * H, MW = T64X + 2 * R + 2, MH = T64Y + 2 * R + 2;
  constexpr int CW = T64X + 2, CH = T64Y + 2;
  __shared__ double s_r[RH * RW], s_m[MH * MW], s_f[Q][CH * CW];
  const int nx = p.nx, ny = p.ny, N = int(p.n), x0 = blockIdx.x * T64X, y0 = blockIdx.y * T64Y;
  const int tid = threadIdx.x;
  for (int e = tid; e < RW * RH; e += T64N) {
    const int ry = e / RW, rx = e - ry * RW;
    int gx = x0 - H + rx, gy = y0 - H + ry;
    gx = wrapn(gx, nx);
    gy = wrapn(gy, ny);
    s_r[e] = rin[gy * nx + gx];
  }
  // the populations of this thread's collided node travel meanwhile
  double f[Q];
  const int cy = tid / CW, cx = tid - cy * CW;
  const bool col = tid < CW * CH;
  const int gx = wrapn(x0 - 1 + cx, nx), gy = wrapn(y0 - 1 + cy, ny);
  if (col) {
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = fin[i * N + gy * nx + gx];
  }
  __syncthreads();
  for (int e = tid; e < MW * MH; e += T64N) {
    const int my = e / MW, mx = e - my * MW, sx = mx + R, sy = my + R;
    const double r = s_r[sy * RW + sx];
    s_m[e] = p.k2 * eos_mu<double>(r, p) - p.kappa * lap2d<S, double>(s_r, RW, sx, sy);
  }
  __syncthreads();
  if (col) {
    const int lx = cx - 1, ly = cy - 1;
    const bool own = lx >= 0 && lx < T64X && ly >= 0 && ly < T64Y && x0 + lx < nx && y0 + ly < ny;
    const double r = s_r[(ly + H) * RW + lx + H];
    double gm[3], gr[3];
    grad2d<S, double>(s_m, MW, lx + R + 1, ly + R + 1, gm[0], gm[1]);
    grad2d<S, double>(s_r, RW, lx + H, ly + H, gr[0], gr[1]);
    gm[2] = gr[2] = 0.0;
    if (own && !(r > 0.0)) atomicMin(aux.bad_step, (unsigned long long)aux.t);
    post64<0, COLL>(p, mrt, f, r, gm, gr, [&](int i, double v) {
      s_f[i][tid] = v;
      if (own) fout[i * N + wrapi(gy + L::ey(i), ny) * nx + wrapi(gx + L::ex(i), nx)] = v;
    });
  }
  __syncthreads();
  if (tid < T64X * T64Y) {
    const int ly = tid / T64X, lx = tid - ly * T64X;
    if (x0 + lx < nx && y0 + ly < ny) {
      double a = 0.0;
#pragma unroll
      for (int i = 0; i < Q; ++i) a += s_f[i][(ly + 1 - L::ey(i)) * CW + lx + 1 - L::ex(i)];
      rout[(y0 + ly) * nx + x0 + lx] = a;
      if (!(a > 0.0)) atomicMin(aux.bad_step, (unsigned long long)(aux.t + 1));
    }
  }
}

template <int Q>
__global__ void k64_rho(const KParams p, const double* f, double* __restrict__ rho,
                        unsigned long long* bad, long long t1) {
  pdl_wait();
  const int n = blockIdx.x * blockDim.x + threadIdx.x, N = int(p.n);
  if (n >= N) return;
  double a = 0.0;
#pragma unroll
  for (int i = 0; i < Q; ++i) a += f[i * N + n];
  rho[n] = a;
  if (!(a > 0.0)) atomicMin(bad, (unsigned long long)t1);
}

}  // namespace lbmd
