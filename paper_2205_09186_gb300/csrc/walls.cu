// Chemical-potential wall boundary (Appendix A) for the explicit schemes
// EFDS2/4/6 on D2Q9 and D3Q19, FP64 and FP32-deviation storage.
//
// A step with walls runs as node-parallel passes (walls break the tile
// regularity the fused kernels rely on; this path is correctness first):
//   1. wall densities, layer 1, 2, 3 in turn (from lists of their nodes): the w_i-weighted average of the
//      neighbours in the layer before (Eq. A.1; layer 0 = fluid);
//   2. mu: k^2 psi'(rho) - kappa-hat lap rho on fluid nodes (Eq. 16), the wall
//      chemical potential mu_w on wall nodes;
//   3. fluid nodes: moments, grad mu and grad rho (Eq. 17-20), F (Eq. 12),
//      BGK or MRT collision with EDM forcing, push streaming with halfway
//      bounce-back off wall nodes;
//   4. next density of the fluid nodes (sum of the populations).
// Wall layers come from the host (lbm_set_solid): 0 fluid, 1..3 the layers
// that fluid stencils reach, 4 deeper (never read, never written).
// Threads: 32 x 8 per CTA over (x, row), row = y + ny z, both grid-strided;
// indices are 32-bit (the handle caps Q N below 2^31).  FP32DEV passes leave the
// FP64 pipe alone (compensated FP32 sums) and every launch overlaps the end of the
// one before: D2Q9 512^2 with a flat wall takes 22 us a step, 48 with FP64 sums and
// six plain launches.
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/lbm.h"
#include "launch.cuh"
#include "mrt.cuh"
#include "walls.cuh"

namespace lbmd {
namespace {

constexpr int WX = 32, WY = 8, WT = WX * WY;

struct Geo {
  int nx, ny, nz, n;
};

// node of (x + dx, y + dy, z + dz) on the periodic lattice, n the node of (x, y,
// z), |d| < the lattice's size along each axis (constant offsets: an axis costs
// nothing where its offset is zero)
__device__ __forceinline__ int at(const Geo& g, int n, int x, int y, int z, int dx, int dy, int dz) {
  if (dx != 0) n += dx + (x + dx < 0 ? g.nx : (x + dx >= g.nx ? -g.nx : 0));
  if (dy != 0) n += (dy + (y + dy < 0 ? g.ny : (y + dy >= g.ny ? -g.ny : 0))) * g.nx;
  if (dz != 0) n += (dz + (z + dz < 0 ? g.nz : (z + dz >= g.nz ? -g.nz : 0))) * g.nx * g.ny;
  return n;
}

// calls fn(x, y, z, node) for every node this thread owns
template <class Fn>
__device__ __forceinline__ void for_nodes(const Geo& g, Fn&& fn) {
  const int rows = g.ny * g.nz;
  for (int r = blockIdx.y * WY + threadIdx.y; r < rows; r += gridDim.y * WY) {
    const int y = r % g.ny, z = r / g.ny;
    for (int x = blockIdx.x * WX + threadIdx.x; x < g.nx; x += gridDim.x * WX) fn(x, y, z, r * g.nx + x);
  }
}

// Eq. A.1 at the nodes list[begin .. end) of layer L, by the threads t, t + nt ...
// The weights are multiples of the smallest one (1 or 4, in 3D 1 or 2): products
// are exact and the FP32DEV sum is compensated, so that the quotient is rounded
// as from FP64, on the FP32 pipe.
template <int LAT, typename Tr>
__device__ __forceinline__ void fill_layer(const Geo& g, const signed char* layer, const int* list, int begin, int end, int L,
                                           Tr* rho, int t, int nt) {
  using Lt = Lattice<LAT>;
  constexpr int Q = LAT == 0 ? 9 : 19;
  for (int k = begin + t; k < end; k += nt) {
    const int n = list[k], r = n / g.nx, x = n - r * g.nx, z = r / g.ny, y = r - z * g.ny;
    int den = 0;
    double num = 0;
    FSum sum;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const int nb = at(g, n, x, y, z, Lt::ex(i), Lt::ey(i), Lt::ez(i));
      if (layer[nb] == L - 1) {
        constexpr int heavy = LAT == 0 ? 4 : 2;
        const int wt = Lt::ex(i) * Lt::ex(i) + Lt::ey(i) * Lt::ey(i) + Lt::ez(i) * Lt::ez(i) == 1 ? heavy : 1;
        if constexpr (sizeof(Tr) == 8) num += double(wt) * rho[nb];
        else sum.add(float(wt) * rho[nb]);
        den += wt;
      }
    }
    if constexpr (sizeof(Tr) == 8) rho[n] = num / double(den);
    else rho[n] = __fdiv_rn(sum.fvalue(), float(den));  // deviations average like densities (normalised weights)
  }
}

// the three layers in turn by one CTA, or one of them by the whole grid (only > 0)
template <int LAT, typename Tr>
__global__ void __launch_bounds__(1024) k_wall_fill(Geo g, const signed char* __restrict__ layer,
                                                    const int* __restrict__ list, int n1, int n2, int n3, int only,
                                                    Tr* rho) {
  pdl_wait();
  const int b[4] = {0, n1, n1 + n2, n1 + n2 + n3};
  for (int L = 1; L <= 3; ++L) {
    if (only == 0) {
      fill_layer<LAT, Tr>(g, layer, list, b[L - 1], b[L], L, rho, threadIdx.x, blockDim.x);
      __syncthreads();
    } else if (only == L) {
      fill_layer<LAT, Tr>(g, layer, list, b[L - 1], b[L], L, rho, blockIdx.x * blockDim.x + threadIdx.x,
                          gridDim.x * blockDim.x);
    }
  }
}

template <int LAT, int S, class P>
__global__ void __launch_bounds__(WT) k_wall_mu(Geo g, KParams p, const signed char* __restrict__ layer,
                                                const typename P::Tr* rho, double mu_w,
                                                typename P::Tm* mu) {
  pdl_wait();
  using Tm = typename P::Tm;
  constexpr int D = LAT == 0 ? 2 : 3, R = Sch<S>::R;
  for_nodes(g, [&](int x, int y, int z, int n) {
    if (layer[n] != 0) {
      mu[n] = Tm(mu_w);
      return;
    }
    // Laplacian of the stored values (deviations in FP32DEV: the weights sum to zero)
    auto st = [&](int dx, int dy, int dz) { return Tm(rho[at(g, n, x, y, z, dx, dy, dz)]); };
    const Tm c0 = Tm(rho[n]);
    Tm lap = Tm(D * Sch<S>::l(0)) * c0;
#pragma unroll
    for (int m = 1; m <= R; ++m) {
      Tm s = (st(m, 0, 0) + st(-m, 0, 0)) + (st(0, m, 0) + st(0, -m, 0));
      if (D == 3) s += st(0, 0, m) + st(0, 0, -m);
      lap += Tm(Sch<S>::l(m)) * s;
    }
    const Tm c = P::DEV ? Tm(p.rho_ref) + c0 : c0;
    mu[n] = Tm(p.k2) * eos_mu<Tm>(c, p) - Tm(p.kappa) * lap;
  });
}

// mode 0: collide and stream; mode 1: F (D x N) and mu (N) as FP64 fields
template <int LAT, int S, class P>
__global__ void __launch_bounds__(WT) k_wall_coll(Geo g, KParams p, Mrt mrt, const signed char* __restrict__ layer,
                                                  const typename P::Tf* fin,
                                                  typename P::Tf* __restrict__ fout,
                                                  const typename P::Tr* rho,
                                                  const typename P::Tm* mu, unsigned long long* bad,
                                                  long long t, int mode, double* F, double* muo) {
  pdl_wait();
  using Lt = Lattice<LAT>;
  using Tc = typename P::Tc;
  using Tm = typename P::Tm;
  using Tf = typename P::Tf;
  constexpr int Q = LAT == 0 ? 9 : 19, D = LAT == 0 ? 2 : 3, R = Sch<S>::R;
  const int N = g.n;
  for_nodes(g, [&](int x, int y, int z, int n) {
    if (layer[n] != 0) {
      if (mode == 1) {  // no force on wall nodes; their mu is mu_w
        for (int a = 0; a < D; ++a) F[a * N + n] = 0.0;
        if (muo) muo[n] = double(mu[n]);
      }
      return;
    }
    Tc fv[Q];
    Tc j[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      fv[i] = Tc(fin[i * N + n]);
      if (Lt::ex(i) != 0) j[0] += Tc(Lt::ex(i)) * fv[i];
      if (Lt::ey(i) != 0) j[1] += Tc(Lt::ey(i)) * fv[i];
      if (Lt::ez(i) != 0) j[2] += Tc(Lt::ez(i)) * fv[i];
    }
    const Tc dsv = Tc(rho[n]);
    const Tc rc = P::DEV ? Tc(p.rho_ref) + dsv : dsv;
    Tc Fv[3] = {0, 0, 0};
#pragma unroll
    for (int a = 0; a < D; ++a) {
      Tm gm = 0;
      Tc gr = 0;
#pragma unroll
      for (int m = 1; m <= R; ++m) {
        const int pp = at(g, n, x, y, z, a == 0 ? m : 0, a == 1 ? m : 0, a == 2 ? m : 0);
        const int qq = at(g, n, x, y, z, a == 0 ? -m : 0, a == 1 ? -m : 0, a == 2 ? -m : 0);
        gm += Tm(Sch<S>::g(m)) * (mu[pp] - mu[qq]);
        gr += Tc(Sch<S>::g(m)) * (Tc(rho[pp]) - Tc(rho[qq]));
      }
      Fv[a] = -rc * Tc(gm) + gr / Tc(3);
    }
    if (mode == 1) {
      for (int a = 0; a < D; ++a) F[a * N + n] = double(Fv[a]);
      if (muo) muo[n] = double(mu[n]);
      return;
    }
    if (!(rc > Tc(0))) atomicMin(bad, (unsigned long long)t);
    const Tc ux = j[0] / rc, uy = j[1] / rc, uz = j[2] / rc;
    const Tc vx = ux + Fv[0] / rc, vy = uy + Fv[1] / rc, vz = uz + Fv[2] / rc;
    Tc post[Q];
    bool done = false;
    if constexpr (LAT == 0) {
      if (mrt.on) {
        mrt_post9<Tc>(fv, dsv, rc, ux, uy, vx, vy, mrt, post);
        done = true;
      }
    }
    if (!done) {
#pragma unroll
      for (int i = 0; i < Q; ++i) post[i] = coll_one<LAT, Tc>(i, fv[i], dsv, rc, Tc(p.omega), ux, uy, uz, vx, vy, vz);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int tg = at(g, n, x, y, z, Lt::ex(i), Lt::ey(i), Lt::ez(i));
      if (layer[tg] != 0) {
        // halfway bounce-back: the population returns to this node reversed
        int o = 0;
#pragma unroll
        for (int k = 0; k < Q; ++k)
          if (Lt::ex(k) == -Lt::ex(i) && Lt::ey(k) == -Lt::ey(i) && Lt::ez(k) == -Lt::ez(i)) o = k;
        fout[o * N + n] = Tf(post[i]);
      } else {
        fout[i * N + tg] = Tf(post[i]);
      }
    }
  });
}

template <int LAT, class P>
__global__ void __launch_bounds__(WT) k_wall_dens(Geo g, KParams p, const signed char* __restrict__ layer,
                                                  const typename P::Tf* f, typename P::Tr* rho,
                                                  unsigned long long* bad, long long t) {
  pdl_wait();
  constexpr int Q = LAT == 0 ? 9 : 19;
  for_nodes(g, [&](int, int, int, int n) {
    if (layer[n] != 0) return;
    if constexpr (P::DEV) {  // compensated: rounded as from an FP64 sum
      FSum s;
#pragma unroll
      for (int i = 0; i < Q; ++i) s.add(f[i * g.n + n]);
      const float v = s.fvalue();
      rho[n] = v;
      if (!(float(p.rho_ref) + v > 0.f)) atomicMin(bad, (unsigned long long)t);
    } else {
      double s = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) s += f[i * g.n + n];
      rho[n] = s;
      if (!(s > 0)) atomicMin(bad, (unsigned long long)t);
    }
  });
}

// observables over fluid nodes, one partial per CTA: max |v| (v = u + F/(2 rho)),
// max |u|, mass, max |rho - snap|
template <int LAT, int S, class P>
__global__ void __launch_bounds__(WT) k_wall_obs(Geo g, KParams p, const signed char* __restrict__ layer,
                                                 const typename P::Tf* __restrict__ f,
                                                 const typename P::Tr* __restrict__ rho,
                                                 const typename P::Tm* __restrict__ mu,
                                                 const typename P::Tr* __restrict__ snap, double* part,
                                                 unsigned long long* bad, long long t) {
  using Lt = Lattice<LAT>;
  constexpr int Q = LAT == 0 ? 9 : 19, D = LAT == 0 ? 2 : 3, R = Sch<S>::R;
  __shared__ double red[4][WT];
  double a0 = 0, a1 = 0, a2 = 0, a3 = 0;
  const int N = g.n;
  for_nodes(g, [&](int x, int y, int z, int n) {
    if (layer[n] != 0) return;
    double j[3] = {0, 0, 0};
    for (int i = 0; i < Q; ++i) {
      const double fi = double(f[i * N + n]);
      j[0] += Lt::ex(i) * fi;
      j[1] += Lt::ey(i) * fi;
      j[2] += Lt::ez(i) * fi;
    }
    const double rc = P::DEV ? p.rho_ref + double(rho[n]) : double(rho[n]);
    double uu = 0, vv = 0;
    for (int a = 0; a < 3; ++a) {
      double Fa = 0;
      if (a < D) {
        double gm = 0, gr = 0;
        for (int m = 1; m <= R; ++m) {
          const int pp = at(g, n, x, y, z, a == 0 ? m : 0, a == 1 ? m : 0, a == 2 ? m : 0);
          const int qq = at(g, n, x, y, z, a == 0 ? -m : 0, a == 1 ? -m : 0, a == 2 ? -m : 0);
          gm += Sch<S>::g(m) * (double(mu[pp]) - double(mu[qq]));
          gr += Sch<S>::g(m) * (double(rho[pp]) - double(rho[qq]));
        }
        Fa = -rc * gm + gr / 3.0;
      }
      const double ua = j[a] / rc, va = ua + Fa / (2.0 * rc);
      uu += ua * ua;
      vv += va * va;
    }
    a0 = fmax(a0, sqrt(vv));
    a1 = fmax(a1, sqrt(uu));
    a2 += rc;
    a3 = fmax(a3, fabs(double(rho[n]) - double(snap[n])));
    if (!(rc > 0.0)) atomicMin(bad, (unsigned long long)t);
  });
  const int tid = threadIdx.y * WX + threadIdx.x;
  red[0][tid] = a0; red[1][tid] = a1; red[2][tid] = a2; red[3][tid] = a3;
  __syncthreads();
  for (int s = WT / 2; s > 0; s >>= 1) {
    if (tid < s) {
      red[0][tid] = fmax(red[0][tid], red[0][tid + s]);
      red[1][tid] = fmax(red[1][tid], red[1][tid + s]);
      red[2][tid] += red[2][tid + s];
      red[3][tid] = fmax(red[3][tid], red[3][tid + s]);
    }
    __syncthreads();
  }
  if (tid == 0) {
    const int b = blockIdx.y * gridDim.x + blockIdx.x;
    for (int q = 0; q < 4; ++q) part[4 * b + q] = red[q][0];
  }
}

// grid over (x, row) with at most max_ctas CTAs (both axes grid-strided)
dim3 wall_grid(const Geo& g, int max_ctas) {
  const int gx = std::min((g.nx + WX - 1) / WX, max_ctas);
  const int rows = g.ny * g.nz;
  const int gy = std::max(1, std::min({(rows + WY - 1) / WY, max_ctas / gx, 65535}));
  return dim3(unsigned(gx), unsigned(gy));
}

template <int LAT, int S, class P>
cudaError_t wall_run(const WallLaunch& w, int mode, int* nblocks) {
  const Geo g{w.c.kp.nx, w.c.kp.ny, w.c.kp.nz, int(w.c.kp.n)};
  using Tr = typename P::Tr;
  using Tf = typename P::Tf;
  using Tm = typename P::Tm;
  const dim3 blk(WX, WY), grid = wall_grid(g, 1 << 20);
  cudaStream_t st = w.c.stream;
  Tr* rin = static_cast<Tr*>(const_cast<void*>(w.c.rin));  // wall layers are refreshed in place
  // Wall densities in one launch while one CTA's rounds are fewer than the launches
  // they replace are worth: 1024 nodes a layer, in FP64, whose pipe one SM has little
  // of, 128.  One launch and three, us a step: FP32 512^2 flat wall (1024 a layer)
  // 22.7 and 24.1, 256^2 (512) 14.8 and 16.2; 32^3 (2048) 24.4 and 17.8, 1800 x 100
  // (3600) 32.5 and 24.8; FP64 64^2 (128) 33.7 and 34.7, 128^2 (256) 45 and 38.5, 24^3
  // (1152) 76 and 56.
  const int *nl = w.nlist, most = std::max({nl[0], nl[1], nl[2]});
  // FP64 launches overlap except where the pass's CTAs find an SM each and are more
  // than half as many: dealt early, two share an SM and its FP64 pipe (us a step
  // overlapped and not: 28^3, 98 CTAs, 82 and 58, 32^3 98 and 60, 192^2, 144 CTAs, 63
  // and 45; 144^2, 90 CTAs, 40 and 45, 24^3 57 and 69, 34^3 98 and 108)
  const long long ctas = (long long)grid.x * grid.y;
  const bool pdl = sizeof(Tr) != 8 || 10 * ctas <= 6 * device_sms() || ctas > device_sms();
  cudaError_t e = cudaSuccess;
  if (most <= (sizeof(Tr) == 8 ? 128 : 1024)) {
    if (most > 0)
      e = launch_if_pdl(pdl, k_wall_fill<LAT, Tr>, dim3(1), 1024, 0, st, g, w.layer, w.list, nl[0], nl[1], nl[2], 0, rin);
  } else {
    for (int L = 1; L <= 3 && e == cudaSuccess; ++L)
      if (nl[L - 1] > 0)
        e = launch_if_pdl(pdl, k_wall_fill<LAT, Tr>, dim3((nl[L - 1] + 255) / 256), 256, 0, st, g, w.layer, w.list, nl[0],
                          nl[1], nl[2], L, rin);
  }
  if (e != cudaSuccess || mode == MODE_WALL_FILL) return e;
  e = launch_if_pdl(pdl, k_wall_mu<LAT, S, P>, grid, blk, 0, st, g, w.c.kp, w.layer, rin, w.mu_w, static_cast<Tm*>(w.mu));
  if (e != cudaSuccess) return e;
  if (mode == MODE_OBS) {
    const dim3 og = wall_grid(g, 4096);
    if (nblocks) *nblocks = int(og.x * og.y);
    k_wall_obs<LAT, S, P><<<og, blk, 0, st>>>(g, w.c.kp, w.layer, static_cast<const Tf*>(w.c.fin), rin,
                                             static_cast<const Tm*>(w.mu), static_cast<const Tr*>(w.c.aux.rho_snap),
                                             w.c.aux.partials, w.c.aux.bad_step, w.c.aux.t);
    return cudaGetLastError();
  }
  const int cm = mode == MODE_FIELDS ? 1 : 0;
  e = launch_if_pdl(pdl, k_wall_coll<LAT, S, P>, grid, blk, 0, st, g, w.c.kp, w.c.mrt, w.layer, static_cast<const Tf*>(w.c.fin),
                    static_cast<Tf*>(w.c.fout), rin, static_cast<const Tm*>(w.mu), w.c.aux.bad_step, w.c.aux.t, cm, w.c.fo.F,
                    w.c.fo.mu);
  if (e == cudaSuccess && mode == MODE_STEP)
    e = launch_if_pdl(pdl, k_wall_dens<LAT, P>, grid, blk, 0, st, g, w.c.kp, w.layer, static_cast<const Tf*>(w.c.fout),
                      static_cast<Tr*>(w.c.rout), w.c.aux.bad_step, w.c.aux.t + 1);
  return e;
}

template <int LAT, class P>
cudaError_t wall_by_scheme(const WallLaunch& w, int scheme, int mode, int* nb) {
  switch (scheme) {
    case S_EFDS2: return wall_run<LAT, S_EFDS2, P>(w, mode, nb);
    case S_EFDS4: return wall_run<LAT, S_EFDS4, P>(w, mode, nb);
    case S_EFDS6: return wall_run<LAT, S_EFDS6, P>(w, mode, nb);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace

cudaError_t wall_step(const WallLaunch& w, int lattice, int scheme, int prec, int mode, int* nblocks) {
  if (mode != MODE_STEP && mode != MODE_OBS && mode != MODE_FIELDS && mode != MODE_WALL_FILL)
    return cudaErrorNotSupported;
  if (lattice == 0) {
    if (prec == 0) return wall_by_scheme<0, PrecF64>(w, scheme, mode, nblocks);
    if (prec == 1) return wall_by_scheme<0, PrecF32>(w, scheme, mode, nblocks);
    return wall_by_scheme<0, PrecF32M64>(w, scheme, mode, nblocks);
  }
  if (prec == 0) return wall_by_scheme<1, PrecF64>(w, scheme, mode, nblocks);
  if (prec == 1) return wall_by_scheme<1, PrecF32>(w, scheme, mode, nblocks);
  return wall_by_scheme<1, PrecF32M64>(w, scheme, mode, nblocks);
}

}  // namespace lbmd
