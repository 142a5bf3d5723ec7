// D3Q19 FP32-deviation step as three node-parallel passes, for lattices whose
// populations stay in the L2 cache and that k_coll3d's tiles do not suit:
//
//  k_node_mu    mu = k^2 psi'(rho) - kappa lap rho (Eq. 16)
//  k_node_coll  F, collision, push streaming, one thread per node
//  k_node_rho   the next density, the sum of the populations pushed into a node
//
// k_coll3d gathers the next density while it collides, which saves reading the
// populations back (76 bytes a node) but costs it about 1200 instructions a node
// on a small lattice: two planes more per chunk of z, lanes past a ragged tile,
// exchanges through shared memory, atomics at the tiles' edges; and its CTAs of 11
// rows by 32 columns leave part of the SMs idle. Reading back from the L2 is cheap:
// 125 x 70 x 43, tau 0.8, took 42.6 us a step and takes 22 (its populations at the
// L2's rate: about 6); 64^3 39 and 17, 32^3 31 and 8.7.
#pragma once
#include "launch.cuh"
#include "step3d_mu.cuh"

namespace lbmd {

constexpr int NODE_T = 128;  // threads per block

// a node's coordinates and the offsets of its neighbours along each axis
struct Node3 {
  int n, x, y, z, nx, ny, nz, nxy;
  // mx, my: ceil(2^32 / nx), ceil(2^32 / ny): quotients at most one too large
  __device__ __forceinline__ Node3(const KParams& p, int n_, unsigned mx, unsigned my)
      : n(n_), nx(p.nx), ny(p.ny), nz(p.nz), nxy(p.nx * p.ny) {
    int r = int(__umulhi(unsigned(n), mx));
    if (r * nx > n) --r;
    x = n - r * nx;
    z = int(__umulhi(unsigned(r), my));
    if (z * ny > r) --z;
    y = r - z * ny;
  }
  __device__ __forceinline__ int dx(int d) const { return d + (x + d < 0 ? nx : (x + d >= nx ? -nx : 0)); }
  __device__ __forceinline__ int dy(int d) const { return (d + (y + d < 0 ? ny : (y + d >= ny ? -ny : 0))) * nx; }
  __device__ __forceinline__ int dz(int d) const { return (d + (z + d < 0 ? nz : (z + d >= nz ? -nz : 0))) * nxy; }
};

template <int S, bool M64>
__global__ void __launch_bounds__(NODE_T) k_node_mu(const KParams p, const unsigned mx, const unsigned my,
                                                    const float* rin, float* __restrict__ mu) {
  pdl_wait();
  constexpr int R = Sch<S>::R;
  const int n = blockIdx.x * NODE_T + threadIdx.x;
  if (n >= int(p.n)) return;
  const Node3 c(p, n, mx, my);
  const float* q = rin + n;
  const float d = q[0];
  float lap = float(3.0 * Sch<S>::l(0)) * d;
#pragma unroll
  for (int m = 1; m <= R; ++m)
    lap += float(Sch<S>::l(m)) * ((q[c.dx(m)] + q[c.dx(-m)]) + (q[c.dy(m)] + q[c.dy(-m)]) + (q[c.dz(m)] + q[c.dz(-m)]));
  mu[n] = mu_value<M64>(p, eos_f(p), MuConst<M64>(p), float(p.k2), float(p.kappa), float(p.rho_ref), d, lap);
}

// OBS: also the observables of the state being advanced (as k_coll3d's), a set per
// block into partials, and snap overwritten with that state's density deviation
template <int S, bool TAU1, bool OBS>
__global__ void __launch_bounds__(NODE_T) k_node_coll(const KParams p, const unsigned mx, const unsigned my,
                                                      const float* fin, float* __restrict__ fout,
                                                      const float* rin, const float* mu,
                                                      unsigned long long* bad, const long long t,
                                                      float* __restrict__ snap, double* __restrict__ partials) {
  pdl_wait();
  using L = Lattice<1>;
  constexpr int Q = 19, R = Sch<S>::R;
  const int N = int(p.n);
  float o_v2 = 0.f, o_u2 = 0.f, o_d = 0.f, o_m = 0.f;  // OBS: maxima (4 |v|^2, |u|^2, |rho - snap|), sum of deviations
  int o_n = 0;
  for (int n = blockIdx.x * NODE_T + threadIdx.x; n < N; n += int(gridDim.x) * NODE_T) {
    float f[Q];
  #pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = fin[i * N + n];
    const Node3 c(p, n, mx, my);
    const float d = rin[n], rc = float(p.rho_ref) + d;
    // grad rho and grad mu
    float gr[3] = {0.f, 0.f, 0.f}, gm[3] = {0.f, 0.f, 0.f};
  #pragma unroll
    for (int m = 1; m <= R; ++m) {
      const float g = float(Sch<S>::g(m));
      const int up[3] = {n + c.dx(m), n + c.dy(m), n + c.dz(m)}, dn[3] = {n + c.dx(-m), n + c.dy(-m), n + c.dz(-m)};
  #pragma unroll
      for (int a = 0; a < 3; ++a) {
        gr[a] += g * (rin[up[a]] - rin[dn[a]]);
        gm[a] += g * (mu[up[a]] - mu[dn[a]]);
      }
    }
    float j[3] = {0.f, 0.f, 0.f};
  #pragma unroll
    for (int i = 1; i < Q; i += 2) {  // e_{i+1} = -e_i for odd i
      const float s = f[i] - f[i + 1];
      const int e[3] = {L::ex(i), L::ey(i), L::ez(i)};
  #pragma unroll
      for (int a = 0; a < 3; ++a)
        if (e[a] != 0) j[a] = e[a] > 0 ? j[a] + s : j[a] - s;
    }
    if (!(rc > 0.f)) atomicMin(bad, (unsigned long long)t);
    // v = u + F / rho, F = -rho grad mu + grad rho / 3 (Eq. 12)
    const float ir = __fdividef(1.f, rc), om = float(p.omega), o1 = 1.f - om;
    float u[3], v[3];
  #pragma unroll
    for (int a = 0; a < 3; ++a) {
      u[a] = __fmul_rn(j[a], ir);  // (roundings spelled out: the same bits with and without OBS)
      v[a] = fmaf(fmaf(-rc, gm[a], gr[a] * (1.f / 3.f)), ir, u[a]);
    }
    if constexpr (OBS) {
      // 2 (u + F / (2 rho)) = u + v
      const float hx = u[0] + v[0], hy = u[1] + v[1], hz = u[2] + v[2];
      o_v2 = fmaxf(o_v2, hx * hx + hy * hy + hz * hz);
      o_u2 = fmaxf(o_u2, u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
      o_d = fmaxf(o_d, fabsf(d - snap[n]));
      snap[n] = d;
      o_m += d;
      ++o_n;
    }
    const float vv = 1.5f * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]), uu = 1.5f * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    // even and odd parts of w rho (E(v) - (1 - omega) E(u)), E(v) = +-3 e.v + 4.5 (e.v)^2 - 1.5 v.v
    const float ev0 = TAU1 ? -vv : fmaf(o1, uu, -vv);
    float s[3];
  #pragma unroll
    for (int a = 0; a < 3; ++a) s[a] = TAU1 ? v[a] : fmaf(-o1, u[a], v[a]);
    const int ox[3] = {c.dx(-1), 0, c.dx(1)}, oy[3] = {c.dy(-1), 0, c.dy(1)}, oz[3] = {c.dz(-1), 0, c.dz(1)};
    auto put = [&](int i, float val) { fout[i * N + n + ox[L::ex(i) + 1] + oy[L::ey(i) + 1] + oz[L::ez(i) + 1]] = val; };
    // the rest population carries the density less the others' shares (rounded weights)
    const float wd1 = float(L::w(1)) * d, wd2 = float(L::w(7)) * d, wd0 = fmaf(-12.f, wd1, d);
    const float wr0 = float(L::w(0)) * rc, wr1 = float(L::w(1)) * rc, wr2 = float(L::w(7)) * rc;
    put(0, TAU1 ? fmaf(wr0, ev0, wd0) : fmaf(o1, f[0], fmaf(om, wd0, wr0 * ev0)));
  #pragma unroll
    for (int i = 1; i < Q; i += 2) {
      const float wd = i < 7 ? wd1 : wd2, wr = i < 7 ? wr1 : wr2;
      const float ev = edot<L>(i, v[0], v[1], v[2]);
      float even = fmaf(4.5f * ev, ev, ev0), odd = 3.f * ev;
      if constexpr (!TAU1) {
        const float eu = edot<L>(i, u[0], u[1], u[2]);
        even = fmaf(-4.5f * o1 * eu, eu, even);
        odd = 3.f * edot<L>(i, s[0], s[1], s[2]);
      }
      const float a = TAU1 ? fmaf(wr, even, wd) : fmaf(om, wd, wr * even), b = wr * odd;
      put(i, TAU1 ? a + b : fmaf(o1, f[i], a + b));
      put(i + 1, TAU1 ? a - b : fmaf(o1, f[i + 1], a - b));
    }
    if constexpr (!OBS) break;  // one node per thread
  }
  if constexpr (OBS) {
    // a thread's few deviations are summed in FP32, the 32 sums of a warp in
    // double-float (as FP64 would, off its pipe), the warps' by one thread in FP64
    __shared__ float red[3][NODE_T / 32];
    __shared__ double mass[NODE_T / 32];
    __shared__ int cnt[NODE_T / 32];
    Df m{o_m, 0.f};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      o_v2 = fmaxf(o_v2, __shfl_xor_sync(0xffffffffu, o_v2, o));
      o_u2 = fmaxf(o_u2, __shfl_xor_sync(0xffffffffu, o_u2, o));
      o_d = fmaxf(o_d, __shfl_xor_sync(0xffffffffu, o_d, o));
      m = df_add(m, Df{__shfl_xor_sync(0xffffffffu, m.h, o), __shfl_xor_sync(0xffffffffu, m.l, o)});
      o_n += __shfl_xor_sync(0xffffffffu, o_n, o);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) red[0][w] = o_v2, red[1][w] = o_u2, red[2][w] = o_d, mass[w] = double(m.h) + double(m.l), cnt[w] = o_n;
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int k = 0; k < NODE_T / 32; ++k) {
        o_v2 = fmaxf(o_v2, red[0][k]);
        o_u2 = fmaxf(o_u2, red[1][k]);
        o_d = fmaxf(o_d, red[2][k]);
        sum += double(cnt[k]) * p.rho_ref + mass[k];
      }
      double* out = partials + 4 * blockIdx.x;
      out[0] = 0.5 * sqrt(double(o_v2));
      out[1] = sqrt(double(o_u2));
      out[2] = sum;
      out[3] = double(o_d);
    }
  }
}

__global__ void __launch_bounds__(NODE_T) k_node_rho(const KParams p, const float* f, float* __restrict__ rho,
                                                     unsigned long long* bad, const long long t1) {
  pdl_wait();
  const int n = blockIdx.x * NODE_T + threadIdx.x, N = int(p.n);
  if (n >= N) return;
  float a[3] = {f[n], 0.f, 0.f};
#pragma unroll
  for (int i = 1; i < 19; i += 2) a[i / 2 % 3] += f[i * N + n] + f[(i + 1) * N + n];
  const float d = a[0] + (a[1] + a[2]);
  rho[n] = d;
  if (!(float(p.rho_ref) + d > 0.f)) atomicMin(bad, (unsigned long long)t1);
}

}  // namespace lbmd
