// D3Q19 FP32-deviation steps at tau = 1 on four moments instead of nineteen
// populations.
//
// With omega = 1 a post-collision population depends on rho and on v = u + F /
// rho alone, and the next step needs only sum f_i and sum e_i f_i of the
// streamed populations (Eq. 1, 6-8).  Between the first and the last step of
// a call the state is therefore the density deviation and the momentum j =
// sum e_i f_i (16 bytes per node instead of 80), advanced by
//
//  k_mom_gather  rho, j of the call's initial populations (once per call)
//  k_mom_mu      mu of every node (each step)
//  k_mom3d       F, v, the nineteen post-collision values of every node on
//                chip, and from them the rho and j of the next step
//  k_mom_expand  the populations of the final state (once per call), pushed
//                from the state before it
//
// A step moves 44 bytes per node (rho in, mu out; rho, mu, j in, rho, j out)
// instead of 172, and skips the stores of populations that nothing reads.  At
// 256^3 (EFDS6) a step takes 0.31 ms against 0.608 for the mu and collision
// passes on populations; gather and expand together cost 0.63 ms per call.
//
// Fields (float): element (x, y, z) at z PL + y LX + 4 + x, LX = 4 ceil(nx /
// 4) + 8: rows start at a 16-byte boundary for every nx.  rho and mu rows
// carry periodic copies of their ends (x = -4 .. -1 and nx .. nx + 3), so
// that no stencil wraps in x; what lies past them is zero.
#pragma once
#include "lbm_device.cuh"
#include "launch.cuh"
#include "pack2.cuh"
#include "step3d_mu.cuh"

namespace lbmd {

// the mu pass of CFDS8: central second derivative of order eight (Sec. 2.3)
constexpr int S_LAP8 = 16;
template <>
struct Sch<S_LAP8> {
  static constexpr int R = 4;
  static constexpr bool ISO = false, GF = false;
  __host__ __device__ static constexpr double g(int) { return 0.0; }
  __host__ __device__ static constexpr double l(int m) {
    return m == 0 ? -205.0 / 72.0 : (m == 1 ? 1.6 : (m == 2 ? -0.2 : (m == 3 ? 8.0 / 315.0 : -1.0 / 560.0)));
  }
};

struct MomGeo {
  int LX, PL;    // row and plane strides
  int P;         // field stride (floats)
  int TW, nt;    // columns per tile of k_mom3d (a multiple of 4, <= 64), tiles
  int RB, nb;    // rows per band, bands
};

// The packed constants of a step.  Kernel parameters, not literals: a packed
// instruction takes no immediate, and the compiler otherwise builds each pair
// in registers again at every use (85 integer instructions per node, moves
// mostly; 35 with them here and the shifted halves added as scalars).
struct MomConst {
  float2 h[3], g[3];  // first-derivative weights / 3 and weights
  float2 m1, c45, m15, m12, w0, w1, w2, t1, t2, n1, n2;  // -1, 4.5, -1.5, -12, 1/3, 1/18, 1/36, +-3/18, +-3/36
};

__device__ __forceinline__ float2 subk(const MomConst& k, float2 a, float2 b) { return fma2(k.m1, b, a); }

// Post-collision populations (deviations) of two nodes at tau = 1: P_i = w_i
// (drho + rho (3 e.v + 4.5 (e.v)^2 - 1.5 v.v)); the opposite directions of a
// pair share everything but the sign of the linear term.
struct Post2 {
  const MomConst& k;
  float2 vx, vy, vz, nvv;                // v, -1.5 v.v
  float2 b1, b2, r1, r2, t1, t2, n1, n2; // w drho, w rho, +-3 w rho of the axes (1/18) and the diagonals (1/36)
  // d, r: density deviation and density (both 0 for a node that is not there)
  __device__ __forceinline__ Post2(const MomConst& k_, float2 d, float2 r, float2 x, float2 y, float2 z)
      : k(k_), vx(x), vy(y), vz(z) {
    nvv = mul2(k.m15, fma2(x, x, fma2(y, y, mul2(z, z))));
    b1 = mul2(k.w1, d);
    b2 = mul2(k.w2, d);
    r1 = mul2(k.w1, r);
    r2 = mul2(k.w2, r);
    t1 = mul2(k.t1, r);
    t2 = mul2(k.t2, r);
    n1 = mul2(k.n1, r);
    n2 = mul2(k.n2, r);
  }
  // drho less what the other eighteen carry of it (12 b1, the diagonals'
  // weight being half the axes'): with rounded weights the populations would
  // sum to 1.0000000xx drho, a drift of 1e-8 per step
  __device__ __forceinline__ float2 rest(float2 d, float2 r) const {
    return fma2(mul2(k.w0, r), nvv, fma2(k.m12, b1, d));
  }
  __device__ __forceinline__ void axis(float2 E, float2& p, float2& m) const {
    const float2 b = fma2(r1, fma2(k.c45, mul2(E, E), nvv), b1);
    p = fma2(t1, E, b);
    m = fma2(n1, E, b);
  }
  __device__ __forceinline__ void diag(float2 E, float2& p, float2& m) const {
    const float2 b = fma2(r2, fma2(k.c45, mul2(E, E), nvv), b2);
    p = fma2(t2, E, b);
    m = fma2(n2, E, b);
  }
};

// ------------------------------------------------------------------ gather
// One thread per element of a padded row: the moments at the lattice's nodes,
// the periodic copies of rho beside them, zeros in the rest of every field
// (rb, mu, jb and, with a compact scheme, the three fields acc are the step's
// other buffers).  A row's last pair of nodes reads one element of it where nx is
// odd; its populations are masked by a factor of zero, so it has to be finite.
__global__ void __launch_bounds__(256) k_mom_gather(const KParams p, const MomGeo g, const float* __restrict__ f,
                                                    const float* __restrict__ rho, float* __restrict__ ra,
                                                    float* __restrict__ ja, float* __restrict__ rb,
                                                    float* __restrict__ mu, float* __restrict__ jb,
                                                    float* __restrict__ acc, unsigned long long* bad, long long t) {
  using L = Lattice<1>;
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e >= g.PL * p.nz) return;
  const int row = e / g.LX, x = e - row * g.LX - 4, nx = p.nx, N = int(p.n);
  if (x >= 0 && x < nx) {
    const float* fn = f + row * nx + x;
    float v[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) v[i] = __ldcs(fn + i * N);
    const float r = rho[row * nx + x];
    float jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
    for (int i = 1; i < 19; i += 2) {
      const float d = v[i] - v[i + 1];
      if (L::ex(i) != 0) jx = L::ex(i) > 0 ? jx + d : jx - d;
      if (L::ey(i) != 0) jy = L::ey(i) > 0 ? jy + d : jy - d;
      if (L::ez(i) != 0) jz = L::ez(i) > 0 ? jz + d : jz - d;
    }
    ra[e] = r;
    ja[e] = jx;
    ja[e + g.P] = jy;
    ja[e + 2 * g.P] = jz;
    if (!(float(p.rho_ref) + r > 0.f)) atomicMin(bad, (unsigned long long)t);
  } else {
    const bool ghost = x < nx + 4;
    ra[e] = ghost ? rho[row * nx + (x < 0 ? x + nx : x - nx)] : 0.f;
    rb[e] = 0.f;
    mu[e] = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      ja[e + a * g.P] = jb[e + a * g.P] = 0.f;
      if (acc) acc[e + a * g.P] = 0.f;
    }
  }
}

// periodic copies of a row's node x beside the row (o: its element)
__device__ __forceinline__ void mom_ghost(float* fld, int o, int x, int nx, float v) {
  if (x < 4) fld[o + nx] = v;
  if (x >= nx - 4) fld[o - nx] = v;
}

// ------------------------------------------------------------------ mu pass
// A thread owns four x-adjacent nodes and marches through zc planes: z
// neighbours in a register queue, x and y neighbours by 16-byte loads that
// hit L1 (the rows of a CTA are adjacent).  No shared memory and no barrier:
// the padded rows need no wrap in x and the queue's next plane is loaded one
// plane ahead.  (__ldca: an ordinary load that the compiler leaves in its place;
// left to it, EFDS6 takes 0.060 ms at 256^3.)  At 256^3 0.058 ms (the zeroing mu pass
// of the population steps takes 0.060), bound by issue (69% of cycles).
template <int S, bool M64>
__global__ void __launch_bounds__(256) k_mom_mu(const KParams p, const MomGeo g, const float* rin,
                                                float* __restrict__ mu, const int zc) {
  pdl_wait();
  constexpr int R = Sch<S>::R;
  const int nx4 = (p.nx + 3) >> 2;
  const int c = blockIdx.x * 256 + threadIdx.x;
  if (c >= nx4 * p.ny) return;
  const int y = c / nx4, x = 4 * (c - y * nx4), nz = p.nz, ny = p.ny, nx = p.nx;
  const int z0 = blockIdx.y * zc, z1 = min(z0 + zc, nz);
  const int col = y * g.LX + 4 + x;
  int yo[2 * R];
#pragma unroll
  for (int m = 1; m <= R; ++m) {
    yo[m - 1] = wrapi(y + m, ny) * g.LX + 4 + x;
    yo[R + m - 1] = wrapi(y - m, ny) * g.LX + 4 + x;
  }
  auto ld = [&](int zo, int o) { return __ldca(reinterpret_cast<const float4*>(rin + zo + o)); };
  const float k2 = float(p.k2), kap = float(p.kappa), rref = float(p.rho_ref);
  const EosF ef = eos_f(p);
  const MuConst<M64> mc(p);
  float4 q[2 * R + 1];
#pragma unroll
  for (int d = 1; d <= 2 * R; ++d) q[d] = ld(wrapi(z0 - R - 1 + d, nz) * g.PL, col);
  float4 nxt = ld(wrapi(z0 + R, nz) * g.PL, col);
  for (int z = z0; z < z1; ++z) {
#pragma unroll
    for (int d = 0; d < 2 * R; ++d) q[d] = q[d + 1];
    q[2 * R] = nxt;
    const int zo = z * g.PL;
    if (z + 1 < z1) nxt = ld(wrapi(z + R + 1, nz) * g.PL, col);
    const float4 lo = ld(zo, col - 4), hi = ld(zo, col + 4), c4 = q[R];
    const float row[12] = {lo.x, lo.y, lo.z, lo.w, c4.x, c4.y, c4.z, c4.w, hi.x, hi.y, hi.z, hi.w};
    float2 la = mul2(f2(float(3.0 * Sch<S>::l(0))), make_float2(c4.x, c4.y));
    float2 lb = mul2(f2(float(3.0 * Sch<S>::l(0))), make_float2(c4.z, c4.w));
#pragma unroll
    for (int m = 1; m <= R; ++m) {
      const float4 a = ld(zo, yo[m - 1]), b = ld(zo, yo[R + m - 1]), e = q[R + m], d = q[R - m];
      const float2 ya = add2(add2(make_float2(a.x, a.y), make_float2(b.x, b.y)),
                             add2(make_float2(e.x, e.y), make_float2(d.x, d.y)));
      const float2 yb = add2(add2(make_float2(a.z, a.w), make_float2(b.z, b.w)),
                             add2(make_float2(e.z, e.w), make_float2(d.z, d.w)));
      la = fma2(f2(float(Sch<S>::l(m))), add2(make_float2(row[4 + m] + row[4 - m], row[5 + m] + row[5 - m]), ya), la);
      lb = fma2(f2(float(Sch<S>::l(m))), add2(make_float2(row[6 + m] + row[6 - m], row[7 + m] + row[7 - m]), yb), lb);
    }
    const float lap[4] = {la.x, la.y, lb.x, lb.y};
    float res[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) res[k] = mu_value<M64>(p, ef, mc, k2, kap, rref, row[4 + k], lap[k]);
    float* out = mu + zo + col;
    if (x + 4 <= nx) *reinterpret_cast<float4*>(out) = make_float4(res[0], res[1], res[2], res[3]);
    if (x < 4 || x + 8 > nx) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (x + k < nx) {
          out[k] = res[k];
          mom_ghost(mu, zo + col + k, x + k, nx, res[k]);
        }
    }
  }
}

// ------------------------------------------------------------------ moment step
// A CTA owns the columns of one tile (up to 64, two adjacent ones per lane)
// and the rows of one band (up to W - 3), and marches through zc planes (plus
// the one before and the one after).  Warps 0 .. W - 2 hold the band's rows
// and the row beyond either side; the last warp holds the column beyond
// either side of the tile for all of them.  So every population that arrives
// at a node of the tile is computed in the CTA: no atomics, no corner pass,
// at (W - 3) / W of the warps' work.  Two nodes per lane make every
// floating-point instruction a packed one (fma.f32x2 and kin).
//  - The density and mu planes are staged in shared memory by 16-byte
//    asynchronous copies two planes ahead (a ring of 2 R + 3 planes).
//  - Populations that move along the row go by shuffle; those that change
//    rows through shared memory, summed where they land together (P, Q: the
//    three in-plane ones as their sum and the difference of the diagonals),
//    double-buffered, so that one CTA barrier per plane covers both the
//    exchange and the staged planes.
//  - Those that change planes stay in registers until their plane completes.
// Bound by shared-memory wavefronts and issue in turn (each about half of the
// cycles: the warps leave the barrier together): 0.252 ms at 256^3, 0.109 at
// 192^3 (16 warps, 121 registers; 12 warps 0.289; 18 and 20 warps do not fit
// their registers and take twice as long).
template <int S, int W>
struct MomShape {
  static constexpr int R = Sch<S>::R;
  static constexpr int NT = 32 * W, ROWS = W - 1, BAND = W - 3;
  static constexpr int GW = 72, GH = ROWS + 2 * R, NS = 2 * R + 3, plane = GW * GH;
  static constexpr int XB = 8 * ROWS * 64;  // floats of one exchange buffer
  static constexpr int EB = 5 * 2 * ROWS;   // of one edge-column buffer
  static constexpr size_t bytes = size_t(2 * NS * plane + 2 * XB + 2 * EB) * 4;
  static constexpr int KC = (GH * (GW / 4) + NT - 1) / NT;
};

// What a thread of the moment step holds and does once F and v of its two nodes
// are known: spread() forms their populations and hands on what leaves, collect()
// (behind a CTA barrier) adds up what arrives and stores the plane before.
template <int W>
struct MomCell {
  static constexpr int ROWS = W - 1, XB = 8 * ROWS * 64, EB = 5 * 2 * ROWS, XK = ROWS * 32;
  // main warps: row w (0: the one below the band), columns 2 lane and 2 lane +
  // 1; the last warp: lane r holds row r's columns beyond the tile (x: left, y: right)
  int lane, w, VW, VH, row, gx0, gx1;
  bool edge, live, tgt;  // live: a row that is collided; tgt: a row of the band
  bool in0, in1, elane, gh, ok;
  unsigned gy, oj0, oj1;
  float2 mask;
  float mL, mR, ex, ey, sg;
  float2 *xw;  // this row's exchange values
  float* ew;
  float2 R0, X0, Sp, Xp, Sm, Xm;
  float2 aR, aX, aY, aZ;  // target plane pc - 1
  float2 bS, bX, bY;      // target plane pc: from plane pc - 1

  __device__ __forceinline__ MomCell(const KParams& p, const MomGeo& g, float* s_x, float* s_e) {
    const int nx = p.nx, ny = p.ny, x0 = blockIdx.x * g.TW, y0 = blockIdx.y * g.RB;
    lane = threadIdx.x & 31;
    w = threadIdx.x >> 5;
    VW = min(g.TW, nx - x0);
    VH = min(g.RB, ny - y0);
    edge = w == ROWS;
    row = edge ? min(lane, VH + 1) : w;
    live = edge || w <= VH + 1;
    tgt = !edge && w >= 1 && w <= VH;
    gy = wrapn(y0 - 1 + row, ny) * g.LX + 4;
    gx0 = edge ? (x0 == 0 ? nx - 1 : x0 - 1) : x0 + 2 * lane;
    gx1 = edge ? (x0 + VW == nx ? 0 : x0 + VW) : gx0 + 1;
    oj0 = gy + gx0;
    oj1 = gy + gx1;
    in0 = edge || 2 * lane < VW;
    in1 = edge || 2 * lane + 1 < VW;
    mask = make_float2(in0 ? 1.f : 0.f, in1 ? 1.f : 0.f);
    mL = lane == 0 ? 0.f : 1.f;  // what arrives by shuffle
    mR = lane == 31 ? 0.f : 1.f;
    // the edge lanes of a row take the populations of the columns beyond: the
    // first lane into its first node, lane rl into the tile's last node
    const int rl = (VW - 1) >> 1;
    elane = lane == 0 || lane == rl;
    const bool esec = lane != 0 && ((VW - 1) & 1) != 0;
    ex = esec ? 0.f : 1.f;
    ey = esec ? 1.f : 0.f;
    sg = lane == 0 ? 1.f : -1.f;
    gh = gx0 < 4 || gx0 + 1 >= nx - 4;  // rho goes beside the row too
    ok = true;
    xw = reinterpret_cast<float2*>(s_x) + row * 32 + lane;
    ew = s_e + (edge ? row : (lane == 0 ? 0 : ROWS) + row);
    aR = aX = aY = aZ = bS = bX = bY = f2(0.f);
  }
  // two nodes of a field at offset zo of a plane
  __device__ __forceinline__ float2 load(const float* q, unsigned zo) const {
    if (edge) return make_float2(q[zo + oj0], q[zo + oj1]);
    return in0 ? *reinterpret_cast<const float2*>(q + (zo + oj0)) : f2(0.f);
  }
  __device__ __forceinline__ void spread(const MomConst& kc, float2 d, float2 r, float2 vx, float2 vy, float2 vz) {
    auto sub = [&](float2 a, float2 b) { return fma2(kc.m1, b, a); };
    const float2 dm = mul2(d, mask), rm = mul2(r, mask);
    const Post2 ps(kc, dm, rm, vx, vy, vz);
    float2 f7, f8, f9, f10;
    ps.diag(add2(vx, vy), f7, f8);
    ps.diag(sub(vx, vy), f9, f10);
    if (!edge) {
      // the sum and the difference of a right-moving and a left-moving
      // population at their targets in the row (nothing enters at the row's
      // ends: that comes from the edge warp); scalar, since the shifted
      // halves lie in two pairs
      auto meet = [&](float2 a, float2 b, float2& s, float2& f) {
        const float qa = __shfl_up_sync(0xffffffffu, a.y, 1), qb = __shfl_down_sync(0xffffffffu, b.x, 1);
        s = make_float2(fmaf(qa, mL, b.y), fmaf(qb, mR, a.x));
        f = make_float2(fmaf(qa, mL, -b.y), fmaf(qb, -mR, a.x));
      };
      float2 s, f;
      {
        float2 f3, f4;
        ps.axis(vy, f3, f4);
        meet(f7, f10, s, f);
        xw[0] = add2(f3, s);
        xw[XK] = f;
        meet(f9, f8, s, f);
        xw[4 * XK] = add2(f4, s);
        xw[5 * XK] = f;
      }
      {
        float2 f15, f16, f17, f18;
        ps.diag(add2(vy, vz), f15, f16);
        ps.diag(sub(vy, vz), f17, f18);
        xw[2 * XK] = f15;
        xw[3 * XK] = f17;
        xw[6 * XK] = f18;
        xw[7 * XK] = f16;
      }
      if (tgt) {
        float2 a, b;
        ps.axis(vx, a, b);
        meet(a, b, s, X0);
        R0 = add2(ps.rest(dm, rm), s);
        float2 f11, f12, f13, f14;
        ps.diag(add2(vx, vz), f11, f12);
        ps.diag(sub(vx, vz), f13, f14);
        ps.axis(vz, a, b);
        meet(f11, f14, s, Xp);
        Sp = add2(a, s);
        meet(f13, f12, s, Xm);
        Sm = add2(b, s);
      }
    } else if (lane <= VH + 1) {
      // left column: the right-moving populations; right column: the left-moving ones
      float2 f1, f2_, f11, f12, f13, f14;
      ps.axis(vx, f1, f2_);
      ps.diag(add2(vx, vz), f11, f12);
      ps.diag(sub(vx, vz), f13, f14);
      ew[0] = f1.x;            ew[ROWS] = f2_.y;
      ew[2 * ROWS] = f11.x;    ew[3 * ROWS] = f14.y;
      ew[4 * ROWS] = f13.x;    ew[5 * ROWS] = f12.y;
      ew[6 * ROWS] = f7.x;     ew[7 * ROWS] = f10.y;
      ew[8 * ROWS] = f9.x;     ew[9 * ROWS] = f8.y;
    }
  }
  // plane pc's neighbours have spread; plane pc - 1 >= z0 is complete
  __device__ __forceinline__ void collect(const MomConst& kc, int pc, int z0, int PL, int nx, float rref, float* rout,
                                          float* jout, float* q1, float* q2) {
    if (tgt) {
      const float2 Pu = xw[-32], Qu = xw[XK - 32], u15 = xw[2 * XK - 32], u17 = xw[3 * XK - 32];
      const float2 Pd = xw[4 * XK + 32], Qd = xw[5 * XK + 32], d18 = xw[6 * XK + 32], d16 = xw[7 * XK + 32];
      R0 = add2(R0, add2(Pu, Pd));
      X0 = add2(X0, add2(Qu, Qd));
      float2 Y0 = subk(kc, Pu, Pd);
      Sp = add2(Sp, add2(u15, d18));
      Sm = add2(Sm, add2(u17, d16));
      const float2 Yp = subk(kc, u15, d18), Ym = subk(kc, u17, d16);
      if (elane) {
        // the columns beyond the tile: from the left one into the first node,
        // from the right one into the last
        const float a0 = ew[0], ap = ew[2 * ROWS], am = ew[4 * ROWS], du = ew[6 * ROWS - 1], dd = ew[8 * ROWS + 1];
        const float in = a0 + (du + dd), df = du - dd, si0 = sg * in, sp = sg * ap, sn = sg * am;
        R0.x = fmaf(ex, in, R0.x);   R0.y = fmaf(ey, in, R0.y);
        X0.x = fmaf(ex, si0, X0.x);  X0.y = fmaf(ey, si0, X0.y);
        Y0.x = fmaf(ex, df, Y0.x);   Y0.y = fmaf(ey, df, Y0.y);
        Sp.x = fmaf(ex, ap, Sp.x);   Sp.y = fmaf(ey, ap, Sp.y);
        Xp.x = fmaf(ex, sp, Xp.x);   Xp.y = fmaf(ey, sp, Xp.y);
        Sm.x = fmaf(ex, am, Sm.x);   Sm.y = fmaf(ey, am, Sm.y);
        Xm.x = fmaf(ex, sn, Xm.x);   Xm.y = fmaf(ey, sn, Xm.y);
      }
      const int zt = pc - 1;
      if (zt >= z0 && in0) {
        const float2 r = add2(aR, Sm), jx = add2(aX, Xm), jy = add2(aY, Ym), jz = subk(kc, aZ, Sm);
        const unsigned o = unsigned(zt) * PL + oj0;
        ok = ok && rref + r.x > 0.f;
        if (in1) {
          ok = ok && rref + r.y > 0.f;
          *reinterpret_cast<float2*>(rout + o) = r;
          *reinterpret_cast<float2*>(jout + o) = jx;
          *reinterpret_cast<float2*>(q1 + o) = jy;
          *reinterpret_cast<float2*>(q2 + o) = jz;
        } else {
          rout[o] = r.x;
          jout[o] = jx.x;
          q1[o] = jy.x;
          q2[o] = jz.x;
        }
        if (gh) {
          mom_ghost(rout, int(o), gx0, nx, r.x);
          if (in1) mom_ghost(rout, int(o) + 1, gx0 + 1, nx, r.y);
        }
      }
      aR = add2(R0, bS);
      aX = add2(X0, bX);
      aY = add2(Y0, bY);
      aZ = bS;
      bS = Sp;
      bX = Xp;
      bY = Yp;
    }
  }
  // the other exchange buffer (par: which one this was)
  __device__ __forceinline__ void flip(int par) {
    xw += par ? -XB / 2 : XB / 2;
    ew += par ? -EB : EB;
  }
};

template <int S, int W>
__global__ void __launch_bounds__(32 * W, 1) k_mom3d(const KParams p, const MomGeo g, const float* rin,
                                                     const float* muf, const float* jin,
                                                     float* __restrict__ rout, float* __restrict__ jout,
                                                     unsigned long long* bad, const long long t, const int zc,
                                                     const __grid_constant__ MomConst kc) {
  using Sh = MomShape<S, W>;
  constexpr int R = Sh::R, GW = Sh::GW, NS = Sh::NS, ROWS = Sh::ROWS, NT = Sh::NT;
  extern __shared__ __align__(16) float sm_mom[];
  constexpr int FLD = NS * Sh::plane;           // floats of one field's ring
  float* s_x = sm_mom + 2 * FLD;
  float* s_e = s_x + 2 * Sh::XB;
  const int tid = threadIdx.x, lane = tid & 31;
  const int nx = p.nx, ny = p.ny, nz = p.nz, LX = g.LX, PL = g.PL;
  const int x0 = blockIdx.x * g.TW, y0 = blockIdx.y * g.RB;
  const int VW = min(g.TW, nx - x0), VH = min(g.RB, ny - y0);
  const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, nz);
  const int pc0 = z0 - 1, pc1 = z1;
  for (int k = tid; k < 2 * FLD; k += NT) sm_mom[k] = 0.f;
  __syncthreads();
  // staging: each thread's chunks of a plane (rows y0 - 1 - R .., columns x0 - 4 ..)
  int soff[Sh::KC];
  unsigned goff[Sh::KC];
#pragma unroll
  for (int k = 0; k < Sh::KC; ++k) {
    const int e = tid + k * NT, ry = e / (GW / 4), cj = 4 * (e - ry * (GW / 4));
    const bool in = ry < VH + 2 + 2 * R && x0 + cj + 4 <= LX;
    soff[k] = in ? ry * GW + cj : -1;
    goff[k] = in ? wrapn(y0 - 1 - R + ry, ny) * LX + x0 + cj : 0;
  }
  auto issue = [&](int q, int slot) {  // slot: offset of the ring slot
    if (q <= pc1 + R) {
      const unsigned zo = wrapi(q, nz) * PL;
#pragma unroll
      for (int k = 0; k < Sh::KC; ++k)
        if (soff[k] >= 0) {
          cpa16(sm_mom + slot + soff[k], rin + (zo + goff[k]));
          cpa16(sm_mom + FLD + slot + soff[k], muf + (zo + goff[k]));
        }
    }
  };
  MomCell<W> cell(p, g, s_x, s_e);
  const bool edge = cell.edge, live = cell.live;
  const int sc0 = edge ? 3 : 4 + 2 * lane;     // first node's column in a staged row
  const int dsc = edge ? 1 + VW : 1;           // to the second node's
  const float rref = float(p.rho_ref);

  pdl_wait();
  // planes pc0 - R .. pc0 + R (one group), then pc0 + R + 1
  for (int q = pc0 - R; q <= pc0 + R; ++q) issue(q, (q - (pc0 - R)) * Sh::plane);
  cpa_commit();
  issue(pc0 + R + 1, (2 * R + 1) * Sh::plane);
  cpa_commit();
  int si = (2 * R + 2) * Sh::plane;  // slot of the next plane issued
  const int smine = (cell.row + R) * GW + sc0;
  int so[2 * R + 1];  // this thread's first node in planes pc - R .. pc + R
#pragma unroll
  for (int d = 0; d <= 2 * R; ++d) so[d] = d * Sh::plane + smine;
  const float *j1 = jin + g.P, *j2 = jin + 2 * g.P;
  float *q1 = jout + g.P, *q2 = jout + 2 * g.P;
  float2 jn[3];
  auto ldj = [&](int pc) {
    const unsigned zo = wrapi(pc, nz) * PL;
    jn[0] = cell.load(jin, zo);
    jn[1] = cell.load(j1, zo);
    jn[2] = cell.load(j2, zo);
  };
  jn[0] = jn[1] = jn[2] = f2(0.f);
  if (live) ldj(pc0);
  cpa_wait_n<1>();
  __syncthreads();
  for (int pc = pc0; pc <= pc1; ++pc) {
    issue(pc + R + 2, si);
    cpa_commit();
    si = si == (NS - 1) * Sh::plane ? 0 : si + Sh::plane;
    if (live) {
      // F_a = rho_a / 3 - rho mu_a (Eq. 12), the third folded into the stencil of rho
      float2 gr[3], gm[3], d;
      auto sub = [&](float2 a, float2 b) { return fma2(kc.m1, b, a); };
      if (!edge) {
        auto two = [&](int o) { return *reinterpret_cast<const float2*>(sm_mom + o); };
        auto grad = [&](int f, const float2* s, float2* o, float2& mid) {
          const float2 b = two(so[R] + f - 2), c = two(so[R] + f), e = two(so[R] + f + 2);
          mid = c;
          o[0] = mul2(s[0], make_float2(c.y - b.y, e.x - c.x));
          if constexpr (R >= 2) o[0] = fma2(s[1], sub(e, b), o[0]);
          if constexpr (R >= 3) {
            const float2 a = two(so[R] + f - 4), h = two(so[R] + f + 4);
            o[0] = fma2(s[2], make_float2(e.y - a.y, h.x - b.x), o[0]);
          }
          o[1] = mul2(s[0], sub(two(so[R] + f + GW), two(so[R] + f - GW)));
          o[2] = mul2(s[0], sub(two(so[R + 1] + f), two(so[R - 1] + f)));
#pragma unroll
          for (int m = 2; m <= R; ++m) {
            o[1] = fma2(s[m - 1], sub(two(so[R] + f + m * GW), two(so[R] + f - m * GW)), o[1]);
            o[2] = fma2(s[m - 1], sub(two(so[R + m] + f), two(so[R - m] + f)), o[2]);
          }
        };
        grad(FLD, kc.g, gm, d);
        grad(0, kc.h, gr, d);
      } else {
        auto two = [&](int o) { return make_float2(sm_mom[o], sm_mom[o + dsc]); };
        auto grad = [&](int f, const float2* s, float2* o, float2& mid) {
          mid = two(so[R] + f);
          o[0] = o[1] = o[2] = f2(0.f);
#pragma unroll
          for (int m = 1; m <= R; ++m) {
            o[0] = fma2(s[m - 1], sub(two(so[R] + f + m), two(so[R] + f - m)), o[0]);
            o[1] = fma2(s[m - 1], sub(two(so[R] + f + m * GW), two(so[R] + f - m * GW)), o[1]);
            o[2] = fma2(s[m - 1], sub(two(so[R + m] + f), two(so[R - m] + f)), o[2]);
          }
        };
        grad(FLD, kc.g, gm, d);
        grad(0, kc.h, gr, d);
      }
      const float2 r = add2(f2(rref), d), nr2 = mul2(kc.m1, r);
      const float2 ir = make_float2(__fdividef(1.f, r.x), __fdividef(1.f, r.y));
      const float2 vx = mul2(add2(jn[0], fma2(nr2, gm[0], gr[0])), ir);
      const float2 vy = mul2(add2(jn[1], fma2(nr2, gm[1], gr[1])), ir);
      const float2 vz = mul2(add2(jn[2], fma2(nr2, gm[2], gr[2])), ir);
      if (pc < pc1) ldj(pc + 1);
      cell.spread(kc, d, r, vx, vy, vz);
    }
    cpa_wait_n<1>();
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 2 * R; ++k) so[k] = so[k + 1];
    so[2 * R] = so[2 * R] == (NS - 1) * Sh::plane + smine ? smine : so[2 * R] + Sh::plane;
    if (cell.tgt) cell.collect(kc, pc, z0, PL, nx, rref, rout, jout, q1, q2);
    cell.flip((pc - pc0) & 1);
  }
  if (!cell.ok) atomicMin(bad, (unsigned long long)(t + 1));
}

// The same with F / rho from the line solves of a compact scheme (acc: three
// fields): nothing is staged but the exchange, so two planes' loads (seven
// fields of the thread's own nodes) are all that is in flight.  192^3: 0.088 ms,
// 230 instructions per node at 52% issue; 24 warps of 80 registers, or two CTAs of
// 12, spill and take half as long again.
template <int W>
__global__ void __launch_bounds__(32 * W, 1) k_mom3d_acc(const KParams p, const MomGeo g, const float* rin,
                                                         const float* acc, const float* jin,
                                                         float* __restrict__ rout, float* __restrict__ jout,
                                                         unsigned long long* bad, const long long t, const int zc,
                                                         const __grid_constant__ MomConst kc) {
  extern __shared__ __align__(16) float sm_mom[];
  MomCell<W> cell(p, g, sm_mom, sm_mom + 2 * MomCell<W>::XB);
  const int nx = p.nx, nz = p.nz, PL = g.PL, P = g.P;
  const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, nz), pc0 = z0 - 1, pc1 = z1;
  const float rref = float(p.rho_ref);
  float *q1 = jout + P, *q2 = jout + 2 * P;
  float2 n[7];  // the next plane's rho, j, F / rho
  auto ld = [&](int pc) {
    const unsigned zo = wrapi(pc, nz) * PL;
    n[0] = cell.load(rin, zo);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      n[1 + a] = cell.load(jin + a * P, zo);
      n[4 + a] = cell.load(acc + a * P, zo);
    }
  };
  pdl_wait();
  if (cell.live) ld(pc0);
  for (int pc = pc0; pc <= pc1; ++pc) {
    if (cell.live) {
      const float2 d = n[0], r = add2(f2(rref), d);
      const float2 ir = make_float2(__fdividef(1.f, r.x), __fdividef(1.f, r.y));
      const float2 vx = fma2(n[1], ir, n[4]), vy = fma2(n[2], ir, n[5]), vz = fma2(n[3], ir, n[6]);
      if (pc < pc1) ld(pc + 1);
      cell.spread(kc, d, r, vx, vy, vz);
    }
    __syncthreads();
    if (cell.tgt) cell.collect(kc, pc, z0, PL, nx, rref, rout, jout, q1, q2);
    cell.flip((pc - pc0) & 1);
  }
  if (!cell.ok) atomicMin(bad, (unsigned long long)(t + 1));
}

// ------------------------------------------------------------------ expand
// The populations after the last step, pushed from the state before it (rin,
// muf, jin; with a compact scheme muf holds F / rho, three fields), and the last density rlast copied into the unpadded field.  One
// thread per node, stencils through L1: bound by the 76-byte stores.
template <int S>
__global__ void __launch_bounds__(256) k_mom_expand(const KParams p, const MomGeo g, const float* __restrict__ rin,
                                                    const float* __restrict__ muf, const float* __restrict__ jin,
                                                    const float* __restrict__ rlast, float* __restrict__ fout,
                                                    float* __restrict__ rout) {
  using L = Lattice<1>;
  constexpr int R = Sch<S>::R;
  const int nx = p.nx, ny = p.ny, nz = p.nz, N = int(p.n), NXY = nx * ny;
  const int n = blockIdx.x * 256 + threadIdx.x;
  if (n >= N) return;
  const int row = n / nx, x = n - row * nx, z = row / ny, y = row - z * ny;
  const int o = z * g.PL + y * g.LX + 4 + x;
  const float d = __ldg(rin + o), r = float(p.rho_ref) + d;
  const float ir = __fdividef(1.f, r);
  float vx, vy, vz;
  if constexpr (Sch<S>::GF) {
    vx = jin[o] * ir + muf[o];
    vy = jin[o + g.P] * ir + muf[o + g.P];
    vz = jin[o + 2 * g.P] * ir + muf[o + 2 * g.P];
  } else {
    float gx = 0.f, gy = 0.f, gz = 0.f, mx = 0.f, my = 0.f, mz = 0.f;
#pragma unroll
    for (int m = 1; m <= R; ++m) {
      const float c = float(Sch<S>::g(m));
      const int yp = o + (wrapi(y + m, ny) - y) * g.LX, ym = o + (wrapi(y - m, ny) - y) * g.LX;
      const int zp = o + (wrapi(z + m, nz) - z) * g.PL, zm = o + (wrapi(z - m, nz) - z) * g.PL;
      gx += c * (__ldg(rin + o + m) - __ldg(rin + o - m));
      mx += c * (__ldg(muf + o + m) - __ldg(muf + o - m));
      gy += c * (__ldg(rin + yp) - __ldg(rin + ym));
      my += c * (__ldg(muf + yp) - __ldg(muf + ym));
      gz += c * (__ldg(rin + zp) - __ldg(rin + zm));
      mz += c * (__ldg(muf + zp) - __ldg(muf + zm));
    }
    vx = (jin[o] + (gx * (1.f / 3.f) - r * mx)) * ir;
    vy = (jin[o + g.P] + (gy * (1.f / 3.f) - r * my)) * ir;
    vz = (jin[o + 2 * g.P] + (gz * (1.f / 3.f) - r * mz)) * ir;
  }
  const float nvv = -1.5f * (vx * vx + (vy * vy + vz * vz));
  rout[n] = rlast[o];
  const int dxp = (x + 1 < nx) ? 1 : 1 - nx, dxm = (x > 0) ? -1 : nx - 1;
  const int dyp = (y + 1 < ny) ? nx : nx - NXY, dym = (y > 0) ? -nx : NXY - nx;
  const int dzp = (z + 1 < nz) ? NXY : NXY - N, dzm = (z > 0) ? -NXY : N - NXY;
#pragma unroll
  for (int i = 0; i < 19; ++i) {
    const float wi = float(L::w(i)), ev = edot<L>(i, vx, vy, vz);
    const float v = i == 0 ? fmaf(-12.f, float(L::w(1)) * d, d) + wi * r * nvv  // (Post2::rest)
                           : wi * d + wi * r * (4.5f * (ev * ev) + nvv) + (3.f * wi) * r * ev;
    const int s = (L::ex(i) > 0 ? dxp : (L::ex(i) < 0 ? dxm : 0)) + (L::ey(i) > 0 ? dyp : (L::ey(i) < 0 ? dym : 0)) +
                  (L::ez(i) > 0 ? dzp : (L::ez(i) < 0 ? dzm : 0));
    __stcs(fout + i * N + n + s, v);
  }
}

}  // namespace lbmd
