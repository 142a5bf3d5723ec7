// D2Q9 FP32-deviation steps at tau = 1 on three moments (density deviation and
// momentum) instead of nine populations; see mom3d.cuh for why they suffice.
// Here a step is one pass, mu included:
//
//  mom2_gather  rho, j of the call's initial populations
//  mom2_tile    rho, j of the next step; in its FINAL form the populations and
//               the density the call leaves behind
//
// A tile is up to 60 columns x 30 rows, done by a CTA of eight warps, two
// adjacent columns per lane (packed arithmetic): rho with a halo of 2 R + 1
// staged in shared memory, mu on the tile and R + 1 beyond, collision of the tile
// and a ring (a warp per row of 64 columns), then the sums of what arrives.
// Populations that move along a row go by shuffle, the others through shared
// memory, summed where they land together.  Three CTA barriers; three CTAs per SM
// cover each other's (34 rows and two CTAs: 57 us a step at 2048^2, 49 this way,
// 46 with each step's launch overlapping the step before).
// A march along y without shared memory or barriers (a warp per 128-column
// strip, queues in registers) needs fewer instructions, but its rows are one
// long chain per warp: 14.3 us a step at 512^2, 6.8 with tiles.
//
// Bytes per node: 12 in, 12 out (88 with populations and a mu field).  In two
// launches on the populations a step took 16.4 us at 512^2 and 472 at 4096^2; 6.8
// and 172 here.
//
// Fields (float): element (x, y) at y LX + 8 + x, LX = 4 ceil(nx / 4) + 16; rho
// and j rows carry eight periodic copies at either end, so nothing wraps in x.
#pragma once
#include "lbm_device.cuh"
#include "pack2.cuh"
#include "step2d_split.cuh"

namespace lbmd {

constexpr int T2W = 60, T2H = 30, T2NT = 256;  // tile columns and rows at most, threads

struct Mom2Geo {
  int LX, P;      // row stride, field stride
  int TW, nt;     // columns per tile (a multiple of 4), tiles across
  int TH, nr;     // rows per tile, tiles down
};

template <int S>
struct Mom2Shape {
  static constexpr int R = Sch<S>::R, H = 2 * R + 1;
  static constexpr int RW = 80;                        // staged columns -8 .. 67 (and padding)
  static constexpr int RR = T2H + 2 * H;               // staged rows
  static constexpr int MW = 72, MR = T2H + 2 + 2 * R;  // mu columns -4 .. 63 (and padding), rows
  static constexpr int XR = T2H + 2;                   // exchange rows of 64 columns
};
constexpr int T2_SMEM = 4 * (Mom2Shape<S_EFDS6>::RW * Mom2Shape<S_EFDS6>::RR + Mom2Shape<S_EFDS6>::MW * Mom2Shape<S_EFDS6>::MR +
                             6 * 64 * Mom2Shape<S_EFDS6>::XR);

constexpr int T2_CTAS = 2 * (T2_SMEM + 1024) <= 152 * 1024 && 3 * (T2_SMEM + 1024) <= 228 * 1024 ? 3 : 2;  // per SM

// packed constants (constant memory: see MomConst); h: first-derivative weights
// / 3, g: the weights, l: Laplacian weights (l[0]: both axes')
struct Mom2Const {
  float2 h[3], g[3], l[4];
  float2 m1, c45, m15, m5, w0, w1, w2, t1, t2, n1, n2;  // -1, 4.5, -1.5, -5, 4/9, 1/9, 1/36, +-3/9, +-3/36
};
constexpr float2 mk2(double v) { return float2{float(v), float(v)}; }
template <int S>
constexpr Mom2Const mom2_const() {
  Mom2Const k{};
  if constexpr (!Sch<S>::ISO) {
    for (int m = 1; m <= Sch<S>::R; ++m) {
      k.h[m - 1] = mk2(Sch<S>::g(m) / 3.0);
      k.g[m - 1] = mk2(Sch<S>::g(m));
      k.l[m] = mk2(Sch<S>::l(m));
    }
    k.l[0] = mk2(2.0 * Sch<S>::l(0));
  }
  k.m1 = mk2(-1.0); k.c45 = mk2(4.5); k.m15 = mk2(-1.5); k.m5 = mk2(-5.0);
  k.w0 = mk2(4.0 / 9); k.w1 = mk2(1.0 / 9); k.w2 = mk2(1.0 / 36);
  k.t1 = mk2(3.0 / 9); k.t2 = mk2(3.0 / 36); k.n1 = mk2(-3.0 / 9); k.n2 = mk2(-3.0 / 36);
  return k;
}
template <int S>
__constant__ constexpr Mom2Const c_mom2 = mom2_const<S>();

// k^2 psi'(rho) - kappa lap of two nodes (eos_mu_f's formula, packed for
// Carnahan-Starling)
__device__ __forceinline__ float2 mu_pair(float2 rho, float2 lap, const EosF& e, float k2, float kap) {
  if (e.eos != 0) return make_float2(k2 * eos_mu_f(rho.x, e) - kap * lap.x, k2 * eos_mu_f(rho.y, e) - kap * lap.y);
  const float2 eta = mul2(f2(e.b4), rho), om = fma2(f2(-e.b4), rho, f2(1.f));
  const float2 num = mul2(eta, fma2(eta, fma2(f2(3.f), eta, f2(-9.f)), f2(8.f))), den = mul2(mul2(om, om), om);
  const float2 hs = make_float2(__fdividef(num.x, den.x), __fdividef(num.y, den.y));
  const float2 lg2 = make_float2(__logf(rho.x), __logf(rho.y));
  const float2 m = fma2(f2(-e.two_a), rho, mul2(f2(e.RT), add2(lg2, hs)));
  return fma2(f2(-kap), lap, mul2(f2(k2), m));
}

// One CTA of T2NT threads: the tile at (x0, y0), VW x VH nodes, of the next state
// from rin, jin (jx, then jy at stride P).  FINAL: into the populations
// fout[9][N] and the density rout of the unpadded lattice; else into the padded
// rout, jout.  The inputs are written by other SMs earlier in the same launch
// (behind a device-wide barrier) where a persistent kernel calls this, so they
// are read by ordinary loads or by copies that bypass L1.  The caller's next
// barrier must lie between this call and the next use of smem.
template <int S, bool FINAL>
__device__ __forceinline__ void mom2_tile(const KParams& p, int LX, int P, const float* rin, const float* jin, float* rout,
                                          float* jout, float* fout, unsigned long long* bad, long long t, int x0, int y0,
                                          int VW, int VH, float* smem, const float* acc = nullptr) {
  using Sh = Mom2Shape<S>;
  constexpr bool GF = Sch<S>::GF;  // compact: F / rho from acc (two unpadded fields)
  constexpr int R = Sh::R, H = Sh::H, RW = Sh::RW, MW = Sh::MW, XK = Sh::XR * 32;
  constexpr bool ISO = Sch<S>::ISO;
  const Mom2Const& kc = c_mom2<S>;
  float* s_r = smem;                                        // row k: y0 - H + k; column j: x0 - 8 + j
  float* s_m = s_r + Sh::RR * RW;                           // row k: y0 - 1 - R + k; column j: x0 - 4 + j
  float2* s_x = reinterpret_cast<float2*>(GF ? smem : s_m + Sh::MR * MW);  // [6][XR][32]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nx = p.nx, ny = p.ny;
  const float rref = float(p.rho_ref);
  if constexpr (!GF) {
    // ---- rho (16-byte chunks; those past the padded row are zeroed)
    for (int e = tid; e < (VH + 2 * H) * 19; e += T2NT) {
      const int k = e / 19, j = 4 * (e - k * 19);
      if (x0 + j + 4 <= LX) cpa16(s_r + k * RW + j, rin + (unsigned(wrapn(y0 - H + k, ny)) * LX + x0 + j));
      else *reinterpret_cast<float4*>(s_r + k * RW + j) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    cpa_commit();
  }
  auto two = [](const float* q) { return *reinterpret_cast<const float2*>(q); };
  // momentum of the warp's next row of the ring, loaded a row ahead
  float2 jx = f2(0.f), jy = f2(0.f), dn = f2(0.f), ax = f2(0.f), ay = f2(0.f);
  const int xa = GF ? wrapn(x0 - 2 + 2 * lane, nx) : 0, xb = GF ? wrapn(x0 - 1 + 2 * lane, nx) : 0;
  auto ldj = [&](int k) {
    if (k < VH + 2 && x0 + 8 + 2 * lane <= LX) {  // inside the padded row
      const int y = wrapn(y0 - 1 + k, ny);
      const unsigned o = unsigned(y) * LX + 6 + x0 + 2 * lane;
      jx = two(jin + o);
      jy = two(jin + P + o);
      if constexpr (GF) {
        dn = two(rin + o);
        const float* a = acc + y * nx;
        ax = make_float2(a[xa], a[xb]);
        ay = make_float2(a[int(p.n) + xa], a[int(p.n) + xb]);
      }
    }
  };
  ldj(w);
  if constexpr (!GF) {
    cpa_wait_all();
    __syncthreads();
  }
  auto sub = [&](float2 a, float2 b) { return fma2(kc.m1, b, a); };
  // ---- mu of the pairs -4 .. 63
  if constexpr (!GF) {
    const float k2 = float(p.k2), kap = float(p.kappa);
    const EosF ef = eos_f(p);
    for (int e = tid; e < (VH + 2 + 2 * R) * 34; e += T2NT) {
      const int k = e / 34, j = 2 * (e - k * 34);
      const float* q = s_r + (k + R) * RW + j + 4;
      const float2 c = two(q);
      float2 lap;
      if constexpr (ISO) {
        float a = 0.f, b = 0.f;
#pragma unroll
        for (int dy = -R; dy <= R; ++dy) {
          float v[2 * R + 2];  // offsets -R .. R + 1
          if constexpr (R == 1) {
            const float2 l = two(q + dy * RW - 2), m = two(q + dy * RW), h = two(q + dy * RW + 2);
            v[0] = l.y; v[1] = m.x; v[2] = m.y; v[3] = h.x;
          } else {
            const float2 l = two(q + dy * RW - 2), m = two(q + dy * RW), h = two(q + dy * RW + 2);
            v[0] = l.x; v[1] = l.y; v[2] = m.x; v[3] = m.y; v[4] = h.x; v[5] = h.y;
          }
#pragma unroll
          for (int dx = -R; dx <= R; ++dx) {
            const double wt = Sch<S>::w2d(dx, dy);
            if (wt == 0.0) continue;
            a += float(2.0 * wt) * (v[dx + R] - c.x);
            b += float(2.0 * wt) * (v[dx + R + 1] - c.y);
          }
        }
        lap = make_float2(a, b);
      } else {
        const float2 l = two(q - 2), h = two(q + 2);
        lap = fma2(kc.l[1], add2(make_float2(l.y + c.y, c.x + h.x), add2(two(q + RW), two(q - RW))), mul2(kc.l[0], c));
        if constexpr (R >= 2) lap = fma2(kc.l[2], add2(add2(l, h), add2(two(q + 2 * RW), two(q - 2 * RW))), lap);
        if constexpr (R >= 3) {
          const float2 a = two(q - 4), b = two(q + 4);
          lap = fma2(kc.l[3], add2(make_float2(a.y + h.y, l.x + b.x), add2(two(q + 3 * RW), two(q - 3 * RW))), lap);
        }
      }
      *reinterpret_cast<float2*>(s_m + k * MW + j) = mu_pair(add2(f2(rref), c), lap, ef, k2, kap);
    }
    __syncthreads();
  }
  // ---- collision: row k of the ring and the tile, columns -2 .. 61
  for (int k = w; k < VH + 2; k += T2NT / 32) {
    float2 d, gmx, gmy, grx, gry;  // grad mu, grad rho / 3
    const float* q = s_r + (k + H - 1) * RW + 6 + 2 * lane;
    const float* m = s_m + (k + R) * MW + 2 + 2 * lane;
    d = GF ? dn : two(q);
    if constexpr (GF) {
      gmx = gmy = grx = gry = f2(0.f);
    } else if constexpr (ISO) {
      auto grad = [&](const float* b, int W, float2& gx, float2& gy) {
        float x0_ = 0.f, x1 = 0.f, y0_ = 0.f, y1 = 0.f;
#pragma unroll
        for (int dy = -R; dy <= R; ++dy) {
          float v[2 * R + 2];
          const float2 l = two(b + dy * W - 2), c = two(b + dy * W), h = two(b + dy * W + 2);
          if constexpr (R == 1) {
            v[0] = l.y; v[1] = c.x; v[2] = c.y; v[3] = h.x;
          } else {
            v[0] = l.x; v[1] = l.y; v[2] = c.x; v[3] = c.y; v[4] = h.x; v[5] = h.y;
          }
#pragma unroll
          for (int dx = -R; dx <= R; ++dx) {
            const double wt = Sch<S>::w2d(dx, dy);
            if (wt == 0.0) continue;
            if (dx != 0) {
              x0_ += float(wt * dx) * v[dx + R];
              x1 += float(wt * dx) * v[dx + R + 1];
            }
            if (dy != 0) {
              y0_ += float(wt * dy) * v[dx + R];
              y1 += float(wt * dy) * v[dx + R + 1];
            }
          }
        }
        gx = make_float2(x0_, x1);
        gy = make_float2(y0_, y1);
      };
      grad(m, MW, gmx, gmy);
      grad(q, RW, grx, gry);
      grx = mul2(f2(1.f / 3.f), grx);
      gry = mul2(f2(1.f / 3.f), gry);
    } else {
      auto grad = [&](const float* b, int W, const float2* s, float2& gx, float2& gy) {
        const float2 l = two(b - 2), c = two(b), h = two(b + 2);
        gx = mul2(s[0], make_float2(c.y - l.y, h.x - c.x));
        gy = mul2(s[0], sub(two(b + W), two(b - W)));
        if constexpr (R >= 2) {
          gx = fma2(s[1], sub(h, l), gx);
          gy = fma2(s[1], sub(two(b + 2 * W), two(b - 2 * W)), gy);
        }
        if constexpr (R >= 3) {
          const float2 a = two(b - 4), z = two(b + 4);
          gx = fma2(s[2], make_float2(h.y - a.y, z.x - l.x), gx);
          gy = fma2(s[2], sub(two(b + 3 * W), two(b - 3 * W)), gy);
        }
      };
      grad(m, MW, kc.g, gmx, gmy);
      grad(q, RW, kc.h, grx, gry);
    }
    const float2 r = add2(f2(rref), d), nr = mul2(kc.m1, r);
    const float2 ir = make_float2(__fdividef(1.f, r.x), __fdividef(1.f, r.y));
    float2 vx, vy;
    if constexpr (GF) {
      vx = fma2(jx, ir, ax);
      vy = fma2(jy, ir, ay);
    } else {
      vx = mul2(add2(jx, fma2(nr, gmx, grx)), ir);
      vy = mul2(add2(jy, fma2(nr, gmy, gry)), ir);
    }
    ldj(k + T2NT / 32);
    // post-collision populations (Eq. 2's order); opposite ones share all but
    // the sign of the linear term; the rest population carries drho less the
    // others' 4 b1 + 4 b2 = 5 b1 (b2 = b1 / 4 exactly): see Post2::rest
    const float2 nvv = mul2(kc.m15, fma2(vx, vx, mul2(vy, vy)));
    const float2 b1 = mul2(kc.w1, d), b2 = mul2(kc.w2, d), r1 = mul2(kc.w1, r), r2 = mul2(kc.w2, r);
    const float2 t1 = mul2(kc.t1, r), t2 = mul2(kc.t2, r), n1 = mul2(kc.n1, r), n2 = mul2(kc.n2, r);
    auto pair = [&](float2 E, float2 rr, float2 b, float2 tt, float2 nn, float2& u, float2& v) {
      const float2 e = fma2(rr, fma2(kc.c45, mul2(E, E), nvv), b);
      u = fma2(tt, E, e);
      v = fma2(nn, E, e);
    };
    float2 f[9];
    f[0] = fma2(mul2(kc.w0, r), nvv, fma2(kc.m5, b1, d));
    pair(vx, r1, b1, t1, n1, f[1], f[3]);
    pair(vy, r1, b1, t1, n1, f[2], f[4]);
    pair(add2(vx, vy), r2, b2, t2, n2, f[5], f[7]);
    pair(sub(vy, vx), r2, b2, t2, n2, f[6], f[8]);
    if constexpr (FINAL) {
      const int c = 2 * lane - 2;
      if (k >= 1 && k <= VH && c >= 0 && c < VW) {
        const int N = int(p.n), y = y0 - 1 + k;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          const int ex = Lattice<0>::ex(i), ey = Lattice<0>::ey(i);
          float* fo = fout + i * N + wrapi(y + ey, ny) * nx;
          fo[wrapi(x0 + c + ex, nx)] = f[i].x;
          if (c + 1 < VW) fo[wrapi(x0 + c + 1 + ex, nx)] = f[i].y;
        }
      }
    }
    // sum and difference of a right-moving and a left-moving population where
    // they land in the row (scalar: the shifted halves lie in two pairs; what
    // enters at the row's ends lands outside the tile)
    auto meet = [&](float2 u, float2 v, float2& s, float2& x) {
      const float l = __shfl_up_sync(0xffffffffu, u.y, 1), h = __shfl_down_sync(0xffffffffu, v.x, 1);
      s = make_float2(l + v.y, u.x + h);
      x = make_float2(l - v.y, u.x - h);
    };
    float2* xr = s_x + k * 32 + lane;
    float2 s, x;
    meet(f[1], f[3], s, x);
    xr[0] = add2(f[0], s);
    xr[XK] = x;
    meet(f[5], f[6], s, x);
    xr[2 * XK] = add2(f[2], s);
    xr[3 * XK] = x;
    meet(f[8], f[7], s, x);
    xr[4 * XK] = add2(f[4], s);
    xr[5 * XK] = x;
  }
  __syncthreads();
  // ---- the next state of the tile's rows
  bool ok = true;
  for (int k = 1 + w; k <= VH; k += T2NT / 32) {
    const int c = 2 * lane - 2;
    if (c < 0 || c >= VW) continue;
    const float2* xr = s_x + k * 32 + lane;
    const float2 u = xr[2 * XK - 32], dn = xr[4 * XK + 32];
    const float2 r = add2(xr[0], add2(u, dn)), jx = add2(xr[XK], add2(xr[3 * XK - 32], xr[5 * XK + 32])), jy = sub(u, dn);
    const bool both = c + 1 < VW;
    ok = ok && rref + r.x > 0.f && (!both || rref + r.y > 0.f);
    const int x = x0 + c, y = y0 + k - 1;
    if constexpr (FINAL) {
      rout[y * nx + x] = r.x;
      if (both) rout[y * nx + x + 1] = r.y;
    } else {
      float *a = rout + (unsigned(y) * LX + 8 + x), *b = jout + (unsigned(y) * LX + 8 + x), *e = b + P;
      if (both) {
        *reinterpret_cast<float2*>(a) = r;
        *reinterpret_cast<float2*>(b) = jx;
        *reinterpret_cast<float2*>(e) = jy;
      } else {
        a[0] = r.x;
        b[0] = jx.x;
        e[0] = jy.x;
      }
      // the periodic copies beside the row
      if (x < 8) { a[nx] = r.x; b[nx] = jx.x; e[nx] = jy.x; }
      if (x >= nx - 8) { a[-nx] = r.x; b[-nx] = jx.x; e[-nx] = jy.x; }
      if (both && x + 1 < 8) { a[1 + nx] = r.y; b[1 + nx] = jx.y; e[1 + nx] = jy.y; }
      if (both && x + 1 >= nx - 8) { a[1 - nx] = r.y; b[1 - nx] = jx.y; e[1 - nx] = jy.y; }
    }
  }
  if (!ok) atomicMin(bad, (unsigned long long)(t + 1));
}

// mu of a compact scheme (central Laplacian of order LO) at 8 rows x 32 columns by a
// warp, from the padded rho into the unpadded mu; ordinary loads (mom2_tile)
template <int LO>
__device__ __forceinline__ void mom2_mu_rows(const KParams& p, int LX, const float* rin, float* mu, int x0, int y0) {
  constexpr int R = LO / 2, U = 8;
  constexpr double l0 = LO == 4 ? -2.5 : (LO == 6 ? -49.0 / 18.0 : -205.0 / 72.0);
  constexpr double l[5] = {l0, LO == 4 ? 4.0 / 3.0 : (LO == 6 ? 1.5 : 1.6), LO == 4 ? -1.0 / 12.0 : (LO == 6 ? -0.15 : -0.2),
                           LO == 6 ? 1.0 / 90.0 : (LO == 8 ? 8.0 / 315.0 : 0.0), LO == 8 ? -1.0 / 560.0 : 0.0};
  const int x = x0 + int(threadIdx.x & 31), nx = p.nx, ny = p.ny;
  if (x >= nx || y0 >= ny) return;
  const float k2 = float(p.k2), kap = float(p.kappa), rref = float(p.rho_ref);
  const EosF ef = eos_f(p);
  float c[U + 2 * R];
#pragma unroll
  for (int k = 0; k < U + 2 * R; ++k) c[k] = rin[wrapn(y0 - R + k, ny) * LX + 8 + x];
#pragma unroll
  for (int r = 0; r < U; ++r) {
    if (y0 + r >= ny) break;
    const float* q = rin + (y0 + r) * LX + 8 + x;
    float lap = float(2.0 * l[0]) * c[r + R];
#pragma unroll
    for (int m = 1; m <= R; ++m) lap += float(l[m]) * ((q[m] + q[-m]) + (c[r + R + m] + c[r + R - m]));
    mu[(y0 + r) * nx + x] = k2 * eos_mu_f(rref + c[r + R], ef) - kap * lap;
  }
}

// moments of the populations f at rows ya .. yb - 1, columns xs .. xs + ow - 1
// (one column per lane and turn), with the copies beside the row
__device__ __forceinline__ void mom2_gather(const KParams& p, int LX, int P, const float* f, const float* rho, float* rout,
                                            float* jout, unsigned long long* bad, long long t, int xs, int ow, int ya,
                                            int yb) {
  const int lane = threadIdx.x & 31, nx = p.nx, N = int(p.n);
  bool ok = true;
  for (int y = ya; y < yb; ++y)
    for (int x = xs + lane; x < xs + ow; x += 32) {
      const float* fn = f + y * nx + x;
      float v[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) v[i] = fn[i * N];
      const float r = rho[y * nx + x];
      const float a = v[5] - v[7], b = v[6] - v[8];
      const float jx = (v[1] - v[3]) + (a - b), jy = (v[2] - v[4]) + (a + b);
      float *o = rout + y * LX + 8 + x, *q = jout + y * LX + 8 + x;
      o[0] = r;
      q[0] = jx;
      q[P] = jy;
      if (x < 8) { o[nx] = r; q[nx] = jx; q[P + nx] = jy; }
      if (x >= nx - 8) { o[-nx] = r; q[-nx] = jx; q[P - nx] = jy; }
      ok = ok && float(p.rho_ref) + r > 0.f;
    }
  if (!ok) atomicMin(bad, (unsigned long long)t);
}

}  // namespace lbmd
