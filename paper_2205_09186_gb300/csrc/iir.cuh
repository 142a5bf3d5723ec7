// F / rho = D rho / (3 rho) - D mu along one axis for the compact schemes, D f the
// solution of Eq. 21 on a periodic line, for steps (the observation and field
// passes keep the separate derivative fields of compact_dev.cuh).
//
// The constant tridiagonal operator of Eq. 21 factors into two first-order
// recursions: alpha E^-1 + 1 + alpha E = (1 + r E^-1)(1 + r E) / (1 + r^2) with r =
// (1 - sqrt(1 - 4 alpha^2)) / (2 alpha) < 1, so that
//
//   y_i = d_i - r y_{i-1},   D f_i = y_i - r D f_{i+1}   (d_i scaled by 1 + r^2),
//
// two multiply-adds per node where cyclic reduction takes three operations on
// each of seven or more levels.  A line is cut into segments of a few nodes, one per
// thread, all in registers: each runs its recursion from zero, and since what
// enters a segment decays as r^k (r = 0.617 for OCFDS4: 2^-27 after 39 nodes),
// the ends of the few segments before it give it exactly, periodic wrap
// included; (-r)^k times it is added.  mu and rho are solved side by side and
// combined at the end: three fields written instead of six.
//
// k_iir_col  lines along y or z: lane = column, warp = segment, ends exchanged in
//            shared memory
// k_iir_row  lines along x: a warp per line, lane = segment, ends by shuffle;
//            staged in shared memory for coalesced access
//
// D3Q19 192^3 OCFDS4 (FP32): 36 us along x, 46 along y and z each; the whole step
// 228 us, 366 with six derivative fields by cyclic reduction and the populations
// moved.  FP64 80^3: 2037 -> 330 us a step.
#pragma once
#include <cuda_runtime.h>

#include "launch.cuh"
#include "lbm_device.cuh"

namespace lbmd {

constexpr int IIR_M = 32;  // nodes per segment at most

template <class T>
struct IirK {
  T nr, a1, a2, a3;  // -r, and the explicit side's a/2, b/4, c/6 times 1 + r^2
  T p[IIR_M + 1];    // (-r)^k
  int K;             // nodes after which r^k is below the type's rounding
};

// element (x, y, z): z pl + y ld + off + x; out: component a at a fs
struct IirGeo {
  int nx, ny, nz, ld, pl, off, fs;
};

// a thread's segment: the right side and the recursions on up to M nodes
template <class T, int M>
struct IirSeg {
  T v[M + 6];
  __device__ __forceinline__ T forward(const IirK<T>& c, int len) {  // v: nodes -3 .. len + 2 -> y_0 .. ; the last y
    T y = 0;
#pragma unroll
    for (int k = 0; k < M; ++k)
      if (k < len) {
        const T d = c.a1 * (v[k + 4] - v[k + 2]) + c.a2 * (v[k + 5] - v[k + 1]) + c.a3 * (v[k + 6] - v[k]);
        y = d + c.nr * y;
        v[k] = y;
      }
    return y;
  }
  __device__ __forceinline__ T backward(const IirK<T>& c, int len, T in) {  // in: what entered; the first z
    T z = 0;
#pragma unroll
    for (int k = M - 1; k >= 0; --k)
      if (k < len) {
        z = v[k] + in * c.p[k + 1] + c.nr * z;
        v[k] = z;
      }
    return z;
  }
};

__device__ __forceinline__ float iir_quot(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double iir_quot(double a, double b) { return a * rcp64(b); }

// LS: log2 of the segments; J: how many of them reach (K nodes of at least L >> LS each)
template <class T, int M, int LS>
__global__ void __launch_bounds__(32 << LS) k_iir_col(const IirGeo g, const int axis, const T* rho,
                                                      const T* mu, T* __restrict__ out, const T rref,
                                                      const int J, const IirK<T> c) {
  constexpr int S = 1 << LS;
  __shared__ T s_f[2][S][32], s_b[2][S][32];
  pdl_wait();
  const int lane = threadIdx.x, s = threadIdx.y;
  const int x = blockIdx.x * 32 + lane, L = axis == 1 ? g.ny : g.nz, st = axis == 1 ? g.ld : g.pl;
  const int base = g.off + min(x, g.nx - 1) + int(blockIdx.y) * (axis == 1 ? g.pl : g.ld);
  const int i0 = s * L >> LS, len = ((s + 1) * L >> LS) - i0, lo = L >> LS;  // segments have lo or lo + 1 nodes
  const T plo = c.p[lo], phi = c.p[min(lo + 1, IIR_M)];
  IirSeg<T, M> m, q;
  if (i0 >= 3 && i0 + len + 3 <= L) {  // (uniform in the warp) no wrap
    const T *a = mu + (base + (i0 - 3) * st), *b = rho + (base + (i0 - 3) * st);
#pragma unroll
    for (int k = 0; k < M + 6; ++k)
      if (k < len + 6) {
        m.v[k] = *a;
        q.v[k] = *b;
        a += st;
        b += st;
      }
  } else {
#pragma unroll
    for (int k = 0; k < M + 6; ++k)
      if (k < len + 6) {
        int i = i0 - 3 + k;
        i = i < 0 ? i + L : (i >= L ? i - L : i);
        m.v[k] = mu[base + i * st];
        q.v[k] = rho[base + i * st];
      }
  }
  s_f[0][s][lane] = m.forward(c, len);
  s_f[1][s][lane] = q.forward(c, len);
  __syncthreads();
  // what enters both fields: the ends of J segments, the nearest last
  T em, eq;
  auto enter = [&](const T(*e)[S][32], int dir) {
    em = eq = 0;
    for (int j = J; j >= 1; --j) {
      const int t = (s + dir * j) & (S - 1);
      const T f = ((t + 1) * L >> LS) - (t * L >> LS) > lo ? phi : plo;
      em = e[0][t][lane] + f * em;
      eq = e[1][t][lane] + f * eq;
    }
  };
  enter(s_f, -1);
  s_b[0][s][lane] = m.backward(c, len, em);
  s_b[1][s][lane] = q.backward(c, len, eq);
  __syncthreads();
  enter(s_b, 1);
  if (x >= g.nx) return;
  const int o0 = base + i0 * st;
#pragma unroll
  for (int k = M - 1; k >= 0; --k)
    if (k < len) {
      em *= c.nr;
      eq *= c.nr;
      const int o = o0 + k * st;
      out[axis * g.fs + o] = iir_quot(q.v[k] + eq, T(3) * (rref + rho[o])) - (m.v[k] + em);
    }
}

template <class T, int M>
__global__ void __launch_bounds__(256) k_iir_row(const IirGeo g, const T* rho, const T* mu,
                                                 T* __restrict__ out, const T rref, const int J, const T close,
                                                 const IirK<T> c) {
  extern __shared__ __align__(16) unsigned char sm_iir[];
  pdl_wait();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, L = g.nx, LP = L + (L >> 5) + 1;
  const int line = blockIdx.x * 8 + w;
  if (line >= g.ny * g.nz) return;  // (no CTA barrier below)
  const int z = line / g.ny, base = g.off + z * g.pl + (line - z * g.ny) * g.ld;
  T* sr = reinterpret_cast<T*>(sm_iir) + w * 2 * LP;  // one element of padding per 32: no bank is hit by every lane
  T* su = sr + LP;
  for (int i = lane; i < L; i += 32) {
    sr[i + (i >> 5)] = rho[base + i];
    su[i + (i >> 5)] = mu[base + i];
  }
  __syncwarp();
  const int i0 = lane * L / 32, len = (lane + 1) * L / 32 - i0;
  IirSeg<T, M> m, q;
#pragma unroll
  for (int k = 0; k < M + 6; ++k)
    if (k < len + 6) {
      int i = i0 - 3 + k;
      i = i < 0 ? i + L : (i >= L ? i - L : i);
      m.v[k] = su[i + (i >> 5)];
      q.v[k] = sr[i + (i >> 5)];
    }
  const T pl = c.p[len];
  T em, eq;
  // what enters: segments' ends with their decay, by doubling until J segments are
  // summed; all 32 of them are one period, 1 / (1 - (-r)^L) closes it
  auto enter = [&](T a, T b, int dir) {
    T f = pl;
    int n = 1;
    for (; n < J && n < 32; n *= 2) {
      const int from = (lane + dir * n) & 31;
      const T a1 = __shfl_sync(0xffffffffu, a, from), b1 = __shfl_sync(0xffffffffu, b, from);
      const T f1 = __shfl_sync(0xffffffffu, f, from);
      a += f * a1;
      b += f * b1;
      f *= f1;
    }
    em = __shfl_sync(0xffffffffu, a, (lane + dir) & 31);
    eq = __shfl_sync(0xffffffffu, b, (lane + dir) & 31);
    if (n == 32) {
      em *= close;
      eq *= close;
    }
  };
  const T fm = m.forward(c, len), fq = q.forward(c, len);
  enter(fm, fq, -1);
  const T bm = m.backward(c, len, em), bq = q.backward(c, len, eq);
  enter(bm, bq, 1);
  __syncwarp();
#pragma unroll
  for (int k = M - 1; k >= 0; --k)
    if (k < len) {
      em *= c.nr;
      eq *= c.nr;
      const int i = i0 + k;
      sr[i + (i >> 5)] = iir_quot(q.v[k] + eq, T(3) * (rref + sr[i + (i >> 5)])) - (m.v[k] + em);
    }
  __syncwarp();
  for (int i = lane; i < L; i += 32) out[base + i] = sr[i + (i >> 5)];
}

// ------------------------------------------------------------------ CTAs of a batch
// The same for D2Q9 lattices in a persistent launch, by a CTA of 256 threads: eight
// lines along x (a warp each), or Q columns (256 / Q segments each). rho is padded
// (row stride ldr, first column at off), mu and out are not. Written earlier in the
// launch, so read by ordinary loads. All threads take part (barriers inside); c and
// smem (IIR_CTA_FLOATS) in shared memory.
//
// The segments lie in shared memory, not in registers as above: the registers are
// the tile kernel's 80, its shared memory leaves the L1 a few KB, and spilled
// segments went to L2 and back (48 cases, 8 of them compact: 111 us a step).
constexpr int IIR_CTA_ROWS = 8, IIR_CTA_LP = 512 + 6 + 16 + 1;  // rows, a padded line
__host__ __device__ constexpr int iir_cta_cols_n(int ny) { return ny <= 256 ? 16 : 8; }
constexpr int IIR_CTA_FLOATS = 4 * (256 + 6) * 16 + 1024 + 64;
static_assert(IIR_CTA_FLOATS >= 4 * IIR_CTA_ROWS * IIR_CTA_LP && IIR_CTA_FLOATS >= 4 * (512 + 6) * 8 + 1024, "fits");

// a segment of both fields: r and u (nodes -3 .. len + 2 about at(0)), y scratch;
// enter(ends, dir): what enters it from the segments before (-1) and after (1)
template <class At, class Enter, class Emit>
__device__ __forceinline__ void iir_cta_seg(const IirK<float>& c, const float* r, const float* u, float* yr, float* yu,
                                            At at, int len, Enter enter, Emit emit) {
  const float a1 = c.a1, a2 = c.a2, a3 = c.a3, nr = c.nr;
  float2 y = make_float2(0.f, 0.f);
  {
    float r0 = r[at(-3)], r1 = r[at(-2)], r2 = r[at(-1)], r3 = r[at(0)], r4 = r[at(1)], r5 = r[at(2)];
    float u0 = u[at(-3)], u1 = u[at(-2)], u2 = u[at(-1)], u3 = u[at(0)], u4 = u[at(1)], u5 = u[at(2)];
#pragma unroll 2
    for (int k = 0; k < len; ++k) {
      const float r6 = r[at(k + 3)], u6 = u[at(k + 3)];
      y.x = a1 * (r4 - r2) + a2 * (r5 - r1) + a3 * (r6 - r0) + nr * y.x;
      y.y = a1 * (u4 - u2) + a2 * (u5 - u1) + a3 * (u6 - u0) + nr * y.y;
      yr[at(k)] = y.x;
      yu[at(k)] = y.y;
      r0 = r1, r1 = r2, r2 = r3, r3 = r4, r4 = r5, r5 = r6;
      u0 = u1, u1 = u2, u2 = u3, u3 = u4, u4 = u5, u5 = u6;
    }
  }
  float2 e = enter(y, -1);
  y = make_float2(0.f, 0.f);
#pragma unroll 2
  for (int k = len - 1; k >= 0; --k) {
    const float p = c.p[k + 1];
    y.x = yr[at(k)] + e.x * p + nr * y.x;
    y.y = yu[at(k)] + e.y * p + nr * y.y;
    yr[at(k)] = y.x;
    yu[at(k)] = y.y;
  }
  e = enter(y, 1);
#pragma unroll 2
  for (int k = len - 1; k >= 0; --k) {
    e.x *= nr;
    e.y *= nr;
    emit(k, yr[at(k)] + e.x, yu[at(k)] + e.y);
  }
}

__device__ __forceinline__ void iir_cta_rows(const IirK<float>& c, int nx, int ny, int ldr, int off, const float* rho,
                                             const float* mu, float* out, float rref, int y0, float* smem) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, y = y0 + w;
  float *sr = smem + w * 4 * IIR_CTA_LP, *su = sr + IIR_CTA_LP, *yr = su + IIR_CTA_LP, *yu = yr + IIR_CTA_LP;
  if (y < ny) {
    for (int k = lane; k < nx + 6; k += 32) {
      int i = k - 3;
      i = i < 0 ? i + nx : (i >= nx ? i - nx : i);
      sr[k + (k >> 5)] = rho[y * ldr + off + i];
      su[k + (k >> 5)] = mu[y * nx + i];
    }
    __syncwarp();
    const int i0 = lane * nx / 32, len = (lane + 1) * nx / 32 - i0, J = (c.K * 32 + nx - 1) / nx + 1;
    const float pl = c.p[len];
    auto at = [&](int k) { return i0 + 3 + k + ((i0 + 3 + k) >> 5); };
    // -r^nx closes the period (doubling sums all 32 segments when J asks for it)
    auto enter = [&](float2 a, int dir) {
      float f = pl;
      int n = 1;
      for (; n < J && n < 32; n *= 2) {
        const int from = (lane + dir * n) & 31;
        const float ax = __shfl_sync(0xffffffffu, a.x, from), ay = __shfl_sync(0xffffffffu, a.y, from);
        const float f1 = __shfl_sync(0xffffffffu, f, from);
        a.x += f * ax;
        a.y += f * ay;
        f *= f1;
      }
      a.x = __shfl_sync(0xffffffffu, a.x, (lane + dir) & 31);
      a.y = __shfl_sync(0xffffffffu, a.y, (lane + dir) & 31);
      return n == 32 ? make_float2(a.x / (1.f - f), a.y / (1.f - f)) : a;
    };
    iir_cta_seg(c, sr, su, yr, yu, at, len, enter,
                [&](int k, float dr, float du) { yu[at(k)] = __fdividef(dr, 3.f * (rref + sr[at(k)])) - du; });
    __syncwarp();
    for (int i = lane; i < nx; i += 32) out[y * nx + i] = yu[i + 3 + ((i + 3) >> 5)];
  }
}

template <int Q>
__device__ __forceinline__ void iir_cta_cols(const IirK<float>& c, int nx, int ny, int ldr, int off, const float* rho,
                                             const float* mu, float* out, float rref, int x0, float* smem) {
  constexpr int S = 256 / Q;
  const int q = threadIdx.x % Q, s = threadIdx.x / Q, x = min(x0 + q, nx - 1), F = (ny + 6) * Q;
  float *sr = smem, *su = sr + F, *yr = su + F, *yu = yr + F;
  float2* se = reinterpret_cast<float2*>(smem + IIR_CTA_FLOATS - 1024);  // [2][S][Q] of ends, forward and back
  for (int r = s; r < ny + 6; r += S) {
    int i = r - 3;
    i = i < 0 ? i + ny : (i >= ny ? i - ny : i);
    sr[r * Q + q] = rho[i * ldr + off + x];
    su[r * Q + q] = mu[i * nx + x];
  }
  __syncthreads();
  const int i0 = s * ny / S, len = (s + 1) * ny / S - i0, lo = ny / S, J = (c.K * S + ny - 1) / ny + 1;
  const float plo = c.p[lo], phi = c.p[lo + 1];
  auto at = [&](int k) { return (i0 + 3 + k) * Q + q; };
  auto enter = [&](float2 v, int dir) {
    float2* f = se + (dir > 0 ? S * Q : 0);
    f[threadIdx.x] = v;
    __syncthreads();
    float2 a = make_float2(0.f, 0.f);
    for (int j = J; j >= 1; --j) {
      const int t = (s + dir * j) & (S - 1);
      const float p = (t + 1) * ny / S - t * ny / S > lo ? phi : plo;
      const float2 b = f[t * Q + q];
      a.x = b.x + p * a.x;
      a.y = b.y + p * a.y;
    }
    return a;
  };
  iir_cta_seg(c, sr, su, yr, yu, at, len, enter, [&](int k, float dr, float du) {
    if (x0 + q < nx) out[(i0 + k) * nx + x] = __fdividef(dr, 3.f * (rref + sr[at(k)])) - du;
  });
}

// coefficients of a scheme (host)
IirK<float> iir_coef(int scheme);

}  // namespace lbmd
