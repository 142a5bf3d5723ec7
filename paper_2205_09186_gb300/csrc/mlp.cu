// Warm-start network: a small fully connected GELU network (FP32) that maps
// droplet parameters to an initial radial density profile.  Forward, backward
// (mean-squared error) and Adam run as CUDA kernels; the training loop stays
// on the device.  There is no counterpart in the paper: the network only
// supplies initial conditions that the solver then relaxes.
//
// Parameter layout (as in the C ABI): per layer W (out x in, row-major) then b.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/lbm.h"
#include "launch.cuh"

namespace {

constexpr int SB = 32;     // samples per CTA
constexpr int MAXW = 128;  // widest layer supported
constexpr int MAXL = 8;    // layers supported

struct Net {
  int nl;
  int sizes[MAXL + 1];
  long long woff[MAXL], boff[MAXL];  // parameter offsets
};

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_d(float x) {
  return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// forward for a block of SB samples; pre-activations z[l][s][o] and
// activations kept for backward in global scratch (act: per layer B x width)
__global__ void k_mlp_forward(const Net net, const float* __restrict__ P, const float* __restrict__ x, int B,
                              float* __restrict__ y, float* __restrict__ zs, float* __restrict__ hs) {
  __shared__ float h[SB][MAXW + 1];
  __shared__ float hn[SB][MAXW + 1];
  const int s0 = blockIdx.x * SB;
  const int ns = min(SB, B - s0);
  const int in0 = net.sizes[0];
  for (int idx = threadIdx.x; idx < SB * in0; idx += blockDim.x) {
    const int s = idx / in0, i = idx - s * in0;
    h[s][i] = s < ns ? x[(long long)(s0 + s) * in0 + i] : 0.f;
  }
  __syncthreads();
  long long zoff = 0;
  for (int l = 0; l < net.nl; ++l) {
    const int in = net.sizes[l], out = net.sizes[l + 1];
    const float* W = P + net.woff[l];
    const float* b = P + net.boff[l];
    for (int o = threadIdx.x; o < out; o += blockDim.x) {
      float acc[SB];
#pragma unroll
      for (int s = 0; s < SB; ++s) acc[s] = b[o];
      for (int i = 0; i < in; ++i) {
        const float w = W[(long long)o * in + i];
#pragma unroll
        for (int s = 0; s < SB; ++s) acc[s] += w * h[s][i];
      }
#pragma unroll
      for (int s = 0; s < SB; ++s) {
        if (s < ns) zs[zoff + (long long)(s0 + s) * out + o] = acc[s];
        hn[s][o] = (l < net.nl - 1) ? gelu(acc[s]) : acc[s];
      }
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < SB * out; idx += blockDim.x) {
      const int s = idx / out, o = idx - s * out;
      h[s][o] = hn[s][o];
      if (s < ns && l < net.nl - 1) hs[zoff + (long long)(s0 + s) * out + o] = hn[s][o];
    }
    __syncthreads();
    zoff += (long long)B * out;
  }
  const int nout = net.sizes[net.nl];
  for (int idx = threadIdx.x; idx < ns * nout; idx += blockDim.x) {
    const int s = idx / nout, o = idx - s * nout;
    y[(long long)(s0 + s) * nout + o] = h[s][o];
  }
}

// backward for a block of samples: per-CTA partial gradients (deterministic
// final reduction in k_reduce); loss partial per CTA
__global__ void k_mlp_backward(const Net net, const float* __restrict__ P, const float* __restrict__ x,
                               const float* __restrict__ t, int B, const float* __restrict__ y,
                               const float* __restrict__ zs, const float* __restrict__ hs, float* __restrict__ gpart,
                               long long nparam, float* __restrict__ lpart) {
  __shared__ float d[SB][MAXW + 1];
  __shared__ float dn[SB][MAXW + 1];
  __shared__ float hin[SB][MAXW + 1];
  __shared__ float red[256];
  const int s0 = blockIdx.x * SB;
  const int ns = min(SB, B - s0);
  const int nl = net.nl, nout = net.sizes[nl];
  const float scale = 2.f / (float(B) * float(nout));
  float lsum = 0.f;
  for (int idx = threadIdx.x; idx < SB * nout; idx += blockDim.x) {
    const int s = idx / nout, o = idx - s * nout;
    float v = 0.f;
    if (s < ns) {
      const float e = y[(long long)(s0 + s) * nout + o] - t[(long long)(s0 + s) * nout + o];
      lsum += e * e;
      v = e * scale;
    }
    d[s][o] = v;
  }
  red[threadIdx.x] = lsum;
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) lpart[blockIdx.x] = red[0];
  // offsets of the stored activations per layer
  long long zoff[MAXL];
  long long acc = 0;
  for (int l = 0; l < nl; ++l) { zoff[l] = acc; acc += (long long)B * net.sizes[l + 1]; }
  float* g = gpart + (long long)blockIdx.x * nparam;
  for (int l = nl - 1; l >= 0; --l) {
    const int in = net.sizes[l], out = net.sizes[l + 1];
    // input activations of layer l
    for (int idx = threadIdx.x; idx < SB * in; idx += blockDim.x) {
      const int s = idx / in, i = idx - s * in;
      float v = 0.f;
      if (s < ns) v = (l == 0) ? x[(long long)(s0 + s) * in + i] : hs[zoff[l - 1] + (long long)(s0 + s) * in + i];
      hin[s][i] = v;
    }
    __syncthreads();
    // dW[o][i] = sum_s d[s][o] hin[s][i]; db[o] = sum_s d[s][o]
    for (int idx = threadIdx.x; idx < out * in; idx += blockDim.x) {
      const int o = idx / in, i = idx - o * in;
      float a = 0.f;
#pragma unroll 8
      for (int s = 0; s < SB; ++s) a += d[s][o] * hin[s][i];
      g[net.woff[l] + idx] = a;
    }
    for (int o = threadIdx.x; o < out; o += blockDim.x) {
      float a = 0.f;
      for (int s = 0; s < SB; ++s) a += d[s][o];
      g[net.boff[l] + o] = a;
    }
    if (l > 0) {
      const float* W = P + net.woff[l];
      for (int idx = threadIdx.x; idx < SB * in; idx += blockDim.x) {
        const int s = idx / in, i = idx - s * in;
        float a = 0.f;
        for (int o = 0; o < out; ++o) a += W[(long long)o * in + i] * d[s][o];
        const float z = s < ns ? zs[zoff[l - 1] + (long long)(s0 + s) * in + i] : 0.f;
        dn[s][i] = a * gelu_d(z);
      }
      __syncthreads();
      for (int idx = threadIdx.x; idx < SB * in; idx += blockDim.x) {
        const int s = idx / in, i = idx - s * in;
        d[s][i] = dn[s][i];
      }
    }
    __syncthreads();
  }
}

// gradient = sum over CTAs of the partials (fixed order); loss likewise
__global__ void k_reduce(const float* __restrict__ gpart, int nblk, long long nparam, float* __restrict__ grad,
                         const float* __restrict__ lpart, float* __restrict__ loss, float lscale) {
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p < nparam) {
    float a = 0.f;
    for (int b = 0; b < nblk; ++b) a += gpart[(long long)b * nparam + p];
    grad[p] = a;
  }
  if (p == 0) {
    float a = 0.f;
    for (int b = 0; b < nblk; ++b) a += lpart[b];
    *loss = a * lscale;
  }
}

// Adam (Kingma and Ba): bias-corrected first and second moments
__global__ void k_adam(long long n, float* __restrict__ P, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, float lr, float b1, float b2, float eps, float c1, float c2) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  P[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ------------------------------------------------------------------ training
// All iterations of a training call in one launch by one cluster of eight
// CTAs.  Each CTA owns an eighth of every layer's outputs: those rows of W and
// b with their Adam moments stay in its shared memory for the whole call.
// An iteration is a chain of 2 nl - 2 exchanges between the layers, a few
// hundred kFLOP each at a few dozen samples, so its time is their latency; a
// cluster barrier and a round trip through L2 take about a microsecond, where a
// launch per pass (forward and backward by one CTA per 32 samples, reduction,
// Adam) took 386 us an iteration for 31 samples of the 4-128-128-128-64
// network, 29 now (77 for 128 samples).
//  forward   z = W h + b for the CTA's outputs; lane = sample, warp = output
//  backward  the CTA's share of W^T d, published; after the barrier the shares
//            are added in the CTAs' order, dW and db are summed over the
//            samples and Adam updates the rows in place
// Activations are kept transposed, [feature][sample] with Bp = 32 ceil(B / 32)
// samples, in global scratch read through L2 (another SM's L1 is not coherent);
// h alternates between two buffers by iteration and the shares by layer, so
// that one barrier separates every write from the next write of the buffer.
constexpr int TC = 8;               // CTAs of the cluster
constexpr int TRO = MAXW / TC;      // outputs per CTA at most
constexpr int TNT = 32 * TRO;       // threads: one warp per output
constexpr int TS = 36;              // row stride of the staged samples (16-byte rows, spread over banks)

struct TrainScratch {
  float* h;    // [2][nl][MAXW][Bp]
  float* z;    // [nl][MAXW][Bp]
  float* d;    // [2][MAXW][Bp]
  float* part; // [2][TC][MAXW][Bp]
  float* lossp;
};

// Adam's constants of an iteration and its update of one parameter
struct AdamK {
  float b1, b2, eps, a, ic2;  // lr / (1 - b1^t), 1 / sqrt(1 - b2^t)
  __device__ __forceinline__ AdamK(float lr, double p1, double p2)
      : b1(0.9f), b2(0.999f), eps(1e-8f), a(lr / (1.f - float(p1))), ic2(1.f / sqrtf(1.f - float(p2))) {}
  __device__ __forceinline__ void step(float* P, float* m, float* v, float g) const {
    const float mi = b1 * *m + (1.f - b1) * g, vi = b2 * *v + (1.f - b2) * g * g;
    *m = mi;
    *v = vi;
    *P -= __fdividef(a * mi, sqrtf(vi) * ic2 + eps);
  }
};

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__host__ __device__ inline int train_ld(int in) { return (in + 3) / 4 * 4; }  // row stride of W in shared memory

// where layer l starts in a copy of the CTA's rows (W, then b, of every layer,
// each layer a multiple of 16 bytes); l = nl: the floats of the copy
__host__ __device__ inline int train_off(const Net& net, int l) {
  int n = 0;
  for (int k = 0; k < l; ++k) n += (((net.sizes[k + 1] + TC - 1) / TC) * (train_ld(net.sizes[k]) + 1) + 3) / 4 * 4;
  return n;
}
__host__ __device__ inline int train_rows(const Net& net) { return train_off(net, net.nl); }

__global__ void __launch_bounds__(TNT, 1) k_mlp_train(const Net net, float* __restrict__ P, float* __restrict__ m,
                                                      float* __restrict__ v, const float* __restrict__ x,
                                                      const float* __restrict__ t, int B, int Bp, TrainScratch sc,
                                                      int iters, float lr, double p1, double p2, float* loss) {
  extern __shared__ __align__(16) float sm[];
  const int nr = train_rows(net), tid = threadIdx.x, lane = tid & 31, w = tid >> 5, c = blockIdx.x;
  float *sP = sm, *sM = sm + nr, *sV = sM + nr;
  float* hT = sV + nr;           // [MAXW][TS]
  float* dT = hT + MAXW * TS;    // [TRO][TS]
  float* zT = dT + TRO * TS;     // [4][TRO][32] partial sums of the forward pass
  __shared__ float red[TNT / 32];
  __shared__ int s_off[MAXL], s_o0[MAXL], s_no[MAXL];
  const int nl = net.nl, nout = net.sizes[nl];
  const float scale = 2.f / (float(B) * float(nout));
  // the CTA's rows of layer l: where they start in sP, their first output, their count
  auto rows = [&](int l, int& off, int& o0, int& no) {
    off = s_off[l];
    o0 = s_o0[l];
    no = s_no[l];
  };
  if (tid < nl) {
    const int ro = (net.sizes[tid + 1] + TC - 1) / TC;
    s_off[tid] = train_off(net, tid);
    s_o0[tid] = c * ro;
    s_no[tid] = max(0, min(ro, net.sizes[tid + 1] - c * ro));
  }
  for (int k = tid; k < 3 * nr; k += TNT) sm[k] = 0.f;
  __syncthreads();
  for (int l = 0; l < nl; ++l) {
    int off, o0, no;
    rows(l, off, o0, no);
    const int in = net.sizes[l], ld = train_ld(in), ro = (net.sizes[l + 1] + TC - 1) / TC;
    for (int k = tid; k < no * in; k += TNT) {
      const int o = k / in, i = k - o * in, to = off + o * ld + i;
      const long long g = net.woff[l] + (long long)(o0 + o) * in + i;
      sP[to] = P[g]; sM[to] = m[g]; sV[to] = v[g];
    }
    for (int o = tid; o < no; o += TNT) {
      const int to = off + ro * ld + o;
      const long long g = net.boff[l] + o0 + o;
      sP[to] = P[g]; sM[to] = m[g]; sV[to] = v[g];
    }
  }
  auto H = [&](int par, int l) { return sc.h + ((long long)par * nl + l) * MAXW * Bp; };
  auto Z = [&](int l) { return sc.z + (long long)l * MAXW * Bp; };
  auto D = [&](int l) { return sc.d + (long long)(l & 1) * MAXW * Bp; };
  auto S = [&](int l, int cta) { return sc.part + ((long long)(l & 1) * TC + cta) * MAXW * Bp; };
  // samples s0 .. s0 + 31 of layer l's input into hT (rows past the input are zero)
  auto stage = [&](int par, int l, int s0) {
    const int in = net.sizes[l], ld = train_ld(in);
    float q[MAXW * 32 / TNT];
#pragma unroll
    for (int k = 0; k < MAXW * 32 / TNT; ++k) {
      const int i = w + k * (TNT / 32);
      q[k] = 0.f;
      if (i < in && s0 + lane < B)
        q[k] = l == 0 ? x[(long long)(s0 + lane) * in + i] : __ldcg(H(par, l - 1) + (long long)i * Bp + s0 + lane);
    }
#pragma unroll
    for (int k = 0; k < MAXW * 32 / TNT; ++k) {
      const int i = w + k * (TNT / 32);
      if (i < ld) hT[i * TS + lane] = q[k];
    }
  };
  float lsum = 0.f;
  for (int it = 0; it < iters; ++it) {
    const int par = it & 1;
    p1 *= double(0.9f);
    p2 *= double(0.999f);
    const AdamK ad(lr, p1, p2);
    lsum = 0.f;
    // ---- forward
    for (int l = 0; l < nl; ++l) {
      int off, o0, no;
      rows(l, off, o0, no);
      const int ld = train_ld(net.sizes[l]), ro = (net.sizes[l + 1] + TC - 1) / TC;
      for (int s0 = 0; s0 < Bp; s0 += 32) {
        __syncthreads();
        stage(par, l, s0);
        __syncthreads();
        // four outputs and a quarter of the inputs per warp: a staged value
        // is read once for four multiply-adds; the quarters meet in zT
        {
          const int og = 4 * (w & 3), kq = w >> 2, n4 = ld >> 2;
          const int ia = 4 * (kq * n4 / 4), ib = 4 * ((kq + 1) * n4 / 4);
          if (og < no) {
            const float* W = sP + off + og * ld;
            const int w1 = og + 1 < no ? ld : 0, w2 = og + 2 < no ? 2 * ld : 0, w3 = og + 3 < no ? 3 * ld : 0;
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll 4
            for (int i = ia; i < ib; i += 4) {
              const float4 q0 = *reinterpret_cast<const float4*>(W + i), q1 = *reinterpret_cast<const float4*>(W + w1 + i),
                           q2 = *reinterpret_cast<const float4*>(W + w2 + i), q3 = *reinterpret_cast<const float4*>(W + w3 + i);
              const float h0 = hT[i * TS + lane], h1 = hT[(i + 1) * TS + lane], h2 = hT[(i + 2) * TS + lane],
                          h3 = hT[(i + 3) * TS + lane];
              a0 += q0.x * h0; a1 += q1.x * h0; a2 += q2.x * h0; a3 += q3.x * h0;
              a0 += q0.y * h1; a1 += q1.y * h1; a2 += q2.y * h1; a3 += q3.y * h1;
              a0 += q0.z * h2; a1 += q1.z * h2; a2 += q2.z * h2; a3 += q3.z * h2;
              a0 += q0.w * h3; a1 += q1.w * h3; a2 += q2.w * h3; a3 += q3.w * h3;
            }
            float* zq = zT + (kq * TRO + og) * 32 + lane;
            zq[0] = a0; zq[32] = a1; zq[64] = a2; zq[96] = a3;
          }
        }
        __syncthreads();
        if (w < no) {
          const float* zq = zT + w * 32 + lane;
          const float a = sP[off + ro * ld + w] +
                          ((zq[0] + zq[TRO * 32]) + (zq[2 * TRO * 32] + zq[3 * TRO * 32]));
          const long long g = (long long)(o0 + w) * Bp + s0 + lane;
          if (l < nl - 1) {
            Z(l)[g] = a;
            __stcg(H(par, l) + g, gelu(a));
          } else {
            float e = 0.f;
            if (s0 + lane < B) e = a - t[(long long)(s0 + lane) * nout + o0 + w];
            lsum += e * e;
            D(l)[g] = e * scale;
          }
        }
      }
      if (l < nl - 1) cluster_sync();
    }
    // ---- backward
    for (int l = nl - 1; l >= 0; --l) {
      int off, o0, no;
      rows(l, off, o0, no);
      const int in = net.sizes[l], ld = train_ld(in), ro = (net.sizes[l + 1] + TC - 1) / TC;
      __syncthreads();
      if (l > 0) {
        // this CTA's share of W^T d: eight inputs per warp
        for (int s0 = 0; s0 < Bp; s0 += 32) {
          float d[TRO];
#pragma unroll
          for (int o = 0; o < TRO; ++o) d[o] = o < no ? D(l)[(long long)(o0 + o) * Bp + s0 + lane] : 0.f;
          const int i0 = w * 8;
          if (i0 < in) {
            float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int o = 0; o < TRO; ++o) {
              if (o >= no) break;
              const float* W = sP + off + o * ld + i0;
              const float4 q = *reinterpret_cast<const float4*>(W);
              a[0] += q.x * d[o]; a[1] += q.y * d[o]; a[2] += q.z * d[o]; a[3] += q.w * d[o];
              if (i0 + 4 < ld) {
                const float4 r = *reinterpret_cast<const float4*>(W + 4);
                a[4] += r.x * d[o]; a[5] += r.y * d[o]; a[6] += r.z * d[o]; a[7] += r.w * d[o];
              }
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (i0 + k < in) __stcg(S(l, c) + (long long)(i0 + k) * Bp + s0 + lane, a[k]);
          }
        }
        cluster_sync();
        // d of the layer below at this CTA's outputs there
        int offp, p0, np;
        rows(l - 1, offp, p0, np);
        for (int s0 = 0; s0 < Bp; s0 += 32)
          if (w < np) {
            const long long g = (long long)(p0 + w) * Bp + s0 + lane;
            float q[TC];
#pragma unroll
            for (int k = 0; k < TC; ++k) q[k] = __ldcg(S(l, k) + g);
            float a = 0.f;
#pragma unroll
            for (int k = 0; k < TC; ++k) a += q[k];
            D(l - 1)[g] = s0 + lane < B ? a * gelu_d(Z(l - 1)[g]) : 0.f;
          }
      }
      // dW, db over the samples, then Adam; thread: input i, outputs 4 og .. + 3
      const int i = tid & (MAXW - 1), og = tid / MAXW;
      float a[4] = {0.f, 0.f, 0.f, 0.f}, ab = 0.f;
      for (int s0 = 0; s0 < Bp; s0 += 32) {
        if (s0 > 0) __syncthreads();
        stage(par, l, s0);
        for (int k = tid; k < TRO * 32; k += TNT) {
          const int o = k >> 5, s = k & 31;
          dT[o * TS + s] = o < no ? D(l)[(long long)(o0 + o) * Bp + s0 + s] : 0.f;
        }
        __syncthreads();
        if (i < in)
#pragma unroll
          for (int s = 0; s < 32; s += 4) {
            const float4 q = *reinterpret_cast<const float4*>(hT + i * TS + s);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float4 e = *reinterpret_cast<const float4*>(dT + (4 * og + k) * TS + s);
              a[k] += (e.x * q.x + e.y * q.y) + (e.z * q.z + e.w * q.w);
            }
          }
        if (tid < no)
          for (int s = 0; s < 32; ++s) ab += dT[tid * TS + s];
      }
      if (i < in)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (4 * og + k < no) ad.step(sP + off + (4 * og + k) * ld + i, sM + off + (4 * og + k) * ld + i, sV + off + (4 * og + k) * ld + i, a[k]);
      if (tid < no) ad.step(sP + off + ro * ld + tid, sM + off + ro * ld + tid, sV + off + ro * ld + tid, ab);
    }
  }
  // the loss of the last evaluated parameters, then the rows back
  for (int k = 16; k > 0; k >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, k);
  if (lane == 0) red[w] = lsum;
  __syncthreads();
  if (tid == 0) {
    float a = 0.f;
    for (int k = 0; k < TNT / 32; ++k) a += red[k];
    __stcg(sc.lossp + c, a);
  }
  for (int l = 0; l < nl; ++l) {
    int off, o0, no;
    rows(l, off, o0, no);
    const int in = net.sizes[l], ld = train_ld(in), ro = (net.sizes[l + 1] + TC - 1) / TC;
    for (int k = tid; k < no * in; k += TNT) {
      const int o = k / in, i = k - o * in, to = off + o * ld + i;
      const long long g = net.woff[l] + (long long)(o0 + o) * in + i;
      P[g] = sP[to]; m[g] = sM[to]; v[g] = sV[to];
    }
    for (int o = tid; o < no; o += TNT) {
      const int to = off + ro * ld + o;
      const long long g = net.boff[l] + o0 + o;
      P[g] = sP[to]; m[g] = sM[to]; v[g] = sV[to];
    }
  }
  cluster_sync();
  if (c == 0 && tid == 0 && iters > 0) {
    float a = 0.f;
    for (int k = 0; k < TC; ++k) a += __ldcg(sc.lossp + k);
    *loss = a / (float(B) * float(nout));
  }
}

// The same for up to 32 samples (one per lane) and networks whose layers fit
// beside each other in shared memory: every layer's input stays staged for the
// backward pass, and what another CTA needs is stored straight into its shared
// memory, so that a barrier is all that lies between two layers (31 samples of
// the 4-128-128-128-64 network: 18 us an iteration against 29 through L2).
//  hT     [nl + 1][MAXW][TS] inputs of the layers; the first hidden one twice,
//         by iteration: it is stored before an iteration's first barrier, when
//         another CTA may still be in the last backward pass (every other
//         buffer's next store lies behind a barrier)
//  part   [2][TC][TRO][32] shares of W^T d at this CTA's inputs, by layer parity
__host__ __device__ inline int one_floats(const Net& net) {
  return 3 * train_rows(net) + ((net.nl + 1) * MAXW + 2 * TRO) * TS + 2 * TC * TRO * 32 + net.nl * TRO * 32 + 4 * TRO * 32;
}

// address of this CTA's shared variable p in CTA `cta` of the cluster
__device__ __forceinline__ unsigned remote(const float* p, int cta) {
  unsigned a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(unsigned(__cvta_generic_to_shared(p))), "r"(cta));
  return a;
}
__device__ __forceinline__ void st_remote(unsigned a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

__global__ void __launch_bounds__(TNT, 1) k_mlp_train_one(const Net net, float* __restrict__ P, float* __restrict__ m,
                                                          float* __restrict__ v, const float* __restrict__ x,
                                                          const float* __restrict__ t, int B, float* lossp, int iters,
                                                          float lr, double p1, double p2, float* loss) {
  extern __shared__ __align__(16) float sm[];
  const int nr = train_rows(net), tid = threadIdx.x, lane = tid & 31, w = tid >> 5, c = blockIdx.x;
  const int nl = net.nl, nout = net.sizes[nl];
  float *sP = sm, *sM = sm + nr, *sV = sM + nr;
  float* hT = sV + nr;                       // layer l's input: slot l, the first hidden one slot 1 or nl
  float* dT = hT + (nl + 1) * MAXW * TS;     // [2][TRO][TS]
  float* part = dT + 2 * TRO * TS;
  float* zs = part + 2 * TC * TRO * 32;      // [nl][TRO][32]
  float* zT = zs + nl * TRO * 32;            // [4][TRO][32]
  __shared__ float red[TNT / 32];
  __shared__ int s_off[MAXL], s_ro[MAXL];
  const float scale = 2.f / (float(B) * float(nout));
  for (int k = tid; k < one_floats(net); k += TNT) sm[k] = 0.f;
  if (tid < nl) {
    s_off[tid] = train_off(net, tid);
    s_ro[tid] = (net.sizes[tid + 1] + TC - 1) / TC;
  }
  __syncthreads();
  // outputs per CTA of layer l, this CTA's first one and their count
  auto cnt = [&](int l) { return max(0, min(s_ro[l], net.sizes[l + 1] - c * s_ro[l])); };
  for (int l = 0; l < nl; ++l) {
    const int off = s_off[l], o0 = c * s_ro[l], no = cnt(l), in = net.sizes[l], ld = train_ld(in);
    for (int k = tid; k < no * in; k += TNT) {
      const int o = k / in, i = k - o * in, to = off + o * ld + i;
      const long long g = net.woff[l] + (long long)(o0 + o) * in + i;
      sP[to] = P[g]; sM[to] = m[g]; sV[to] = v[g];
    }
    for (int o = tid; o < no; o += TNT) {
      const int to = off + s_ro[l] * ld + o;
      const long long g = net.boff[l] + o0 + o;
      sP[to] = P[g]; sM[to] = m[g]; sV[to] = v[g];
    }
  }
  for (int k = tid; k < net.sizes[0] * 32; k += TNT) {
    const int i = k >> 5, s = k & 31;
    if (s < B) hT[i * TS + s] = x[(long long)s * net.sizes[0] + i];
  }
  const float tgt = lane < B && w < cnt(nl - 1) ? t[(long long)lane * nout + c * s_ro[nl - 1] + w] : 0.f;
  auto slot = [&](int l, int it) { return hT + (l == 1 && (it & 1) ? nl : l) * MAXW * TS; };
  cluster_sync();  // every CTA's buffers are zeroed before anything is stored into them
  float lsum = 0.f;
  for (int it = 0; it < iters; ++it) {
    p1 *= double(0.9f);
    p2 *= double(0.999f);
    const AdamK ad(lr, p1, p2);
    // ---- forward
    for (int l = 0; l < nl; ++l) {
      const int off = s_off[l], no = cnt(l), ld = train_ld(net.sizes[l]);
      const float* h = slot(l, it);
      const int og = 4 * (w & 3), kq = w >> 2, n4 = ld >> 2;
      const int ia = 4 * (kq * n4 / 4), ib = 4 * ((kq + 1) * n4 / 4);
      if (og < no) {
        const float* W = sP + off + og * ld;
        const int w1 = og + 1 < no ? ld : 0, w2 = og + 2 < no ? 2 * ld : 0, w3 = og + 3 < no ? 3 * ld : 0;
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll 4
        for (int i = ia; i < ib; i += 4) {
          const float4 q0 = *reinterpret_cast<const float4*>(W + i), q1 = *reinterpret_cast<const float4*>(W + w1 + i),
                       q2 = *reinterpret_cast<const float4*>(W + w2 + i), q3 = *reinterpret_cast<const float4*>(W + w3 + i);
          const float h0 = h[i * TS + lane], h1 = h[(i + 1) * TS + lane], h2 = h[(i + 2) * TS + lane],
                      h3 = h[(i + 3) * TS + lane];
          a0 += q0.x * h0; a1 += q1.x * h0; a2 += q2.x * h0; a3 += q3.x * h0;
          a0 += q0.y * h1; a1 += q1.y * h1; a2 += q2.y * h1; a3 += q3.y * h1;
          a0 += q0.z * h2; a1 += q1.z * h2; a2 += q2.z * h2; a3 += q3.z * h2;
          a0 += q0.w * h3; a1 += q1.w * h3; a2 += q2.w * h3; a3 += q3.w * h3;
        }
        float* zq = zT + (kq * TRO + og) * 32 + lane;
        zq[0] = a0; zq[32] = a1; zq[64] = a2; zq[96] = a3;
      }
      __syncthreads();
      if (w < no) {
        const float* zq = zT + w * 32 + lane;
        const float a = sP[off + s_ro[l] * ld + w] + ((zq[0] + zq[TRO * 32]) + (zq[2 * TRO * 32] + zq[3 * TRO * 32]));
        if (l < nl - 1) {
          zs[(l * TRO + w) * 32 + lane] = a;
          const float g = lane < B ? gelu(a) : 0.f;
          const float* to = slot(l + 1, it) + (c * s_ro[l] + w) * TS + lane;
#pragma unroll
          for (int k = 0; k < TC; ++k) st_remote(remote(to, k), g);
        } else {
          const float e = lane < B ? a - tgt : 0.f;
          lsum = e * e;
          dT[((l & 1) * TRO + w) * TS + lane] = e * scale;
        }
      }
      if (l < nl - 1) cluster_sync();
    }
    __syncthreads();
    // ---- backward
    for (int l = nl - 1; l >= 0; --l) {
      const int off = s_off[l], no = cnt(l), in = net.sizes[l], ld = train_ld(in);
      const float* d0 = dT + (l & 1) * TRO * TS;
      if (l > 0) {
        // this CTA's share of W^T d, eight inputs per warp, to the CTAs that own them
        const int i0 = w * 8;
        if (i0 < in) {
          float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
          for (int o = 0; o < no; ++o) {
            const float d = d0[o * TS + lane];
            const float* W = sP + off + o * ld + i0;
            const float4 q = *reinterpret_cast<const float4*>(W);
            a[0] += q.x * d; a[1] += q.y * d; a[2] += q.z * d; a[3] += q.w * d;
            if (i0 + 4 < ld) {
              const float4 r = *reinterpret_cast<const float4*>(W + 4);
              a[4] += r.x * d; a[5] += r.y * d; a[6] += r.z * d; a[7] += r.w * d;
            }
          }
          const int rp = s_ro[l - 1];
          const float* mine = part + ((l & 1) * TC + c) * TRO * 32 + lane;
          int own = i0 / rp, at = i0 - own * rp;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            if (i0 + k < in) st_remote(remote(mine + at * 32, own), a[k]);
            if (++at == rp) { at = 0; ++own; }
          }
        }
        cluster_sync();
        // d of the layer below at this CTA's outputs there
        if (w < cnt(l - 1)) {
          const float* q = part + (l & 1) * TC * TRO * 32 + w * 32 + lane;
          float a = 0.f;
#pragma unroll
          for (int k = 0; k < TC; ++k) a += q[k * TRO * 32];
          dT[(((l - 1) & 1) * TRO + w) * TS + lane] = lane < B ? a * gelu_d(zs[((l - 1) * TRO + w) * 32 + lane]) : 0.f;
        }
      }
      // dW, db over the samples, then Adam; thread: input i, outputs 4 og .. + 3
      const int i = tid & (MAXW - 1), og = tid / MAXW;
      const float* h = slot(l, it) + i * TS;
      if (i < in && 4 * og < no) {
        float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int s = 0; s < 32; s += 4) {
          const float4 q = *reinterpret_cast<const float4*>(h + s);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float4 e = *reinterpret_cast<const float4*>(d0 + (4 * og + k) * TS + s);
            a[k] += (e.x * q.x + e.y * q.y) + (e.z * q.z + e.w * q.w);
          }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (4 * og + k < no) {
            const int at = off + (4 * og + k) * ld + i;
            ad.step(sP + at, sM + at, sV + at, a[k]);
          }
      }
      if (tid < no) {
        float ab = 0.f;
#pragma unroll
        for (int s = 0; s < 32; s += 4) {
          const float4 e = *reinterpret_cast<const float4*>(d0 + tid * TS + s);
          ab += (e.x + e.y) + (e.z + e.w);
        }
        const int at = off + s_ro[l] * ld + tid;
        ad.step(sP + at, sM + at, sV + at, ab);
      }
      __syncthreads();
    }
  }
  // the loss of the last evaluated parameters, then the rows back
  for (int k = 16; k > 0; k >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, k);
  if (lane == 0) red[w] = lsum;
  __syncthreads();
  if (tid == 0) {
    float a = 0.f;
    for (int k = 0; k < TNT / 32; ++k) a += red[k];
    __stcg(lossp + c, a);
  }
  for (int l = 0; l < nl; ++l) {
    const int off = s_off[l], o0 = c * s_ro[l], no = cnt(l), in = net.sizes[l], ld = train_ld(in);
    for (int k = tid; k < no * in; k += TNT) {
      const int o = k / in, i = k - o * in, to = off + o * ld + i;
      const long long g = net.woff[l] + (long long)(o0 + o) * in + i;
      P[g] = sP[to]; m[g] = sM[to]; v[g] = sV[to];
    }
    for (int o = tid; o < no; o += TNT) {
      const int to = off + s_ro[l] * ld + o;
      const long long g = net.boff[l] + o0 + o;
      P[g] = sP[to]; m[g] = sM[to]; v[g] = sV[to];
    }
  }
  cluster_sync();
  if (c == 0 && tid == 0 && iters > 0) {
    float a = 0.f;
    for (int k = 0; k < TC; ++k) a += __ldcg(lossp + k);
    *loss = a / (float(B) * float(nout));
  }
}

}  // namespace

struct lbm_mlp {
  Net net{};
  long long nparam = 0;
  int max_batch = 0;
  cudaStream_t stream = nullptr;
  lbm_allocator alloc{};
  float *P = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr, *gpart = nullptr, *lpart = nullptr;
  float *x = nullptr, *t = nullptr, *y = nullptr, *zs = nullptr, *hs = nullptr, *loss = nullptr;
  size_t act_floats = 0;
  float* train = nullptr;  // scratch of k_mlp_train (null: training on the separate passes)
  int train_max = 0;       // samples up to which training runs in one launch
  int ndata = 0;
  int adam_t = 0;
  std::vector<std::pair<void*, size_t>> blocks;
};

// dynamic shared memory and scratch of k_mlp_train
static size_t train_smem(const Net& net) { return size_t(3 * train_rows(net) + (MAXW + TRO) * TS + 4 * TRO * 32) * 4; }
static size_t train_floats(const Net& net, int Bp) { return size_t(3 * net.nl + 2 + 2 * TC) * MAXW * Bp + TC; }

static void free_cb(void* p, size_t, void*) { cudaFree(p); }

// Samples up to which training runs in one launch (a multiple of 32).  Eight CTAs take
// blocks of 32 samples in turn, the separate passes a CTA per block: theirs is a fixed
// time up to thousands of samples, long where layers are wide.  Both as fitted, us an
// iteration: 12 + per layer 4.5 + 130 in out / 128^2 (60 for the first, which hands
// nothing back) against, per block, 2.4 a layer + 3.1 in out / 128^2 (4.6).  Measured,
// separate and one launch: 4-128-128-128-64 with 512 samples 398 and 270, 640 399 and
// 335, 1024 402 and 532; 128-128 320 77 and 71, 384 77 and 86; 4-64-64-64 256 94 and
// 78, 384 94 and 113; 4-16-16-2 96 32 and 28, 128 32 and 35; 1-1 160 17 and 10, 384 17
// and 21.
static int train_limit(const Net& net) {
  double passes = 12.0, block = 0.0;
  for (int l = 0; l < net.nl; ++l) {
    const double p = double(net.sizes[l]) * net.sizes[l + 1] / (128.0 * 128.0);
    passes += 4.5 + (l == 0 ? 60.0 : 130.0) * p;
    block += 2.4 + (l == 0 ? 4.6 : 3.1) * p;
  }
  return 32 * int(std::max(1.0, passes / block));
}

static float* mget(lbm_mlp* m, size_t floats) {
  const size_t b = floats * 4 + 256;
  void* p = m->alloc.alloc(b, m->alloc.ctx);
  if (p) m->blocks.push_back({p, b});
  return static_cast<float*>(p);
}

extern "C" void lbm_mlp_destroy(lbm_mlp* m) {
  if (!m) return;
  cudaStreamSynchronize(m->stream);
  for (auto& b : m->blocks) m->alloc.free(b.first, b.second, m->alloc.ctx);
  delete m;
}

extern "C" int lbm_mlp_create(const int* sizes, int nlayers, int max_batch, void* stream, const lbm_allocator* alloc,
                              lbm_mlp** out) {
  if (!out || !sizes || nlayers < 1 || nlayers > MAXL || max_batch < 1) return LBM_EINVAL;
  *out = nullptr;
  for (int l = 0; l <= nlayers; ++l)
    if (sizes[l] < 1 || sizes[l] > MAXW) return LBM_EINVAL;
  lbm_mlp* m = new (std::nothrow) lbm_mlp();
  if (!m) return LBM_ENOMEM;
  m->stream = static_cast<cudaStream_t>(stream);
  if (alloc && alloc->alloc && alloc->free) m->alloc = *alloc;
  else { m->alloc.alloc = lbmd::device_malloc; m->alloc.free = free_cb; m->alloc.ctx = nullptr; }
  m->net.nl = nlayers;
  long long off = 0;
  size_t act = 0;
  for (int l = 0; l <= nlayers; ++l) m->net.sizes[l] = sizes[l];
  for (int l = 0; l < nlayers; ++l) {
    m->net.woff[l] = off;
    off += (long long)sizes[l + 1] * sizes[l];
    m->net.boff[l] = off;
    off += sizes[l + 1];
    act += size_t(sizes[l + 1]);
  }
  m->nparam = off;
  m->max_batch = max_batch;
  m->act_floats = act * size_t(max_batch);
  const int nblk = (max_batch + SB - 1) / SB;
  m->P = mget(m, off);
  m->m = mget(m, off);
  m->v = mget(m, off);
  m->grad = mget(m, off);
  m->gpart = mget(m, size_t(off) * nblk);
  m->lpart = mget(m, size_t(nblk));
  m->x = mget(m, size_t(max_batch) * sizes[0]);
  m->t = mget(m, size_t(max_batch) * sizes[nlayers]);
  m->y = mget(m, size_t(max_batch) * sizes[nlayers]);
  m->zs = mget(m, m->act_floats);
  m->hs = mget(m, m->act_floats);
  m->loss = mget(m, 1);
  if (!m->P || !m->m || !m->v || !m->grad || !m->gpart || !m->lpart || !m->x || !m->t || !m->y || !m->zs || !m->hs ||
      !m->loss) {
    lbm_mlp_destroy(m);
    return LBM_ENOMEM;
  }
  m->train_max = std::min(train_limit(m->net), (max_batch + 31) / 32 * 32);
  if (train_smem(m->net) <= size_t(227) * 1024) m->train = mget(m, train_floats(m->net, m->train_max));
  cudaMemsetAsync(m->m, 0, size_t(off) * 4, m->stream);
  cudaMemsetAsync(m->v, 0, size_t(off) * 4, m->stream);
  if (cudaStreamSynchronize(m->stream) != cudaSuccess) { lbm_mlp_destroy(m); return LBM_ECUDA; }
  *out = m;
  return LBM_OK;
}

extern "C" long long lbm_mlp_param_count(const lbm_mlp* m) { return m ? m->nparam : -1; }

extern "C" int lbm_mlp_set_params(lbm_mlp* m, const float* host) {
  if (!m || !host) return LBM_EINVAL;
  cudaError_t e = cudaMemcpyAsync(m->P, host, size_t(m->nparam) * 4, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->m, 0, size_t(m->nparam) * 4, m->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->v, 0, size_t(m->nparam) * 4, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  m->adam_t = 0;
  return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

extern "C" int lbm_mlp_get_params(lbm_mlp* m, float* host) {
  if (!m || !host) return LBM_EINVAL;
  cudaError_t e = cudaMemcpyAsync(host, m->P, size_t(m->nparam) * 4, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

static cudaError_t run_forward(lbm_mlp* m, const float* dx, int B, float* dy) {
  const int nblk = (B + SB - 1) / SB;
  k_mlp_forward<<<nblk, 128, 0, m->stream>>>(m->net, m->P, dx, B, dy, m->zs, m->hs);
  return cudaGetLastError();
}

static cudaError_t run_grad(lbm_mlp* m, const float* dx, const float* dt, int B) {
  cudaError_t e = run_forward(m, dx, B, m->y);
  if (e != cudaSuccess) return e;
  const int nblk = (B + SB - 1) / SB;
  k_mlp_backward<<<nblk, 256, 0, m->stream>>>(m->net, m->P, dx, dt, B, m->y, m->zs, m->hs, m->gpart, m->nparam,
                                              m->lpart);
  const int nout = m->net.sizes[m->net.nl];
  k_reduce<<<unsigned((m->nparam + 255) / 256), 256, 0, m->stream>>>(m->gpart, nblk, m->nparam, m->grad, m->lpart,
                                                                      m->loss, 1.f / (float(B) * float(nout)));
  return cudaGetLastError();
}

extern "C" int lbm_mlp_forward(lbm_mlp* m, const float* host_x, int batch, float* host_y) {
  if (!m || !host_x || !host_y || batch < 1 || batch > m->max_batch) return LBM_EINVAL;
  const int in = m->net.sizes[0], out = m->net.sizes[m->net.nl];
  cudaError_t e = cudaMemcpyAsync(m->x, host_x, size_t(batch) * in * 4, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = run_forward(m, m->x, batch, m->y);
  if (e == cudaSuccess) e = cudaMemcpyAsync(host_y, m->y, size_t(batch) * out * 4, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

extern "C" int lbm_mlp_loss_grad(lbm_mlp* m, const float* host_x, const float* host_t, int batch, float* host_loss,
                                 float* host_grad) {
  if (!m || !host_x || !host_t || batch < 1 || batch > m->max_batch) return LBM_EINVAL;
  const int in = m->net.sizes[0], out = m->net.sizes[m->net.nl];
  cudaError_t e = cudaMemcpyAsync(m->x, host_x, size_t(batch) * in * 4, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(m->t, host_t, size_t(batch) * out * 4, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = run_grad(m, m->x, m->t, batch);
  if (e == cudaSuccess && host_grad)
    e = cudaMemcpyAsync(host_grad, m->grad, size_t(m->nparam) * 4, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess && host_loss) e = cudaMemcpyAsync(host_loss, m->loss, 4, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

extern "C" int lbm_mlp_set_data(lbm_mlp* m, const float* host_x, const float* host_t, int n) {
  if (!m || !host_x || !host_t || n < 1 || n > m->max_batch) return LBM_EINVAL;
  const int in = m->net.sizes[0], out = m->net.sizes[m->net.nl];
  cudaError_t e = cudaMemcpyAsync(m->x, host_x, size_t(n) * in * 4, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(m->t, host_t, size_t(n) * out * 4, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  m->ndata = n;
  return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

// n iterations by k_mlp_train_one where the samples and the network fit it, else
// by k_mlp_train; false (nothing launched) if it cannot be launched
static bool launch_train(lbm_mlp* m, int n, float lr) {
  const int B = m->ndata, Bp = (B + 31) / 32 * 32;
  const bool one = B <= 32 && size_t(one_floats(m->net)) * 4 <= size_t(227) * 1024;
  const size_t smem = one ? size_t(one_floats(m->net)) * 4 : train_smem(m->net);
  const void* fn = one ? reinterpret_cast<const void*>(k_mlp_train_one) : reinterpret_cast<const void*>(k_mlp_train);
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  TrainScratch sc;
  sc.h = m->train;
  sc.z = sc.h + size_t(2) * m->net.nl * MAXW * Bp;
  sc.d = sc.z + size_t(m->net.nl) * MAXW * Bp;
  sc.part = sc.d + size_t(2) * MAXW * Bp;
  sc.lossp = sc.part + size_t(2) * TC * MAXW * Bp;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = TC;
  cfg.blockDim = TNT;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = m->stream;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = TC;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const double p1 = std::pow(double(0.9f), double(m->adam_t)), p2 = std::pow(double(0.999f), double(m->adam_t));
  const float *dx = m->x, *dt = m->t;
  const cudaError_t e =
      one ? cudaLaunchKernelEx(&cfg, k_mlp_train_one, m->net, m->P, m->m, m->v, dx, dt, B, sc.lossp, n, lr, p1, p2, m->loss)
          : cudaLaunchKernelEx(&cfg, k_mlp_train, m->net, m->P, m->m, m->v, dx, dt, B, Bp, sc, n, lr, p1, p2, m->loss);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  m->adam_t += n;
  return true;
}

// iters full-batch Adam steps on the data set by lbm_mlp_set_data; the final
// loss (of the parameters before the last update) is returned in *host_loss
extern "C" int lbm_mlp_train(lbm_mlp* m, int iters, float lr, float* host_loss) {
  if (!m || iters < 0 || m->ndata < 1) return LBM_EINVAL;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  // a launch per 2000 iterations (some tens of milliseconds): other work on
  // the GPU's queue is not kept waiting by a long training call
  int done = 0;
  while (m->train && m->ndata <= m->train_max && done < iters) {
    const int n = iters - done < 2000 ? iters - done : 2000;
    if (!launch_train(m, n, lr)) break;
    done += n;
  }
  for (int it = done; it < iters; ++it) {
    cudaError_t e = run_grad(m, m->x, m->t, m->ndata);
    if (e != cudaSuccess) return LBM_ECUDA;
    m->adam_t += 1;
    const float c1 = 1.f - std::pow(b1, float(m->adam_t)), c2 = 1.f - std::pow(b2, float(m->adam_t));
    k_adam<<<unsigned((m->nparam + 255) / 256), 256, 0, m->stream>>>(m->nparam, m->P, m->m, m->v, m->grad, lr, b1, b2,
                                                                      eps, c1, c2);
    if (cudaGetLastError() != cudaSuccess) return LBM_ECUDA;
  }
  cudaError_t e = cudaSuccess;
  if (host_loss) e = cudaMemcpyAsync(host_loss, m->loss, 4, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
}
