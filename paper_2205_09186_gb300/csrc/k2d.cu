// Instantiations of the fused D2Q9 step for the explicit and isotropic schemes.
#include <type_traits>

#include <cstdint>

#include "launch.cuh"
#include "step2d.cuh"
#include "step2d_node.cuh"
#include "step2d_split.cuh"

namespace lbmd {

constexpr int TX2 = 32, TY2 = 8;

namespace {

template <int S, class P, int MODE>
cudaError_t launch_mode(const Launch& c, int* nblocks) {
  using Sh = Step2DShape<S, P, TX2, TY2>;
  auto k = k_step2d<S, P, TX2, TY2, MODE>;
  if (cudaError_t e = ensure_smem(k, Sh::bytes); e != cudaSuccess) return e;
  dim3 grid((c.kp.nx + TX2 - 1) / TX2, (c.kp.ny + TY2 - 1) / TY2, 1);
  if (nblocks) *nblocks = int(grid.x * grid.y);
  using Tf = typename P::Tf;
  using Tr = typename P::Tr;
  k<<<grid, NT2, Sh::bytes, c.stream>>>(c.kp, static_cast<const Tf*>(c.fin), static_cast<Tf*>(c.fout),
                                        static_cast<const Tr*>(c.rin), static_cast<Tr*>(c.rout),
                                        c.aux, c.fo, c.gi, c.mrt);
  return cudaGetLastError();
}

// FP32 deviation storage with FP32 mu: mu pass + row-per-warp collision pass,
// tiles of RPT rows per thread
template <int S, bool TAU1, int RPT>
cudaError_t launch_split2d_t(const Launch& c, int* nblocks) {
  using Sh = Split2DShape<S, RPT>;
  constexpr int M2Y = Tile2<RPT>::M2Y, T2Y = Tile2<RPT>::T2Y;
  if (cudaError_t e = ensure_smem(k_mu2d<S, RPT>, Sh::bytes); e != cudaSuccess) return e;
  if (cudaError_t e = ensure_smem(k_coll2d<S, TAU1, RPT>, Sh::bytes); e != cudaSuccess) return e;
  // overlapped launches, except where an isotropic scheme's tiles find an SM each: a
  // launch's blocks are dealt while those before still run, two then share an SM
  // (E8 at tau 0.9, us a step overlapped and not: 300^2 14.9 and 12.3, 420^2 12.5 and
  // 16.4, 600^2 19.0 and 20.6; EFDS6 at tau 0.8: 300^2 8.6 to 11.7 and 12.3, 512^2
  // 14.1 and 17.8, 1024^2 32.8 and 36.2).  Nor where the SMs hold more than one and a
  // half to two tiles each and the second of them waits for longer than a launch: the
  // widest stencil behind its vector mu pass, and it and the isotropic ones on
  // lattices of two tile rows (EFDS6 at tau 1: 3600 x 40 14.8 and 12.4, 900 x 240 14.8
  // and 14.4; 900 x 210 12.1 and 14.4, 700 x 390 13.1 and 16.4; E8 4000 x 40 15.3 and
  // 14.4; EFDS4 12.2 and 12.3)
  const dim3 gc((c.kp.nx + T2X - 1) / T2X, (c.kp.ny + T2Y - 1) / T2Y);
  const long long tiles = (long long)gc.x * gc.y, sms = device_sms();
  const bool wide = Sch<S>::R == 3, two = 2 * tiles > 3 * sms && tiles <= 2 * sms;
  const bool late = two && ((wide && c.kp.nx % 4 == 0 && !c.mrt.on) || (gc.y <= 2 && (wide || Sch<S>::ISO)));
  const bool pdl = !late && (!Sch<S>::ISO || tiles > sms);
  cudaError_t e = cudaSuccess;
  if constexpr (!Sch<S>::ISO) {
    if (c.kp.nx % 4 == 0 && (reinterpret_cast<uintptr_t>(c.rin) & 15) == 0 && (reinterpret_cast<uintptr_t>(c.mu) & 15) == 0) {
      // rows per thread: about four CTAs of 8 warps per SM, 2..32 rows
      const int gx = (c.kp.nx + 63) / 64;
      const int sms = device_sms();
      const int want_gy = (4 * sms + gx - 1) / gx;
      int rows = (c.kp.ny + 16 * want_gy - 1) / (16 * want_gy);
      rows = rows < 2 ? 2 : (rows > 32 ? 32 : rows);
      dim3 gm(gx, (c.kp.ny + 16 * rows - 1) / (16 * rows));
      e = launch_if_pdl(pdl, k_mu2d_ym<S>, gm, YMT, 0, c.stream, c.kp, static_cast<const float*>(c.rin), static_cast<float*>(c.mu),
                     rows);
    } else {
      dim3 gm((c.kp.nx + M2X - 1) / M2X, (c.kp.ny + M2Y - 1) / M2Y);
      e = launch_if_pdl(pdl, k_mu2d<S, RPT>, gm, NT2S, Sh::bytes, c.stream, c.kp, static_cast<const float*>(c.rin),
                     static_cast<float*>(c.mu));
    }
  } else {
    dim3 gm((c.kp.nx + M2X - 1) / M2X, (c.kp.ny + M2Y - 1) / M2Y);
    e = launch_if_pdl(pdl, k_mu2d<S, RPT>, gm, NT2S, Sh::bytes, c.stream, c.kp, static_cast<const float*>(c.rin),
                   static_cast<float*>(c.mu));
  }
  if (e != cudaSuccess) return e;
  if (c.ev_mid) cudaEventRecord(c.ev_mid, c.stream);
  if (nblocks) *nblocks = int(gc.x * gc.y);
  return launch_if_pdl(pdl, k_coll2d<S, TAU1, RPT>, gc, NT2S, Sh::bytes, c.stream, c.kp, static_cast<const float*>(c.fin),
                    static_cast<float*>(c.fout), static_cast<const float*>(c.rin), static_cast<const float*>(c.mu),
                    static_cast<float*>(c.rout), c.aux, c.mrt);
}

// Whether a step runs on node-parallel passes (step2d_node.cuh) or on the tiled mu
// and collision passes: us a step at tau 0.8 on the tiled passes and here, 64^2 EFDS6
// 8.0 and 5.1, 128^2 8.3 and 5.2, 200^2 8.8 and 7.9, 256^2 10.8 and 11.4; E8 at tau
// 0.9, 64^2 7.5 and 5.9, 128^2 7.9 and 7.1, 200^2 9.9 and 10.8.
bool node2_rule(const KParams& kp) { return kp.n <= 32768; }

// the three node-parallel passes (step2d_node.cuh)
template <int S>
cudaError_t launch_node2(const Launch& c, int* nblocks) {
  const KParams& kp = c.kp;
  const int g = int((kp.n + NODE2_T - 1) / NODE2_T);
  if (nblocks) *nblocks = g;
  const unsigned mx = unsigned(((1ull << 32) + kp.nx - 1) / kp.nx);
  const float *fin = static_cast<const float*>(c.fin), *rin = static_cast<const float*>(c.rin);
  float *fout = static_cast<float*>(c.fout), *rout = static_cast<float*>(c.rout), *mu = static_cast<float*>(c.mu);
  cudaError_t e = launch_pdl(k_node2_mu<S>, g, NODE2_T, 0, c.stream, kp, mx, rin, mu);
  if (e != cudaSuccess) return e;
  if (c.ev_mid) cudaEventRecord(c.ev_mid, c.stream);
  auto k = c.mrt.on ? k_node2_coll<S, 2> : (kp.omega == 1.0 ? k_node2_coll<S, 0> : k_node2_coll<S, 1>);
  e = launch_pdl(k, g, NODE2_T, 0, c.stream, kp, mx, fin, fout, rin, mu, c.aux.bad_step, c.aux.t, c.mrt);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_node2_rho, g, NODE2_T, 0, c.stream, kp, fout, rout, c.aux.bad_step, c.aux.t + 1);
}

// tile rows per thread of the handle (Launch::rpt2d: 1, 2 or 4; 0 = default)
template <int S, bool TAU1>
cudaError_t launch_split2d(const Launch& c, int* nblocks) {
  if (c.rpt2d == 1) return launch_split2d_t<S, TAU1, 1>(c, nblocks);
  if (c.rpt2d == 4) return launch_split2d_t<S, TAU1, 4>(c, nblocks);
  return launch_split2d_t<S, TAU1, 2>(c, nblocks);
}

template <int S, class P>
cudaError_t launch(const Launch& c, int mode, int* nblocks) {
  if constexpr (std::is_same<P, PrecF32>::value) {
    if (mode == MODE_STEP && c.mu && !c.tiled && node2_rule(c.kp)) return launch_node2<S>(c, nblocks);
    if (mode == MODE_STEP && c.mu)
      return c.kp.omega == 1.0 ? launch_split2d<S, true>(c, nblocks) : launch_split2d<S, false>(c, nblocks);
  }
  if (mode == MODE_STEP_OBS) return cudaErrorNotSupported;
  if (mode == MODE_STEP) return launch_mode<S, P, MODE_STEP>(c, nblocks);
  if (mode == MODE_OBS) return launch_mode<S, P, MODE_OBS>(c, nblocks);
  return launch_mode<S, P, MODE_FIELDS>(c, nblocks);
}

template <int S>
StepFn pick(int prec) {
  if (prec == 0) return launch<S, PrecF64>;
  if (prec == 1) return launch<S, PrecF32>;
  return launch<S, PrecF32M64>;
}
}  // namespace

long long step2d_obs_ctas(const KParams& kp) {
  return (long long)((kp.nx + TX2 - 1) / TX2) * ((kp.ny + TY2 - 1) / TY2);
}

bool split2d_scheme(int scheme, int prec) {
  return prec == 1 && (scheme == S_EFDS2 || scheme == S_EFDS4 || scheme == S_EFDS6 || scheme == S_E4 || scheme == S_E8);
}

StepFn step2d_fn(int scheme, int prec) {
  switch (scheme) {
    case S_EFDS2: return pick<S_EFDS2>(prec);
    case S_EFDS4: return pick<S_EFDS4>(prec);
    case S_EFDS6: return pick<S_EFDS6>(prec);
    case S_E4: return pick<S_E4>(prec);
    case S_E8: return pick<S_E8>(prec);
    default: return nullptr;
  }
}

}  // namespace lbmd
