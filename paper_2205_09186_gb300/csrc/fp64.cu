// Launchers of the FP64 step (fp64.cuh).
#include "fp64.cuh"
#include "launch.cuh"

namespace lbmd {

namespace {

// nodes per block: 128, fewer where that would leave SMs without a block
int block64(const KParams& kp) {
  const long long sms = device_sms();
  return kp.n >= 4 * 128 * sms ? 128 : (kp.n >= 4 * 64 * sms ? 64 : 32);
}

template <int S, int LAT>
cudaError_t step(const Launch& c, double* mu) {
  const KParams& kp = c.kp;
  const int bs = block64(kp), g = int((kp.n + bs - 1) / bs);
  const double *fin = static_cast<const double*>(c.fin), *rin = static_cast<const double*>(c.rin);
  double *fout = static_cast<double*>(c.fout), *rout = static_cast<double*>(c.rout);
  if constexpr (LAT == 0 && !Sch<S>::GF) {
    const dim3 t((kp.nx + T64X - 1) / T64X, (kp.ny + T64Y - 1) / T64Y);
    if ((long long)t.x * t.y <= device_sms()) {
      auto k = c.mrt.on ? k64_tile<S, 2> : (kp.omega == 1.0 ? k64_tile<S, 0> : k64_tile<S, 1>);
      return launch_pdl(k, t, T64N, 0, c.stream, kp, fin, fout, rin, rout, c.aux, c.mrt);
    }
  }
  cudaError_t e = cudaSuccess;
  if constexpr (!Sch<S>::GF) e = launch_pdl(k64_mu<S, LAT>, g, bs, 0, c.stream, kp, rin, mu);
  if (e != cudaSuccess) return e;
  auto k = kp.omega == 1.0 ? k64_coll<S, LAT, 0> : k64_coll<S, LAT, 1>;
  if constexpr (LAT == 0) {
    if (c.mrt.on) k = k64_coll<S, LAT, 2>;
  }
  e = launch_pdl(k, g, bs, 0, c.stream, kp, fin, fout, rin, mu, c.gi, c.aux, c.mrt);
  if (e != cudaSuccess) return e;
  return launch_pdl(k64_rho<Lattice<LAT>::Q>, g, bs, 0, c.stream, kp, fout, rout, c.aux.bad_step, c.aux.t + 1);
}

}  // namespace

cudaError_t step64(const Launch& c, int D, int scheme, double* mu) {
  const bool two = D == 2;
  switch (scheme) {
    case S_EFDS2: return two ? step<S_EFDS2, 0>(c, mu) : step<S_EFDS2, 1>(c, mu);
    case S_EFDS4: return two ? step<S_EFDS4, 0>(c, mu) : step<S_EFDS4, 1>(c, mu);
    case S_EFDS6: return two ? step<S_EFDS6, 0>(c, mu) : step<S_EFDS6, 1>(c, mu);
    case S_E4: return two ? step<S_E4, 0>(c, mu) : step<S_E4, 1>(c, mu);
    case S_E8: return two ? step<S_E8, 0>(c, mu) : cudaErrorNotSupported;
    case S_CFDS4:
    case S_CFDS6:
    case S_CFDS8:
    case S_OCFDS4: return two ? step<S_CFDS4, 0>(c, mu) : step<S_CFDS4, 1>(c, mu);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace lbmd
