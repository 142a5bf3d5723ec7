// Launchers of the compact schemes' accelerations (iir.cuh).
#include <algorithm>
#include <cmath>

#include "compact.cuh"
#include "iir.cuh"

namespace lbmd {

namespace {

template <class T>
IirK<T> coef(int scheme) {
  double al, a, b, cc;
  compact_coeffs(scheme, &al, &a, &b, &cc);
  const double r = (1.0 - std::sqrt(1.0 - 4.0 * al * al)) / (2.0 * al), s = 1.0 + r * r;
  IirK<T> k{};
  k.nr = T(-r);
  k.a1 = T(0.5 * a * s);
  k.a2 = T(0.25 * b * s);
  k.a3 = T(cc / 6.0 * s);
  double p = 1.0;
  for (int j = 0; j <= IIR_M; ++j, p *= -r) k.p[j] = T(p);
  k.K = int(std::ceil((sizeof(T) == 4 ? 27 : 57) * std::log(2.0) / -std::log(r)));
  return k;
}

template <class T, int M, int LS>
cudaError_t col(const IirGeo& g, int axis, const T* rho, const T* mu, T* out, T rref, const IirK<T>& c, cudaStream_t st) {
  const int L = axis == 1 ? g.ny : g.nz, J = (c.K + (L >> LS) - 1) / (L >> LS);
  const dim3 grid((g.nx + 31) / 32, axis == 1 ? g.nz : g.ny);
  return launch_pdl(k_iir_col<T, M, LS>, grid, dim3(32, 1 << LS), 0, st, g, axis, rho, mu, out, rref, J, c);
}

template <class T, int M>
cudaError_t row(const IirGeo& g, const T* rho, const T* mu, T* out, T rref, const IirK<T>& c, cudaStream_t st) {
  const size_t smem = size_t(16) * (g.nx + g.nx / 32 + 1) * sizeof(T);
  if (cudaError_t e = ensure_smem(k_iir_row<T, M>, smem); e != cudaSuccess) return e;
  const int J = (c.K * 32 + g.nx - 1) / g.nx + 1;  // K nodes of nx / 32 each
  return launch_pdl(k_iir_row<T, M>, dim3((g.ny * g.nz + 7) / 8), dim3(256), smem, st, g, rho, mu, out, rref, J,
                    T(1.0 / (1.0 - std::pow(double(c.nr), g.nx))), c);
}

template <class T>
cudaError_t run(const IirGeo& g, int scheme, const T* rho, const T* mu, T* out, T rref, cudaStream_t st) {
  const IirK<T> c = coef<T>(scheme);
  const int mx = (g.nx + 31) / 32;
  cudaError_t e = mx <= 2 ? row<T, 2>(g, rho, mu, out, rref, c, st)
                : mx <= 4 ? row<T, 4>(g, rho, mu, out, rref, c, st)
                : mx <= 6 ? row<T, 6>(g, rho, mu, out, rref, c, st)
                : mx <= 8 ? row<T, 8>(g, rho, mu, out, rref, c, st)
                : mx <= 12 ? row<T, 12>(g, rho, mu, out, rref, c, st)
                           : row<T, 16>(g, rho, mu, out, rref, c, st);
  for (int axis = 1; axis < (g.nz > 1 ? 3 : 2) && e == cudaSuccess; ++axis) {
    // segments of eight nodes or more, sixteen of them on long lines
    const int L = axis == 1 ? g.ny : g.nz;
    e = L < 32 ? col<T, 8, 2>(g, axis, rho, mu, out, rref, c, st)
      : L < 64 ? col<T, 16, 2>(g, axis, rho, mu, out, rref, c, st)
      : L < 128 ? col<T, 16, 3>(g, axis, rho, mu, out, rref, c, st)
      : L <= 192 ? col<T, 12, 4>(g, axis, rho, mu, out, rref, c, st)
      : L <= 256 ? col<T, 16, 4>(g, axis, rho, mu, out, rref, c, st)
      : L <= 384 ? col<T, 24, 4>(g, axis, rho, mu, out, rref, c, st)
                 : col<T, 32, 4>(g, axis, rho, mu, out, rref, c, st);
  }
  return e;
}

}  // namespace

IirK<float> iir_coef(int scheme) { return coef<float>(scheme); }

// segments: at most 16 nodes on 32 lanes along x, 32 on 16 warps along y and z
bool iir_ok(const KParams& kp) { return kp.nx <= 512 && kp.ny <= 512 && kp.nz <= 512; }

cudaError_t iir_acc(const IirGeo& g, int scheme, const float* rho, const float* mu, float* out, float rref, cudaStream_t st) {
  return run<float>(g, scheme, rho, mu, out, rref, st);
}
cudaError_t iir_acc(const IirGeo& g, int scheme, const double* rho, const double* mu, double* out, double rref,
                    cudaStream_t st) {
  return run<double>(g, scheme, rho, mu, out, rref, st);
}

}  // namespace lbmd
