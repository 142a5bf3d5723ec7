"""The table-driven logarithm, the reciprocal and the equations of state of the FP64
kernels and the double-float chemical potential of mu_fp64, compiled for the host (the
same arithmetic: every operation rounded to nearest, no contraction but the fused ones
written out) and compared with 64-bit mantissas."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2205_09186_gb300", "csrc")
SHIM = r"""
#include <cmath>
#include <cstring>
struct double2 { double x, y; };
struct float4 { float x, y, z, w; };
#define __device__
#define __forceinline__ inline
static inline int __double2hiint(double x) { long long b; std::memcpy(&b, &x, 8); return int(b >> 32); }
static inline int __double2loint(double x) { long long b; std::memcpy(&b, &x, 8); return int(b); }
static inline double __hiloint2double(int h, int l) {
  const long long b = (long long)((unsigned long long)(unsigned)h << 32 | (unsigned)l);
  double x; std::memcpy(&x, &b, 8); return x;
}
static inline int __float_as_int(float x) { int b; std::memcpy(&b, &x, 4); return b; }
static inline float __int_as_float(int b) { float x; std::memcpy(&x, &b, 4); return x; }
static inline float __frcp_rn(float x) { return 1.f / x; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
using std::fma; using std::fmaf; using std::fabs; using std::log;
namespace lbmd {
struct KParams { int eos; double rho_ref, k2, kappa, RT, b4, two_a, c1, aa; };
}
#include "eos64.cuh"
using namespace lbmd;
extern "C" {
void t_log(const double* x, double* y, int n) { for (int i = 0; i < n; ++i) y[i] = log64(x[i]); }
void t_rcp(const double* x, double* y, int n) { for (int i = 0; i < n; ++i) y[i] = rcp64(x[i]); }
void t_mu(const KParams* p, const double* x, double* y, int n) { for (int i = 0; i < n; ++i) y[i] = eos_mu64(x[i], *p); }
void t_df(const KParams* p, const float* d, const float* lap, float* y, int* ok, int n) {
  const CsDf c = cs_df(*p);
  for (int i = 0; i < n; ++i) ok[i] = cs_mu_df(d[i], lap[i], c, y + i);
}
}
"""


class KParams(ctypes.Structure):
    _fields_ = [("eos", ctypes.c_int)] + [(n, ctypes.c_double) for n in
                                          ("rho_ref", "k2", "kappa", "RT", "b4", "two_a", "c1", "aa")]


@pytest.fixture(scope="module")
def H(tmp_path_factory):
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no long double of 64 bits")
    d = tmp_path_factory.mktemp("eos64")
    (d / "cuda_runtime.h").write_text("")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", str(d), "-I", CSRC,
                           str(d / "shim.cpp"), "-o", so])
    return ctypes.CDLL(so)


def call(fn, *a):
    x = np.ascontiguousarray(a[-1], np.float64)
    y = np.empty_like(x)
    args = list(a[:-1]) + [x.ctypes.data_as(ctypes.c_void_p), y.ctypes.data_as(ctypes.c_void_p), x.size]
    fn(*args)
    return y


def samples():
    rng = np.random.default_rng(0)
    edges = 1.0 + np.arange(513) / 512.0
    near = 1.0 + np.concatenate([s * 2.0 ** -np.arange(1, 53) for s in (1.0, -1.0)])
    return np.concatenate([np.exp(rng.uniform(-700, 700, 200000)), rng.uniform(0.5, 2.0, 400000),
                           1.0 + rng.uniform(-4e-3, 4e-3, 200000), near, edges, np.nextafter(edges, 0), edges / 2,
                           np.nextafter(edges / 2, 0), 2.0 ** np.arange(-1000, 1000)])


def test_logarithm_to_two_ulp_everywhere(H):
    # a table entry and its sum with the rest, a rounding each, and ln 2's own: 1.5 ulp
    x = samples()
    y = call(H.t_log, x)
    want = np.log(x.astype(np.longdouble))
    err = np.abs(y.astype(np.longdouble) - want)
    assert np.all(err <= 2.0 * np.spacing(np.abs(want.astype(np.float64)))), float(np.max(err))
    odd = np.array([0.0, -1.0, np.inf, np.nan, 5e-324, 1e-310])
    with np.errstate(all="ignore"):
        assert np.array_equal(call(H.t_log, odd), np.log(odd), equal_nan=True)


def test_reciprocal_to_one_ulp(H):
    rng = np.random.default_rng(1)
    x = np.concatenate([samples(), -np.exp(rng.uniform(-60, 60, 10000)), [1e-300, 1e300, 5e-324]])
    with np.errstate(all="ignore"):
        want = 1.0 / x.astype(np.longdouble)
        fin = np.abs(want) < np.finfo(np.float64).max
        y = call(H.t_rcp, x)
        assert np.all(np.abs(y[fin].astype(np.longdouble) - want[fin]) <= np.spacing(np.abs(want[fin].astype(np.float64))))
        odd = np.array([0.0, -0.0, np.inf, -np.inf, np.nan])
        assert np.array_equal(call(H.t_rcp, odd), 1.0 / odd, equal_nan=True)


# the chemical potential against its terms: RT (ln + repulsion) - attraction, each
# rounded a few times.  b = 1e-9 leaves the logarithm alone, through rho = 1, where it
# vanishes; b = 4 is the usual fluid
@pytest.mark.parametrize("eos", [0, 1, 2, 3])
@pytest.mark.parametrize("b", [4.0, 2.0 / 21.0, 1e-9])
def test_chemical_potential_to_a_few_roundings_of_its_terms(H, eos, b):
    rng = np.random.default_rng(2)
    top = (1.0 if eos else 4.0) / b
    rho = np.concatenate([top * np.exp(rng.uniform(-25, -0.01, 100000)), top * rng.uniform(0.01, 0.9, 100000)])
    if b < 1e-6:
        rho = np.concatenate([rho, rng.uniform(0.5, 2.0, 200000), 1.0 + rng.uniform(-1e-6, 1e-6, 100000)])
    RT, a = 0.3 * b, 0.5 * b * b if b < 1e-6 else 0.8 * b
    p = KParams(eos, 0.0, 1.0, 0.0, RT, 0.25 * b, 2.0 * a, 0.1 * RT, 0.2 * a)
    y = call(H.t_mu, ctypes.byref(p), rho)
    lr, x = rho.astype(np.longdouble), np.longdouble(p.b4) * rho
    if eos == 0:
        hs = x * (8 - 9 * x + 3 * x * x) / (1 - x) ** 3
        terms = [RT * np.log(lr), RT * hs, -np.longdouble(p.two_a) * lr]
        amp = 1 / (1 - x)  # of the rounding of 1 - eta
    else:
        x = 4 * x
        io = 1 / (1 - x)
        terms = [RT * np.log(lr * io), RT * io]
        if eos == 2:
            terms.append(-np.longdouble(p.two_a) * lr)
        elif eos == 3:
            terms += [-np.longdouble(p.c1) * np.log(1 + x), -np.longdouble(p.aa) * lr / (1 + x)]
        else:
            s2 = np.sqrt(np.longdouble(2))
            terms += [-np.longdouble(p.c1) * np.log((s2 - 1 + x) / (s2 + 1 - x)),
                      -np.longdouble(p.aa) * lr / (1 + x * (2 - x))]
        amp = io
    scale = sum(np.abs(t) for t in terms)
    if eos:  # the logarithms' arguments are rounded before they are taken
        scale = scale + RT + p.c1
    err = np.abs(y.astype(np.longdouble) - sum(terms))
    assert np.all(err <= 8 * 2.0 ** -53 * scale * amp), float(np.max(err / (scale * amp)) * 2.0 ** 53)


# double-float: the float that FP64 gives, but where the value lies next to the middle
# between two floats.  The terms carry 2^-45 each and their sum may cancel; rho_ref
# carries 2^-48, which a density far below it has magnified in its logarithm
@pytest.mark.parametrize("Tr,rho_ref", [(0.3, 1e-5), (0.6, 2e-3), (0.9, 0.05)])  # about the gas densities
def test_double_float_chemical_potential_rounds_as_fp64(H, Tr, rho_ref):
    rng = np.random.default_rng(3)
    b, a, k2, kappa = 4.0, 1.0, 0.0625, 0.1
    RT = Tr * 0.094328  # R T_c of a = 1, b = 4
    p = KParams(0, rho_ref, k2, kappa, RT, 0.25 * b, 2.0 * a, 0.0, 0.0)
    n = 400000
    rho = np.concatenate([np.exp(rng.uniform(np.log(0.1 * rho_ref), np.log(0.9), n)), rng.uniform(0.001, 0.9, n)])
    d = (rho - rho_ref).astype(np.float32)
    lap = (rng.standard_normal(2 * n) * 1e-2).astype(np.float32)
    y, ok = np.empty(2 * n, np.float32), np.empty(2 * n, np.int32)
    H.t_df(ctypes.byref(p), *(v.ctypes.data_as(ctypes.c_void_p) for v in (d, lap, y, ok)), 2 * n)
    r = np.longdouble(rho_ref) + d.astype(np.longdouble)
    use = ok != 0
    assert np.array_equal(use, use & (r > 0)) and np.count_nonzero(use) == np.count_nonzero(r > 0)
    e = np.longdouble(p.b4) * r[use]
    terms = [np.longdouble(k2) * RT * np.log(r[use]), np.longdouble(k2) * RT * e * (8 - 9 * e + 3 * e * e) / (1 - e) ** 3,
             -np.longdouble(k2) * p.two_a * r[use], -np.longdouble(kappa) * lap[use]]
    want, scale = sum(terms), sum(np.abs(t) for t in terms)
    err = np.abs(y[use].astype(np.longdouble) - want)
    scale += k2 * RT * (rho_ref / r[use]) / 8
    assert np.all(err <= 0.5 * np.spacing(np.abs(want.astype(np.float32))) + 2.0 ** -44 * scale)
    assert np.count_nonzero(y[use] != want.astype(np.float32)) < 1e-5 * np.count_nonzero(use)
