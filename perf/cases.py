"""The work a user of this library has it do, as cases that can be timed.

A case is one call pattern of the public binding (paper_2205_09186_gb300.lbm):
a simulation advanced by the steps between two looks at it, a batch of droplets
advanced and read back, an observed run from a host density to a host density,
or warm-start training.  `exact` restates each in 64-bit torch, from the
equations, without the library.
"""
import ctypes
import math
import random

import numpy as np
import torch

from paper_2205_09186_gb300 import lbm as L

MLP_SIZES = [4, 128, 128, 128, 64]  # the warm-start network
WALL_ROWS = 8                       # rows (planes) of the flat wall


def _sim(name, lattice, nx, ny, nz, scheme, steps, precision="fp32", mu64=0, tau=1.0, collision="BGK", eos="CS",
         Tr=0.8, k=0.25, kind="steps"):
    return {"name": name, "kind": kind, "lattice": lattice, "nx": nx, "ny": ny, "nz": nz, "scheme": scheme,
            "steps": steps, "precision": precision, "mu64": mu64, "tau": tau, "collision": collision, "eos": eos,
            "Tr": Tr, "k": k}


def listed():
    return [
        # the smallest configuration: a 64^2 droplet in full FP64, relaxed
        # between two looks at max |d rho / dt| (launch and latency bound)
        _sim("d2q9_64_fp64", "D2Q9", 64, 64, 1, "EFDS2", 200, "fp64", Tr=0.85),
        # the scheme sweep's lattice, one droplet by itself
        _sim("d2q9_512", "D2Q9", 512, 512, 1, "EFDS6", 200),
        # a 2D lattice that exceeds the caches
        _sim("d2q9_4096", "D2Q9", 4096, 4096, 1, "EFDS6", 20),
        # wetting: a droplet on a flat wall, multiple-relaxation-time collision
        _sim("d2q9_512_wall_mrt", "D2Q9", 512, 512, 1, "EFDS4", 50, tau=0.8, collision="MRT", kind="walls"),
        # the parameter sweep: droplets of uneven sizes and schemes in one batch
        {"name": "batch_48", "kind": "batch", "cases": 48, "smallest": 64, "largest": 512, "steps": 100,
         "precision": "fp32"},
        # the headline droplet
        _sim("d3q19_256", "D3Q19", 256, 256, 256, "EFDS6", 50),
        # the same lattice colder, with the chemical potential in FP64
        _sim("d3q19_256_mu64", "D3Q19", 256, 256, 256, "EFDS6", 20, mu64=1, Tr=0.5),
        # the same lattice with the observables of every step read back, from
        # a pinned host density to a pinned host density
        _sim("d3q19_256_observed", "D3Q19", 256, 256, 256, "EFDS6", 20, kind="observed"),
        # the warm-start study's lattice with the optimal compact scheme
        _sim("d3q19_192_ocfds4", "D3Q19", 192, 192, 192, "OCFDS4", 20),
        # odd sizes, tau away from 1 and the paper's Peng-Robinson fluid
        _sim("d3q19_125x70x43_pr", "D3Q19", 125, 70, 43, "EFDS4", 50, tau=0.8, eos="PR", Tr=0.8, k=0.2),
        # the plain FP64 relaxation the warm start is judged against
        _sim("d3q19_80_fp64", "D3Q19", 80, 80, 80, "EFDS6", 20, "fp64"),
        # the warm-start network's training on 31 relaxed droplets
        {"name": "mlp_train_31", "kind": "mlp", "samples": 31, "iters": 50},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["d2", "d2", "d3", "d3", "d3", "compact", "fp64", "walls", "batch", "observed", "mlp"])
    if kind == "mlp":
        return {"kind": "mlp", "samples": _log(rng, 8, 128), "iters": rng.randint(10, 50)}
    if kind == "batch":
        return {"kind": "batch", "cases": rng.randint(8, 48), "smallest": 64, "largest": rng.randint(128, 512),
                "steps": rng.randint(20, 100), "precision": "fp32"}
    # tau 1 is what every configuration of the method's study runs; other
    # relaxation times and MRT are the options beside it
    tau = rng.choice([1.0, 1.0, 1.0, 0.8, 0.9])
    explicit, compact = ["EFDS4", "EFDS6", "EFDS6"], ["CFDS4", "CFDS6", "CFDS8", "OCFDS4", "OCFDS4"]
    eos = "PR" if rng.random() < 0.15 else "CS"
    phys = dict(tau=tau, eos=eos, Tr=round(rng.uniform(0.75, 0.9), 3) if eos == "PR" else round(rng.uniform(0.5, 0.9), 3),
                k=0.2 if eos == "PR" else round(rng.uniform(0.15, 0.35), 3))
    scheme = rng.choice(explicit)
    if kind == "d2":
        if rng.random() < 0.25 and eos == "CS":
            scheme, phys["Tr"] = rng.choice(["EFDS2", "E4", "E8"]), round(rng.uniform(0.86, 0.93), 3)
        nx, ny = _log(rng, 64, 4096), _log(rng, 64, 4096)
        if rng.random() < 0.5:
            nx -= nx % 4
        steps = min(200, max(10, int(1e9 / (nx * ny))))
        c = _sim("", "D2Q9", nx, ny, 1, scheme, steps, collision=rng.choice(["BGK", "BGK", "BGK", "MRT"]), **phys)
    elif kind == "walls":
        nx, ny = _log(rng, 64, 768), _log(rng, 64, 768)
        c = _sim("", "D2Q9", nx, ny, 1, scheme, rng.randint(20, 60), collision=rng.choice(["BGK", "MRT"]), kind="walls",
                 **phys)
    elif kind == "fp64":
        d3 = rng.random() < 0.5
        n = [_log(rng, 32, 96) for _ in range(3)] if d3 else [_log(rng, 64, 512), _log(rng, 64, 512), 1]
        steps = min(200, max(4, int((4e6 if d3 else 1.5e7) / (n[0] * n[1] * n[2]))))
        c = _sim("", "D3Q19" if d3 else "D2Q9", *n, rng.choice(explicit + ["OCFDS4"]), steps, "fp64", **phys)
    else:
        n = [_log(rng, 32, 256) for _ in range(3)]
        if rng.random() < 0.6:
            n[0] -= n[0] % 4
        steps = min(50, max(10, int(3e8 / (n[0] * n[1] * n[2]))))
        if kind == "observed":
            c = _sim("", "D3Q19", *n, scheme, min(steps, 20), kind="observed", **phys)
        elif kind == "compact":
            c = _sim("", "D3Q19", *n, rng.choice(compact), min(steps, 20), **phys)
        else:
            c = _sim("", "D3Q19", *n, scheme, steps, mu64=int(rng.random() < 0.2), **phys)
            if c["mu64"]:
                c["steps"] = min(c["steps"], 20)
    del c["name"]
    return c


# ------------------------------------------------------------------ physics of a case
def _phys(case):
    """Constants of the equation of state and kappa-hat (the paper's water for
    Peng-Robinson, with the kappa-hat its densities allow)."""
    if case.get("eos", "CS") == "PR":
        return dict(eos="PR", a=2.0 / 49.0, b=2.0 / 21.0, R=1.0, acentric=0.344, kappa=0.01)
    return dict(eos="CS", a=1.0, b=4.0, R=1.0, acentric=0.344, kappa=0.1)


def _params(case, rho_ref=0.0):
    return L.make_params(lattice=L.LBM_D2Q9 if case["lattice"] == "D2Q9" else L.LBM_D3Q19, nx=case["nx"], ny=case["ny"],
                         nz=case["nz"], Tr=case["Tr"], k=case["k"], tau=case["tau"], scheme=case["scheme"],
                         precision=L.LBM_FP64 if case["precision"] == "fp64" else L.LBM_FP32DEV, mu_fp64=case["mu64"],
                         collision=case["collision"], rho_ref=rho_ref, **_phys(case))


def _droplet(case, seed):
    """Centre (x, y, z) and radius of a seed's droplet."""
    r = random.Random(seed)
    n = [case["nx"], case["ny"]] + ([case["nz"]] if case["lattice"] == "D3Q19" else [])
    R = min(n) / 4.0 * r.uniform(0.85, 1.0)
    c = [m / 2.0 + r.uniform(-2.0, 2.0) for m in n] + [0.0] * (3 - len(n))
    if case["kind"] == "walls":
        c[1] = WALL_ROWS + 0.8 * R
    return c, R


def _wall(case):
    m = np.zeros((case["ny"], case["nx"]), np.uint8)
    m[:WALL_ROWS] = 1
    return m


def _batch(case, seed):
    """Droplets of a sweep: size, radius, T_r, k and scheme; the schemes that
    go unstable on cold droplets are run on warm ones.  The lattices are the
    sweep's; the droplets on them come from the seed."""
    size, r = random.Random(case["cases"] * 1000 + case["largest"]), random.Random(seed)
    out = []
    for j in range(case["cases"]):
        scheme = ["EFDS2", "EFDS4", "EFDS6", "E4", "E8", "OCFDS4"][j % 6]
        nx, ny = (size.randint(case["smallest"], case["largest"]) for _ in range(2))
        warm = scheme in ("EFDS2", "E4", "E8")
        out.append(dict(lattice="D2Q9", nx=nx, ny=ny, nz=1, scheme=scheme, precision=case["precision"], mu64=0, tau=1.0,
                        collision="BGK", eos="CS", kind="steps", Tr=r.uniform(0.86, 0.93) if warm else r.uniform(0.5, 0.93),
                        k=math.exp(r.uniform(math.log(0.15), math.log(0.4))), radius=r.uniform(12.0, min(nx, ny) / 4.0)))
    return out


def _training(case, seed):
    """Normalised droplet profiles as the solver relaxes them (tanh-like) and
    their parameters, and initial weights."""
    rng = np.random.default_rng(seed)
    m = case["samples"]
    Tr, k, R = rng.uniform(0.6, 0.85, m), np.exp(rng.uniform(np.log(0.2), np.log(0.35), m)), rng.uniform(14, 34, m)
    x = np.stack([Tr, np.log(k), R / 64.0, np.full(m, 2 / 8.0)], 1)
    r = np.maximum(0.0, R - 16.0)[:, None] + 0.5 * np.arange(64)[None]
    t = 0.5 - 0.5 * np.tanh((r - R[:, None]) * k[:, None] * (1.2 - Tr[:, None]) * 2.0)
    p = []
    for i, o in zip(MLP_SIZES[:-1], MLP_SIZES[1:]):
        p += [rng.standard_normal(o * i) * math.sqrt(2.0 / i), np.zeros(o)]
    return x.astype(np.float32), t.astype(np.float32), np.concatenate(p).astype(np.float32)


# ------------------------------------------------------------------ the calls
class _OnDevice:
    """A handle's device array as torch sees it (the handle lives as long)."""

    def __init__(self, sim, ptr, shape, kind):
        self.sim = sim
        self.__cuda_array_interface__ = {"shape": shape, "typestr": kind, "data": (ptr, False), "version": 2}


def _state(sim, case):
    f, rho = sim.lbm_device_state()
    kind = "<f8" if case["precision"] == "fp64" else "<f4"
    return {"f": torch.as_tensor(_OnDevice(sim, f, (sim.Q,) + sim.shape, kind), device="cuda"),
            "rho": torch.as_tensor(_OnDevice(sim, rho, sim.shape, kind), device="cuda")}


OBS = ("max_v", "max_u", "rho_center", "rho_corner")


def prepare(case, seed):
    if case["kind"] == "mlp":
        x, t, p = _training(case, seed)
        net = L.MLP(MLP_SIZES, max(case["samples"], 32))
        net.lbm_mlp_set_params(p)
        net.lbm_mlp_set_data(x, t)
        return case, net
    if case["kind"] == "batch":
        cs = _batch(case, seed)
        b = L.Batch([_params(dict(c)) for c in cs])
        b.lbm_batch_init_droplets([c["radius"] for c in cs])
        return case, b
    sim = L.Sim(_params(case))
    c, R = _droplet(case, seed)
    sim.lbm_init_droplet(R, center=c)
    if case["kind"] == "walls":
        p = sim.params
        sim.lbm_set_solid(_wall(case), L.lbm_bulk_mu(p, L.lbm_maxwell(p)[0]) - 0.005 * _phys(case)["kappa"] / 0.1)
    if case["kind"] == "observed":
        rho0 = torch.empty(sim.shape, dtype=torch.float64, pin_memory=True).numpy()
        sim.lbm_get_density(out=rho0)
        rec = torch.zeros(ctypes.sizeof(L.lbm_obs) * case["steps"], dtype=torch.uint8, pin_memory=True)
        return case, sim, rho0, torch.empty(sim.shape, dtype=torch.float64, pin_memory=True).numpy(), rec
    return case, sim


def run(state):
    case, sim = state[:2]
    if case["kind"] == "mlp":
        loss = sim.lbm_mlp_train(case["iters"], 1e-3)
        return {"params": sim.lbm_mlp_get_params(), "loss": loss}
    if case["kind"] == "batch":
        sim.lbm_batch_step(case["steps"])
        _, obs = sim.lbm_batch_observables()
        out = {"obs": np.array([[o[k] for k in OBS] for o in obs], np.float32),
               "mass": np.array([o["mass"] for o in obs], np.float32)}
        for c in range(sim.n):
            out["rho%02d" % c] = sim.lbm_batch_get_density(c).astype(np.float32)
        return out
    if case["kind"] == "observed":
        _, _, rho0, rho1, rec = state
        sim.lbm_init_density(rho0)
        for s in range(case["steps"]):
            sim.lbm_step_observe_async(1, rec.data_ptr() + s * ctypes.sizeof(L.lbm_obs))
        sim.lbm_get_density(out=rho1)
        r = np.frombuffer((L.lbm_obs * case["steps"]).from_address(rec.data_ptr()), dtype=np.dtype(L.lbm_obs))
        return dict(_state(sim, case), obs=np.stack([r[k] for k in OBS + ("max_drho",)], 1).astype(np.float32),
                    mass=r["mass"].astype(np.float32))
    sim.lbm_step(case["steps"])
    out = _state(sim, case)
    if case["kind"] == "walls":  # the populations and densities of wall nodes are not defined
        return {"f": out["f"][:, WALL_ROWS:], "rho": out["rho"][WALL_ROWS:]}
    return out


def work(case):
    if case["kind"] == "mlp":
        par = sum((i + 1) * o for i, o in zip(MLP_SIZES[:-1], MLP_SIZES[1:]))
        return {"bytes": 4 * (6 * par + 68 * case["samples"]), "flops": 6 * par * case["samples"] * case["iters"]}
    if case["kind"] == "batch":
        # FP32 populations and densities in and out, the densities once more in FP64
        n = sum(c["nx"] * c["ny"] for c in _batch(case, 0))
        return {"bytes": n * (2 * 10 * 4 + 8), "flops": n * case["steps"] * 200}
    q, size = (9 if case["lattice"] == "D2Q9" else 19), (8 if case["precision"] == "fp64" else 4)
    n = case["nx"] * case["ny"] * case["nz"]
    # the state once in and once out of the call; about 12 operations per
    # population and 60 for the chemical potential and the force of each step
    b = n * 2 * (q + 1) * size
    if case["kind"] == "observed":
        b = n * (2 * 8 + (q + 1) * size)
    return {"bytes": b, "flops": n * case["steps"] * (12 * q + 60)}


# ------------------------------------------------------------------ 64-bit restatement
def _mu_bulk(case, rho, T, log):
    """psi'(rho), additive constant dropped (Eq. 10, 13-15)."""
    p = _phys(case)
    RT = p["R"] * T
    if p["eos"] == "PR":
        kap = 0.37464 + p["acentric"] * (1.54226 - 0.26992 * p["acentric"])
        aa = p["a"] * (1.0 + kap * (1.0 - math.sqrt(case["Tr"]))) ** 2
        x, s2 = p["b"] * rho, math.sqrt(2.0)
        return (RT * (log(rho / (1 - x)) + 1 / (1 - x)) - aa / (2 * s2 * p["b"]) * log((s2 - 1 + x) / (s2 + 1 - x))
                - aa * rho / (1 + 2 * x - x * x))
    e = 0.25 * p["b"] * rho
    return RT * (log(rho) + e * (8 + e * (-9 + 3 * e)) / (1 - e) ** 3) - 2 * p["a"] * rho


def _pressure(case, rho, T):
    p = _phys(case)
    if p["eos"] == "PR":
        kap = 0.37464 + p["acentric"] * (1.54226 - 0.26992 * p["acentric"])
        aa = p["a"] * (1.0 + kap * (1.0 - math.sqrt(case["Tr"]))) ** 2
        x = p["b"] * rho
        return rho * p["R"] * T / (1 - x) - aa * rho * rho / (1 + 2 * x - x * x)
    e = 0.25 * p["b"] * rho
    return rho * p["R"] * T * (1 + e + e * e - e ** 3) / (1 - e) ** 3 - p["a"] * rho * rho


def _bisect(f, lo, hi):
    up = f(hi) > 0
    for _ in range(200):
        m = 0.5 * (lo + hi)
        if (f(m) > 0) == up:
            hi = m
        else:
            lo = m
    return 0.5 * (lo + hi)


def _temperature(case):
    """T = T_r T_c with p0' = p0'' = 0 at the critical point."""
    p = _phys(case)
    if p["eos"] == "PR":
        # h(x) = x^2 / D, D = 1 + 2x - x^2: 2 h' = (1 - x) h'', R T_c = (a / b)(1 - x)^2 h'
        D = lambda x: 1 + 2 * x - x * x  # noqa: E731
        h1 = lambda x: 2 * x * (1 + x) / D(x) ** 2  # noqa: E731
        h2 = lambda x: (2 * (1 + 2 * x) * D(x) - 8 * x * (1 + x) * (1 - x)) / D(x) ** 3  # noqa: E731
        x = _bisect(lambda x: 2 * h1(x) - (1 - x) * h2(x), 1e-6, 0.9)
        return case["Tr"] * p["a"] / p["b"] * (1 - x) ** 2 * h1(x) / p["R"]
    num = lambda e: 1 + 4 * e + 4 * e ** 2 - 4 * e ** 3 + e ** 4  # noqa: E731
    c1 = lambda e: num(e) / (1 - e) ** 4  # noqa: E731
    d1 = lambda e: (4 + 8 * e - 12 * e ** 2 + 4 * e ** 3) / (1 - e) ** 4 + 4 * num(e) / (1 - e) ** 5  # noqa: E731
    e = _bisect(lambda e: e * d1(e) - c1(e), 1e-6, 0.5)
    return case["Tr"] * 8 * p["a"] / (p["b"] * p["R"] * d1(e))


def _maxwell(case):
    """Gas and liquid densities of equal pressure and chemical potential."""
    p, T = _phys(case), _temperature(case)
    top = (1.0 if p["eos"] == "PR" else 4.0) / p["b"]
    dp = lambda r: (_pressure(case, r * (1 + 1e-6), T) - _pressure(case, r * (1 - 1e-6), T))  # noqa: E731
    grid = np.exp(np.linspace(math.log(top * 1e-9), math.log(top * 0.999), 40001))
    neg = np.nonzero(dp(grid) < 0)[0]
    sg, sl = grid[neg[0] - 1], grid[neg[-1] + 1]
    mu = lambda r: _mu_bulk(case, r, T, math.log)  # noqa: E731
    gas = lambda m: math.exp(_bisect(lambda s: mu(math.exp(s)) - m, math.log(top) - 60.0, math.log(sg)))  # noqa: E731
    liq = lambda m: _bisect(lambda r: mu(r) - m, sl, top * (1 - 1e-12))  # noqa: E731
    m = _bisect(lambda m: _pressure(case, gas(m), T) - _pressure(case, liq(m), T), mu(sl), mu(sg))
    return gas(m), liq(m)


_E = {"D2Q9": [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)],
      "D3Q19": [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
                (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
                (0, -1, 1)]}
_W = {"D2Q9": [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, "D3Q19": [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12}
_FIRST = {2: [1 / 2], 4: [2 / 3, -1 / 12], 6: [3 / 4, -3 / 20, 1 / 60]}
_SECOND = {2: [-2.0, 1.0], 4: [-5 / 2, 4 / 3, -1 / 12], 6: [-49 / 18, 3 / 2, -3 / 20, 1 / 90],
           8: [-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560]}
_ORDER = {"EFDS2": 2, "EFDS4": 4, "EFDS6": 6, "CFDS4": 4, "CFDS6": 6, "CFDS8": 8, "OCFDS4": 4}
# alpha f'_{i-1} + f'_i + alpha f'_{i+1} = a (f_{i+1} - f_{i-1}) / 2 + b (f_{i+2} - f_{i-2}) / 4 + c (f_{i+3} - f_{i-3}) / 6
_OA, _OC = 0.446776, -0.0541132
_OB = (6 * _OA - (1 + 2 * _OA) - 8 * _OC) / 3
_COMPACT = {"CFDS4": (1 / 4, 3 / 2, 0.0, 0.0), "CFDS6": (1 / 3, 14 / 9, 1 / 9, 0.0), "CFDS8": (3 / 8, 25 / 16, 1 / 5, -1 / 80),
            "OCFDS4": (_OA, 1 + 2 * _OA - _OB - _OC, _OB, _OC)}
_ISO = {"E4": {2: {1: 1 / 3, 2: 1 / 12}, 3: {1: 1 / 6, 2: 1 / 12}},
        "E8": {2: {1: 4 / 21, 2: 4 / 45, 4: 1 / 60, 5: 2 / 315, 8: 1 / 5040}}}
_M9 = [[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1], [0, 1, 0, -1, 0, 1, -1, -1, 1],
       [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
       [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]]


class _Exact:
    """The time step of Sec. 2.1-2.2 in 64-bit torch.  Fields are (z,) y, x."""

    def __init__(self, case):
        self.c, self.e, self.w = case, _E[case["lattice"]], _W[case["lattice"]]
        self.D = 2 if case["lattice"] == "D2Q9" else 3
        self.T, self.kappa = _temperature(case), _phys(case)["kappa"]
        self.shape = (case["nz"], case["ny"], case["nx"])[3 - self.D:]
        self.solid = None
        if case["scheme"] in _COMPACT:
            al, a, b, c = _COMPACT[case["scheme"]]
            self.der = []
            for ax in range(self.D):
                n = self.shape[self.D - 1 - ax]
                lhs, rhs = np.eye(n), np.zeros((n, n))
                i = np.arange(n)
                for s in (1, -1):
                    lhs[i, (i + s) % n] += al
                    for m, q in ((1, a / 2), (2, b / 4), (3, c / 6)):
                        rhs[i, (i + s * m) % n] += s * q
                self.der.append(torch.from_numpy(np.linalg.solve(lhs, rhs)).cuda())

    def at(self, q, e):  # q(x + e)
        return torch.roll(q, [-e[a] for a in range(self.D)], [self.D - 1 - a for a in range(self.D)])

    def along(self, q, ax, m):
        return torch.roll(q, -m, self.D - 1 - ax)

    def grad(self, q, ax):
        s = self.c["scheme"]
        if s in _COMPACT:
            d = self.D - 1 - ax
            return torch.movedim(torch.movedim(q, d, -1) @ self.der[ax].T, -1, d)
        if s in _ISO:
            r = torch.zeros_like(q)
            for o, w in self.offsets():
                if o[ax]:
                    r += w * o[ax] * self.at(q, o)
            return r
        return sum(g * (self.along(q, ax, m + 1) - self.along(q, ax, -m - 1)) for m, g in enumerate(_FIRST[_ORDER[s]]))

    def offsets(self):
        w = _ISO[self.c["scheme"]][self.D]
        k = range(-2, 3)
        return [((x, y, z), w[x * x + y * y + z * z]) for x in k for y in k for z in (k if self.D == 3 else (0,))
                if x * x + y * y + z * z in w]

    def lap(self, q):
        if self.c["scheme"] in _ISO:
            return sum(2 * w * (self.at(q, o) - q) for o, w in self.offsets())
        l = _SECOND[_ORDER[self.c["scheme"]]]
        return sum(l[0] * q + sum(l[m] * (self.along(q, ax, m) + self.along(q, ax, -m)) for m in range(1, len(l)))
                   for ax in range(self.D))

    def start(self, center, R, width=10.0):
        g, l = _maxwell(self.c)
        self.g = g
        d2 = 0.0
        for ax in range(self.D):
            n = self.shape[self.D - 1 - ax]
            x = torch.arange(n, dtype=torch.float64, device="cuda") - center[ax]
            d2 = d2 + (x * x).reshape([-1 if self.D - 1 - ax == d else 1 for d in range(self.D)])
        rho = 0.5 * (l + g) - 0.5 * (l - g) * torch.tanh(2.0 * (torch.sqrt(d2) - R) / width)
        self.f = [w * rho for w in self.w]
        self.snap = sum(self.f)

    def walls(self, mask, mu_w):
        self.solid, self.mu_w = torch.from_numpy(mask != 0).cuda(), mu_w
        self.layers, done = [], ~self.solid
        for _ in range(3):
            new = torch.zeros_like(done)
            for e in self.e[1:]:
                new |= self.at(done, e)
            new &= ~done
            self.layers.append((new, done.clone() if not self.layers else self.layers[-1][0]))
            done = done | new

    def fields(self):
        rho = sum(self.f)
        j = [sum(e[a] * f for e, f in zip(self.e, self.f) if e[a]) for a in range(self.D)]
        if self.solid is not None:  # Eq. A.1, layer after layer
            rho = torch.where(self.solid, torch.full_like(rho, self.g), rho)
            for here, before in self.layers:
                num = sum(w * self.at(rho * before, e) for w, e in zip(self.w[1:], self.e[1:]))
                den = sum(w * self.at(before.double(), e) for w, e in zip(self.w[1:], self.e[1:]))
                rho = torch.where(here, num / torch.where(here, den, torch.ones_like(den)), rho)
        mu = self.c["k"] ** 2 * _mu_bulk(self.c, rho, self.T, torch.log) - self.kappa * self.lap(rho)
        if self.solid is not None:
            mu = torch.where(self.solid, torch.full_like(mu, self.mu_w), mu)
        F = [-rho * self.grad(mu, a) + self.grad(rho, a) / 3.0 for a in range(self.D)]
        return rho, [q / rho for q in j], F

    def observe(self, dt):
        rho, u, F = self.fields()
        v = [a + 0.5 * b / rho for a, b in zip(u, F)]
        o = [math.sqrt(float(sum(a * a for a in v).max())), math.sqrt(float(sum(a * a for a in u).max())),
             float(rho[tuple(n // 2 for n in self.shape)]), float(rho[(0,) * self.D]),
             float((rho - self.snap).abs().max()) / dt if dt else 0.0]
        self.snap = rho
        return o, float(rho.sum())

    def step(self):
        rho, u, F = self.fields()
        v = [a + b / rho for a, b in zip(u, F)]
        feq = lambda i, q, qq: (lambda eq: self.w[i] * rho * (1 + eq * (3 + 4.5 * eq) - 1.5 * qq))(  # noqa: E731
            sum(e * x for e, x in zip(self.e[i], q)))
        uu, vv = sum(a * a for a in u), sum(a * a for a in v)
        om = 1.0 / self.c["tau"]
        if self.c["collision"] == "MRT":
            M = torch.tensor(_M9, dtype=torch.float64)
            S = torch.diag(torch.tensor([1, 1.64, 1.54, 1, 1.7, 1, 1.7, om, om], dtype=torch.float64))
            K = (torch.linalg.inv(M) @ S @ M).cuda()
            ne = torch.stack([f - feq(i, u, uu) for i, f in enumerate(self.f)])
            ne = torch.einsum("ij,j...->i...", K, ne)
            post = [f - ne[i] + feq(i, v, vv) - feq(i, u, uu) for i, f in enumerate(self.f)]
        elif om == 1.0:
            post = [feq(i, v, vv) for i in range(len(self.f))]
        else:
            post = [(1 - om) * f + (om - 1) * feq(i, u, uu) + feq(i, v, vv) for i, f in enumerate(self.f)]
        out = [torch.roll(p, [e[a] for a in range(self.D)], [self.D - 1 - a for a in range(self.D)])
               for p, e in zip(post, self.e)]
        if self.solid is not None:  # halfway bounce-back
            opp = [self.e.index(tuple(-x for x in e)) for e in self.e]
            out = [torch.where(torch.roll(self.solid, [e[a] for a in range(self.D)],
                                          [self.D - 1 - a for a in range(self.D)]), post[opp[i]], o)
                   for i, (o, e) in enumerate(zip(out, self.e))]
        self.f = out

    def state(self):
        dev = self.g if self.c["precision"] == "fp32" else 0.0
        rho = sum(self.f)
        return {"f": torch.stack([f - w * dev for f, w in zip(self.f, self.w)]), "rho": rho - dev}


def _exact_mlp(case, seed):
    x, t, p0 = (torch.from_numpy(a.astype(np.float64)).cuda() for a in _training(case, seed))
    p = p0.clone().requires_grad_(True)
    m, v, loss = torch.zeros_like(p0), torch.zeros_like(p0), None
    for it in range(1, case["iters"] + 1):
        h, at = x, 0
        for l, (i, o) in enumerate(zip(MLP_SIZES[:-1], MLP_SIZES[1:])):
            h = h @ p[at:at + o * i].reshape(o, i).T + p[at + o * i:at + o * i + o]
            at += o * i + o
            if l < len(MLP_SIZES) - 2:
                h = torch.nn.functional.gelu(h)
        loss = ((h - t) ** 2).mean()
        g, = torch.autograd.grad(loss, p)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = (p.detach() - 1e-3 * (m / (1 - 0.9 ** it)) / ((v / (1 - 0.999 ** it)).sqrt() + 1e-8)).requires_grad_(True)
    return {"params": p.detach(), "loss": float(loss)}


def exact(case, seed):
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    if case["kind"] == "batch":
        obs, mass, out = [], [], {}
        for j, c in enumerate(_batch(case, seed)):
            x = _Exact(c)
            x.start([c["nx"] // 2, c["ny"] // 2], c["radius"])
            for _ in range(case["steps"]):
                x.step()
            o, s = x.observe(0)
            obs.append(o[:4])
            mass.append(s)
            out["rho%02d" % j] = sum(x.f)
        return dict(out, obs=np.array(obs), mass=np.array(mass))
    x = _Exact(case)
    x.start(*_droplet(case, seed))
    if case["kind"] == "walls":
        x.walls(_wall(case), case["k"] ** 2 * _mu_bulk(case, x.g, x.T, math.log) - 0.005 * x.kappa / 0.1)
    obs, mass = [], []
    for s in range(case["steps"]):
        if case["kind"] == "observed":
            o, m = x.observe(min(s, 1))
            obs.append(o)
            mass.append(m)
        x.step()
    out = x.state()
    if case["kind"] == "walls":
        return {"f": out["f"][:, WALL_ROWS:], "rho": out["rho"][WALL_ROWS:]}
    if case["kind"] == "observed":
        return dict(out, obs=np.array(obs), mass=np.array(mass))
    return out
