"""Steps on the moments (tau = 1: the populations between the steps of one call
are not needed) against the same number of single steps, which carry the
populations, and against the oracle."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2205_09186_gb300 as pkg
    pkg.build()
    from paper_2205_09186_gb300 import lbm
    return lbm


def start(L, lattice, shape, **kw):
    nx, ny, nz = shape
    s = L.Sim(L.make_params(lattice=lattice, nx=nx, ny=ny, nz=nz, Tr=0.9, k=0.3, kappa=0.1, **kw))
    rng = np.random.default_rng(nx * 1000 + ny * 10 + nz)
    rho = 0.15 + 0.01 * rng.standard_normal((nz, ny, nx))
    s.lbm_init_density(rho)
    return s, rho


def check(L, a, b, steps, tol):
    # FP32: each path rounds a population of about 0.15 a few times per step
    # (2^-24 each), on either side: a few 1e-8 of the density per step
    a.lbm_step(steps)
    for _ in range(steps):
        b.lbm_step(1)
    assert a.lbm_get_step() == b.lbm_get_step() == steps
    fa, fb = a.lbm_get_f(), b.lbm_get_f()
    assert np.max(np.abs(fa - fb)) / 0.15 < tol
    ra, rb = a.lbm_get_density(), b.lbm_get_density()
    assert np.max(np.abs(ra - rb)) / 0.15 < tol
    assert np.max(np.abs(ra - fa.sum(0).reshape(ra.shape))) / 0.15 < 1e-6  # the density is that of the populations
    oa, ob = a.lbm_observables(), b.lbm_observables()
    assert oa["status"] == ob["status"] == 0
    assert oa["mass"] == pytest.approx(ob["mass"], rel=1e-6)


# tiles of up to 64 columns, two per lane: odd nx ends a row in half a pair, 65
# and 130 cut into 36 + 29 and 44 + 44 + 42; bands of up to 13 rows: 13 fills
# one, 14 and 27 cut unevenly; 8 wraps every halo; 2 and 3 steps end in either
# buffer
@pytest.mark.parametrize("shape", [(8, 8, 8), (64, 13, 8), (65, 14, 12), (130, 27, 9), (33, 40, 21), (12, 9, 30)])
@pytest.mark.parametrize("scheme,mu64,steps", [("EFDS2", 0, 2), ("EFDS4", 0, 3), ("EFDS6", 0, 12), ("EFDS6", 1, 3)])
def test_d3q19_steps_on_moments(L, shape, scheme, mu64, steps):
    kw = dict(scheme=scheme, precision=L.LBM_FP32DEV, mu_fp64=mu64)
    (a, rho), (b, _) = start(L, L.LBM_D3Q19, shape, **kw), start(L, L.LBM_D3Q19, shape, **kw)
    check(L, a, b, steps, 1e-6)
    o = O.Sim(lattice=O.D3Q19, nx=shape[0], ny=shape[1], nz=shape[2], Tr=0.9, k=0.3, kappa=0.1, scheme=scheme)
    o.set_f(np.stack([w * rho for w in O.lattice(O.D3Q19)[1]]))
    assert o.step(steps) == 0
    assert np.max(np.abs(a.lbm_get_density() - o.density())) / 0.15 < 1e-5


# compact schemes: lines cut into segments on 32 lanes (along x) and on 4, 8 or 16
# warps (y, z; from 64 and 128 nodes on): lengths that do not divide, shorter
# than the lanes, of exactly 64 and 128, longer than the periodic wrap of what
# enters a segment; 12 x 9 x 30 falls back to the populations
@pytest.mark.parametrize("shape", [(33, 8, 21), (12, 9, 30), (100, 64, 9), (40, 63, 128), (65, 130, 10), (513, 8, 8)])
@pytest.mark.parametrize("scheme,precision,steps", [("OCFDS4", 1, 6), ("CFDS4", 1, 2), ("CFDS6", 1, 3), ("CFDS8", 1, 5),
                                                    ("OCFDS4", 0, 4), ("CFDS8", 0, 3)])
def test_d3q19_compact_steps(L, shape, scheme, precision, steps):
    kw = dict(scheme=scheme, precision=precision)
    (a, rho), (b, _) = start(L, L.LBM_D3Q19, shape, **kw), start(L, L.LBM_D3Q19, shape, **kw)
    check(L, a, b, steps, 1e-6 if precision else 1e-12)
    o = O.Sim(lattice=O.D3Q19, nx=shape[0], ny=shape[1], nz=shape[2], Tr=0.9, k=0.3, kappa=0.1, scheme=scheme)
    o.set_f(np.stack([w * rho for w in O.lattice(O.D3Q19)[1]]))
    assert o.step(steps) == 0
    assert np.max(np.abs(a.lbm_get_density() - o.density())) / 0.15 < (1e-5 if precision else 1e-12)


@pytest.mark.parametrize("shape", [(48, 70, 1), (300, 150, 1)])
def test_d2q9_fp64_compact_steps(L, shape):
    kw = dict(scheme="OCFDS4", precision=0, tau=0.8)
    a, rho = start(L, L.LBM_D2Q9, shape, **kw)
    a.lbm_step(5)
    o = O.Sim(lattice=O.D2Q9, nx=shape[0], ny=shape[1], Tr=0.9, k=0.3, kappa=0.1, scheme="OCFDS4", tau=0.8)
    o.set_f(np.stack([w * rho[0] for w in O.lattice(O.D2Q9)[1]]))
    assert o.step(5) == 0
    assert np.max(np.abs(a.lbm_get_density() - o.density())) / 0.15 < 1e-12


# tiles of up to 60 columns x 30 rows, two columns per lane: 60 x 30 fills one,
# 61 cuts into 32 + 29, odd widths end a row in half a pair, 41 nearly fills the
# scratch, 40 is the narrowest on the moments and 33 falls back to the
# populations; 700 rows cut into many tiles
@pytest.mark.parametrize("shape", [(40, 8, 1), (33, 12, 1), (41, 40, 1), (60, 30, 1), (61, 31, 1), (119, 64, 1), (230, 37, 1),
                                   (64, 700, 1)])
@pytest.mark.parametrize("scheme,steps", [("EFDS2", 2), ("EFDS4", 3), ("EFDS6", 20), ("E4", 5), ("E8", 8)])
def test_d2q9_steps_on_moments(L, shape, scheme, steps):
    kw = dict(scheme=scheme, precision=L.LBM_FP32DEV)
    (a, rho), (b, _) = start(L, L.LBM_D2Q9, shape, **kw), start(L, L.LBM_D2Q9, shape, **kw)
    check(L, a, b, steps, 1e-6)
    o = O.Sim(lattice=O.D2Q9, nx=shape[0], ny=shape[1], Tr=0.9, k=0.3, kappa=0.1, scheme=scheme)
    o.set_f(np.stack([w * rho[0] for w in O.lattice(O.D2Q9)[1]]))
    assert o.step(steps) == 0
    assert np.max(np.abs(a.lbm_get_density() - o.density())) / 0.15 < 1e-5


def test_moments_with_another_equation_of_state(L):
    # the chemical potential of a node pair takes the scalar form
    kw = dict(lattice=L.LBM_D2Q9, nx=96, ny=60, Tr=0.85, k=0.2, kappa=0.01, scheme="EFDS4", eos="PR", a=2 / 49,
              b=2 / 21, precision=L.LBM_FP32DEV)
    a, b = L.Sim(L.make_params(**kw)), L.Sim(L.make_params(**kw))
    for s in (a, b):
        s.lbm_init_droplet(14.0)
    a.lbm_step(30)
    for _ in range(30):
        b.lbm_step(1)
    ra, rb = a.lbm_get_density(), b.lbm_get_density()
    assert np.max(np.abs(ra - rb)) / np.max(rb) < 2e-6


def test_moments_report_the_first_bad_step(L):
    # a cold second-order droplet: the density goes non-positive within the call
    kw = dict(lattice=L.LBM_D3Q19, nx=48, ny=40, nz=36, Tr=0.3, k=0.3, kappa=0.1, scheme="EFDS2",
              precision=L.LBM_FP32DEV)
    a, b = L.Sim(L.make_params(**kw)), L.Sim(L.make_params(**kw))
    for s in (a, b):
        s.lbm_init_droplet(9.0)
    a.lbm_step(400)
    for _ in range(400):
        b.lbm_step(1)
    oa, ob = a.lbm_observables(), b.lbm_observables()
    assert oa["status"] == ob["status"] == L.LBM_EUNSTABLE
    assert abs(oa["step"] - ob["step"]) <= 2


# node-parallel D3Q19 steps: 512 nodes, a last block of part of its threads, sizes
# either side of the ranges (rows of whole 16-byte chunks up to 1.2 million nodes,
# others up to 4.2, with observables 0.6) against the oracle
@pytest.mark.parametrize("shape", [(8, 8, 8), (9, 11, 13), (33, 20, 17), (64, 40, 24)])
@pytest.mark.parametrize("scheme,tau,mu64", [("EFDS2", 0.8, 0), ("EFDS4", 1.3, 0), ("EFDS6", 1.0, 0), ("EFDS4", 0.7, 1)])
def test_d3q19_node_steps(L, shape, scheme, tau, mu64):
    kw = dict(scheme=scheme, precision=L.LBM_FP32DEV, mu_fp64=mu64, tau=tau)
    (a, rho), (b, _) = start(L, L.LBM_D3Q19, shape, **kw), start(L, L.LBM_D3Q19, shape, **kw)
    o = O.Sim(lattice=O.D3Q19, nx=shape[0], ny=shape[1], nz=shape[2], Tr=0.9, k=0.3, kappa=0.1, scheme=scheme, tau=tau)
    o.set_f(np.stack([w * rho for w in O.lattice(O.D3Q19)[1]]))
    for _ in range(4):
        a.lbm_step(1)
        oo = o.observables()
        ob = b.lbm_step_observe(1)  # of the state before the step, like the oracle's
        assert o.step(1) == 0
        for key in ("max_v", "max_u"):
            assert ob[key] == pytest.approx(oo[key], rel=1e-3, abs=1e-6), key
        assert ob["mass"] == pytest.approx(oo["mass"], rel=1e-6)
    # FP32: a few roundings of 2^-24 of a population a step
    assert np.max(np.abs(a.lbm_get_density() - o.density())) / 0.15 < 1e-5
    assert np.max(np.abs(a.lbm_get_f() - o.get_f().reshape(a.lbm_get_f().shape))) / 0.15 < 1e-5
    assert np.array_equal(a.lbm_get_f(), b.lbm_get_f())


@pytest.mark.parametrize("shape", [(104, 104, 108), (160, 100, 75), (161, 161, 162), (161, 161, 161), (80, 75, 100), (84, 75, 100)])
def test_d3q19_node_range(L, shape):
    kw = dict(scheme="EFDS4", precision=L.LBM_FP32DEV, tau=0.8)
    a, rho = start(L, L.LBM_D3Q19, shape, **kw)
    b, _ = start(L, L.LBM_D3Q19, shape, **dict(kw, precision=L.LBM_FP64))
    ob = [a.lbm_step_observe(1), b.lbm_step_observe(1)]
    assert ob[0]["max_u"] == pytest.approx(ob[1]["max_u"], rel=1e-3, abs=1e-6)
    a.lbm_step(2)
    b.lbm_step(2)
    assert np.max(np.abs(a.lbm_get_density() - b.lbm_get_density())) / 0.15 < 1e-5


# D2Q9 steps at any tau and MRT: node-parallel up to 32768 nodes (181^2 and 128 x 256
# below and at the line, 129 x 255 beyond it), then tiles with overlapped launches
# (350 x 400: more tiles than SMs), against the oracle
@pytest.mark.parametrize("shape", [(8, 8, 1), (33, 17, 1), (181, 181, 1), (128, 256, 1), (129, 255, 1), (350, 400, 1)])
@pytest.mark.parametrize("scheme,tau,mrt", [("EFDS2", 0.8, 0), ("EFDS4", 1.0, 1), ("EFDS6", 1.3, 0), ("E4", 0.9, 1), ("E8", 0.9, 0)])
def test_d2q9_steps_with_relaxation(L, shape, scheme, tau, mrt):
    kw = dict(scheme=scheme, precision=L.LBM_FP32DEV, tau=tau, collision=mrt)
    a, rho = start(L, L.LBM_D2Q9, shape, **kw)
    b, _ = start(L, L.LBM_D2Q9, shape, **dict(kw, precision=L.LBM_FP64))
    a.lbm_step(3)
    a.lbm_step(1)
    b.lbm_step(4)
    # FP32: a few roundings of 2^-24 of a population a step
    assert np.max(np.abs(a.lbm_get_density() - b.lbm_get_density())) / 0.15 < 1e-5
    assert np.max(np.abs(a.lbm_get_f() - b.lbm_get_f())) / 0.15 < 1e-5
    oa, ob = a.lbm_observables(), b.lbm_observables()
    assert oa["status"] == ob["status"] == 0
    assert oa["mass"] == pytest.approx(ob["mass"], rel=1e-6)
    if shape[0] * shape[1] < 1000 and not mrt:
        o = O.Sim(lattice=O.D2Q9, nx=shape[0], ny=shape[1], Tr=0.9, k=0.3, kappa=0.1, scheme=scheme, tau=tau)
        o.set_f(np.stack([w * rho[0] for w in O.lattice(O.D2Q9)[1]]))
        assert o.step(4) == 0
        assert np.max(np.abs(a.lbm_get_density() - o.density())) / 0.15 < 1e-5


# the other population buffer is the steps' scratch and holds whatever its memory
# held: rows of odd width end in half a pair, whose other half lies in the padding
@pytest.mark.parametrize("lattice,shape,scheme", [("D3", (33, 9, 10), s) for s in ("CFDS4", "CFDS6", "CFDS8", "OCFDS4")] +
                         [("D3", (65, 14, 12), s) for s in ("OCFDS4", "EFDS2", "EFDS6")] +
                         [("D2", (61, 31, 1), s) for s in ("EFDS2", "EFDS6", "E8")] +
                         [("batch", (61, 31, 1), s) for s in ("EFDS6", "E8", "CFDS4", "OCFDS4")])
@pytest.mark.parametrize("steps", [2, 3])
def test_moments_do_not_read_what_memory_held(L, monkeypatch, lattice, shape, scheme, steps):
    import ctypes
    import torch

    def run(byte):
        class Filled(L.TorchAllocator):
            def __init__(self, *a, **kw):
                super().__init__(*a, **kw)
                held = self.held = {}

                def alloc(nbytes, ctx):
                    t = torch.full((int(nbytes),), byte, dtype=torch.uint8, device="cuda")
                    torch.cuda.synchronize()
                    held[t.data_ptr()] = t
                    return t.data_ptr()

                def free(ptr, nbytes, ctx):
                    torch.cuda.synchronize()
                    held.pop(int(ptr), None)

                self._a, self._f = L.ALLOC_FN(alloc), L.FREE_FN(free)
                self.struct = L.lbm_allocator(self._a, self._f, ctypes.c_void_p())

        monkeypatch.setattr(L, "TorchAllocator", Filled)
        nx, ny, nz = shape
        p = L.make_params(lattice=L.LBM_D3Q19 if lattice == "D3" else L.LBM_D2Q9, nx=nx, ny=ny, nz=nz, Tr=0.9, k=0.3,
                          kappa=0.1, scheme=scheme, precision=L.LBM_FP32DEV)
        if lattice == "batch":
            b = L.Batch([p, p])
            b.lbm_batch_init_droplets([7.0, 5.0])
            b.lbm_batch_step(steps)
            return [b.lbm_batch_get_density(c) for c in range(2)]
        s = L.Sim(p)
        s.lbm_init_droplet(3.0)
        s.lbm_step(steps)
        return [s.lbm_get_f(), s.lbm_get_density()]

    for a, b in zip(run(0), run(255)):  # zeros, NaN
        assert np.array_equal(a, b)


def best_ms(call, repeats=5, calls=8):
    import torch
    out = []
    for _ in range(repeats):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        call()
        e0.record()
        for _ in range(calls):
            call()
        e1.record()
        torch.cuda.synchronize()
        out.append(e0.elapsed_time(e1) / calls)
    return min(out)


def test_zchunk_does_not_reach_the_moments(L):
    # chunks of one plane collide three planes for each of theirs (and five more in
    # the prologue): two to four times the time where they are used
    kw = dict(lattice=L.LBM_D3Q19, nx=128, ny=128, nz=128, Tr=0.9, k=0.3, kappa=0.1, scheme="EFDS6",
              precision=L.LBM_FP32DEV)
    ms = []
    for zc in (0, 1):
        s = L.Sim(L.make_params(**kw))
        s.lbm_set_zchunk(zc)
        s.lbm_init_droplet(30.0)
        ms.append(best_ms(lambda: s.lbm_step(20)))
    assert ms[1] < 1.4 * ms[0], ms


def test_autotune_times_the_passes_it_cuts(L):
    # a million nodes: single steps run node-parallel, observed ones on the tiled
    # collision pass, whose time depends on the chunk by a factor of two; steps that
    # do not use it would leave the choice to chance
    kw = dict(lattice=L.LBM_D3Q19, nx=100, ny=100, nz=100, Tr=0.9, k=0.3, kappa=0.1, scheme="EFDS6",
              precision=L.LBM_FP32DEV)
    s = L.Sim(L.make_params(**kw))
    fixed = {}
    for zc in (100, 50, 25, 20, 13, 10, 7, 5):
        s.lbm_set_zchunk(zc)
        s.lbm_init_droplet(25.0)
        fixed[zc] = best_ms(lambda: s.lbm_step_observe(1))
    for _ in range(6):
        zc = s.lbm_autotune()
        assert zc > 0
        s.lbm_init_droplet(25.0)
        ms = best_ms(lambda: s.lbm_step_observe(1))
        assert ms < 1.25 * min(fixed.values()), (zc, ms, fixed)


# launches that overlap the end of the one before read what it wrote: the same bits as
# from steps that are waited for one by one (and, on the moments, from launches with
# events between them)
@pytest.mark.parametrize("lattice,shape,kw,steps", [
    ("D3", (8, 9, 10), dict(scheme="EFDS6", precision=1, tau=0.8), 3000),
    ("D3", (33, 20, 17), dict(scheme="EFDS2", precision=1, tau=0.8), 2000),
    ("D2", (16, 12, 1), dict(scheme="EFDS6", precision=1, tau=0.8), 3000),
    ("D2", (96, 70, 1), dict(scheme="E8", precision=1, collision=1), 2000),
    ("D2", (300, 150, 1), dict(scheme="EFDS4", precision=1, tau=0.9), 1000),
    ("D2", (64, 64, 1), dict(scheme="EFDS2", precision=0), 2000),
    ("D2", (100, 130, 1), dict(scheme="EFDS4", precision=0, tau=0.9), 500),
    ("D3", (12, 13, 14), dict(scheme="EFDS4", precision=0), 500),
    ("D3", (24, 20, 16), dict(scheme="OCFDS4", precision=0), 300),
    ("D2", (64, 48, 1), dict(scheme="EFDS4", precision=1, walls=True), 400),  # (the oracle diverges at 590)
    ("D3", (16, 12, 1), dict(scheme="EFDS2", precision=1, walls=True), 500),
    ("D3", (32, 24, 20), dict(scheme="EFDS6", precision=1, moments=True), 1000),
    ("D3", (33, 20, 21), dict(scheme="OCFDS4", precision=1, moments=True), 500),
    ("D2", (64, 60, 1), dict(scheme="EFDS6", precision=1, moments=True), 2000)])
def test_overlapped_launches_agree_with_separate_ones(L, lattice, shape, kw, steps):
    import torch
    kw = dict(kw)
    walls, moments = kw.pop("walls", False), kw.pop("moments", False)
    nx, ny, nz = shape if lattice == "D2" or shape[2] > 1 else shape[:2] + (12,)
    out = []
    for overlapped in (True, False):
        p = L.make_params(lattice=L.LBM_D3Q19 if lattice == "D3" else L.LBM_D2Q9, nx=nx, ny=ny, nz=nz, Tr=0.9, k=0.2,
                          kappa=0.1, **kw)
        s = L.Sim(p)
        s.lbm_init_droplet(min(d for d in (nx, ny, nz) if d > 1) / 4.0)
        if walls:
            mask = np.zeros(s.shape, np.uint8)
            mask[:3] = 1
            s.lbm_set_solid(mask, L.lbm_bulk_mu(p, L.lbm_maxwell(p)[0]))
        if overlapped:
            s.lbm_step(steps)
        elif moments:
            s.lbm_step_timed(steps)
        else:
            for _ in range(steps):
                s.lbm_step(1)
                torch.cuda.synchronize()
        rho = s.lbm_get_density()
        assert np.all(np.isfinite(rho))
        out.append(rho)
    assert np.array_equal(out[0], out[1])


# sizes in the range of the node-parallel passes whose lattice fills its tiles: a step
# is not to cost more a node than one of the same cross section just beyond the range,
# which runs on the tiled passes (on the node-parallel ones it cost 15 to 20% more)
@pytest.mark.parametrize("shape,beyond", [((96, 99, 120), 130), ((128, 88, 96), 110), ((153, 153, 153), 182)])
@pytest.mark.parametrize("scheme", ["EFDS2", "EFDS4"])
def test_d3q19_single_steps_across_the_node_range(L, shape, beyond, scheme):
    kw = dict(lattice=L.LBM_D3Q19, nx=shape[0], ny=shape[1], Tr=0.9, k=0.3, kappa=0.1, scheme=scheme,
              precision=L.LBM_FP32DEV)
    ns = []
    for nz in (shape[2], beyond):
        s = L.Sim(L.make_params(nz=nz, **kw))
        s.lbm_init_droplet(25.0)
        ns.append(best_ms(lambda: s.lbm_step(1), calls=20) / nz)
    assert ns[0] < 1.09 * ns[1], ns


# a call of two steps costs no more than two single ones where the
# populations are cheap to carry (it took 17% more on the moments)
@pytest.mark.parametrize("scheme,n,steps", [("EFDS6", 160, 2), ("EFDS2", 160, 2), ("CFDS4", 128, 2), ("CFDS4", 160, 2),
                                            ("OCFDS4", 160, 2)])
def test_short_calls_cost_no_more_than_single_steps(L, scheme, n, steps):
    s = L.Sim(L.make_params(lattice=L.LBM_D3Q19, nx=n, ny=n, nz=n, Tr=0.9, k=0.3, kappa=0.1, scheme=scheme,
                            precision=L.LBM_FP32DEV))
    s.lbm_init_droplet(30.0)
    single = best_ms(lambda: s.lbm_step(1), calls=24)
    call = best_ms(lambda: s.lbm_step(steps), calls=12) / steps
    assert call < 1.06 * single, (call, single)


# the cut of a lattice is searched in every call: on long lattices that took tens of
# thousands of trips, half a millisecond of the caller's time
@pytest.mark.parametrize("lattice,shape", [("D2", (40, 500000, 1)), ("D3", (16, 400000, 16))])
def test_calls_on_long_lattices_return_at_once(L, lattice, shape):
    import time
    import torch
    us = []
    for s3 in ((40, 64, 1) if lattice == "D2" else (16, 64, 16), shape):
        s = L.Sim(L.make_params(lattice=L.LBM_D3Q19 if lattice == "D3" else L.LBM_D2Q9, nx=s3[0], ny=s3[1], nz=s3[2],
                                Tr=0.9, k=0.3, kappa=0.1, scheme="EFDS2", precision=L.LBM_FP32DEV))
        s.lbm_init_droplet(4.0)
        best = 1e9
        for _ in range(30):
            torch.cuda.synchronize()
            t = time.perf_counter()
            s.lbm_step(2)
            best = min(best, time.perf_counter() - t)
        us.append(1e6 * best)
        s.close()
    assert us[1] < 3 * us[0] + 20, us
