"""The tiled collision pass of D3Q19 FP32DEV steps (k_coll3d) and the tiled D2Q9 steps at
the edges of their tiles.  Smaller lattices run one thread per node and calls of several
steps at tau = 1 carry the moments, so: lattices beyond those sizes, a step a call (long
in z, which costs nothing but chunks).  Against FP64 handles, which share no kernel with
them, and against themselves bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL32 = 1e-5  # of the density scale: a few roundings of 2^-24 of a population a step


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2205_09186_gb300 as pkg
    pkg.build()
    from paper_2205_09186_gb300 import lbm
    return lbm


def sim(L, shape, precision=1, **kw):
    nx, ny, nz = shape
    return L.Sim(L.make_params(lattice=L.LBM_D3Q19 if nz > 1 else L.LBM_D2Q9, nx=nx, ny=ny, nz=nz, Tr=0.9, k=0.3, kappa=0.1,
                               precision=precision, **kw))


def noise(shape):
    nx, ny, nz = shape
    rho = 0.15 + 0.01 * np.random.default_rng(nx * 1000 + ny * 10 + nz).standard_normal((nz, ny, nx))
    return rho


# tiles of 32 columns x 11 rows.  Rows of whole 16-byte chunks (tensor copies), beyond 1.2
# million nodes: 45 rows leave a last band of one row, which takes one from the band
# before; 11 are one band whose edge rows feed each other; 8 columns are one tile that
# wraps; 36 leave a last tile of four columns.  Other rows (4-byte copies), beyond 4.2
# million: 33 and 65 leave a last tile of one column; 9 wrap; 42.  The last chunk of z
# is a shorter one
ALIGNED = [(64, 45, 421), (68, 11, 1609), (8, 45, 3347), (36, 12, 2779), (32, 23, 1637)]
RAGGED = [(65, 45, 1447), (33, 11, 11579), (9, 45, 10391), (42, 26, 3851), (33, 34, 3761)]


@pytest.mark.parametrize("shape", ALIGNED + RAGGED)
@pytest.mark.parametrize("scheme,tau,mu64", [("EFDS2", 1.0, 0), ("EFDS6", 1.0, 0), ("EFDS4", 0.8, 0), ("EFDS6", 1.3, 1)])
def test_single_steps_at_the_edges_of_tiles(L, shape, scheme, tau, mu64):
    assert np.prod(shape) > (1200000 if shape[0] % 4 == 0 else 4200000)
    rho = noise(shape)
    a, b = sim(L, shape, scheme=scheme, tau=tau, mu_fp64=mu64), sim(L, shape, 0, scheme=scheme, tau=tau)
    for s in (a, b):
        s.lbm_init_density(rho)
        for _ in range(4):
            s.lbm_step(1)
    assert np.max(np.abs(a.lbm_get_density() - b.lbm_get_density())) / 0.15 < TOL32
    assert np.max(np.abs(a.lbm_get_f() - b.lbm_get_f())) / 0.15 < TOL32


# with observables, beyond 0.6 million nodes
@pytest.mark.parametrize("shape", [(64, 45, 211), (68, 11, 811), (8, 45, 1681), (36, 12, 1397), (65, 45, 211), (33, 11, 1663),
                                   (9, 45, 1493), (42, 26, 557)])
@pytest.mark.parametrize("scheme,tau", [("EFDS6", 1.0), ("EFDS2", 0.8)])
def test_observed_steps_at_the_edges_of_tiles(L, shape, scheme, tau):
    assert np.prod(shape) > 600000
    rho = noise(shape)
    a, b = sim(L, shape, scheme=scheme, tau=tau), sim(L, shape, 0, scheme=scheme, tau=tau)
    for s in (a, b):
        s.lbm_init_density(rho)
    for _ in range(3):
        oa, ob = a.lbm_step_observe(1), b.lbm_step_observe(1)
        assert oa["status"] == ob["status"] == 0
        for key in ("max_v", "max_u", "max_drho"):
            assert oa[key] == pytest.approx(ob[key], rel=1e-3, abs=1e-6), key
        assert oa["mass"] == pytest.approx(ob["mass"], rel=1e-6)
    assert np.max(np.abs(a.lbm_get_density() - b.lbm_get_density())) / 0.15 < TOL32


# band edge rows and tile edge columns receive two atomic additions onto zero, corners
# exact integer additions: runs agree bit for bit, whatever the chunk
@pytest.mark.parametrize("shape", [(64, 45, 421), (65, 45, 1447)])
@pytest.mark.parametrize("observed", [False, True])
def test_tiled_steps_are_bitwise_reproducible_over_chunks(L, shape, observed):
    outs = []
    for zc in (0, 0, 5, 64, shape[2], -1):
        s = sim(L, shape, scheme="EFDS6", tau=0.8)
        if zc < 0:
            assert s.lbm_autotune() > 0
        else:
            s.lbm_set_zchunk(zc)
        s.lbm_init_density(noise(shape))
        for _ in range(5):
            s.lbm_step_observe(1) if observed else s.lbm_step(1)
        outs.append((s.lbm_get_f(), s.lbm_get_density()))
    for f, r in outs[1:]:
        assert np.array_equal(f, outs[0][0]) and np.array_equal(r, outs[0][1])


# tiles of 16, 32 and 64 rows beyond 32768 nodes: the same arithmetic per node
@pytest.mark.parametrize("shape", [(300, 150, 1), (301, 127, 1), (40, 900, 1)])
@pytest.mark.parametrize("scheme,kw", [("EFDS6", dict(tau=0.8)), ("EFDS2", dict(tau=1.0)), ("E8", dict(tau=0.9)),
                                       ("E4", dict(collision=1))])
def test_d2q9_tile_rows_beyond_the_node_range(L, shape, scheme, kw):
    assert np.prod(shape) > 32768
    out = {}
    for rows in (1, 2, 4):
        s = sim(L, shape, scheme=scheme, **kw)
        s.lbm_set_tile_rows(rows)
        s.lbm_init_density(noise(shape))
        for _ in range(10):
            s.lbm_step(1)
        out[rows] = s.lbm_get_f()
    assert np.array_equal(out[1], out[2]) and np.array_equal(out[4], out[2])
    b = sim(L, shape, 0, scheme=scheme, **kw)
    b.lbm_init_density(noise(shape))
    b.lbm_step(10)
    assert np.max(np.abs(out[2] - b.lbm_get_f())) / 0.15 < TOL32
