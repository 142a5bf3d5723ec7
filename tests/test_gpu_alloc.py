"""Allocations that fail: reported by their call, not by the next one; buffers the
library can do without (the FP64 step's chemical potential, the training launch's
scratch) leave the slower passes, with the same results."""
import ctypes

import numpy as np
import pytest

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


def refusing(L, base, refuse):
    """The allocator `base` returning NULL where refuse(bytes, calls so far) holds."""
    class Refusing(base):
        def __init__(self, *a, **kw):
            super().__init__(*a, **kw)
            inner, self.calls, self.refused = self._a, [], []

            def alloc(nbytes, ctx):
                self.calls.append(nbytes)
                if refuse(nbytes, self.calls):
                    self.refused.append(nbytes)
                    return None
                return inner(nbytes, ctx)

            self.inner, self._a = inner, L.ALLOC_FN(alloc)
            self.struct = L.lbm_allocator(self._a, self._f, ctypes.c_void_p())
    return Refusing


@pytest.mark.parametrize("call", ["observables", "forward", "compact", "get_f"])
def test_failed_allocation_leaves_no_error_behind(L, call):
    kw = dict(lattice=L.LBM_D3Q19, nx=32, ny=32, nz=32, Tr=0.9, k=0.3, kappa=0.1, precision=L.LBM_FP32DEV)
    s = L.Sim(L.make_params(scheme="OCFDS4" if call == "compact" else "EFDS4", **kw))
    s.lbm_init_droplet(8.0)
    m = L.MLP([4, 8, 2], 4)
    m.lbm_mlp_set_params(np.zeros(m.nparam))
    with pytest.raises(L.LBMError) as e:
        L.MLP([128, 128], 1 << 30, allocator=None)  # 2 TB of gradient shares
    assert e.value.code == L.LBM_ENOMEM
    if call == "observables":
        assert s.lbm_observables()["status"] == 0
    elif call == "forward":
        assert np.array_equal(m.lbm_mlp_forward(np.ones((2, 4))), np.zeros((2, 2)))
    elif call == "compact":
        s.lbm_step(1)
        assert s.lbm_get_step() == 1
    else:
        assert np.all(np.isfinite(s.lbm_get_f()))


@pytest.mark.parametrize("lattice,shape,scheme", [("D2", (48, 40, 1), "EFDS6"), ("D2", (48, 40, 1), "E8"),
                                                  ("D3", (16, 12, 20), "EFDS4"), ("D3", (16, 12, 20), "E4")])
def test_fp64_steps_without_their_chemical_potential_buffer(L, monkeypatch, lattice, shape, scheme):
    nx, ny, nz = shape
    p = L.make_params(lattice=L.LBM_D3Q19 if lattice == "D3" else L.LBM_D2Q9, nx=nx, ny=ny, nz=nz, Tr=0.9, k=0.3,
                      kappa=0.1, scheme=scheme, tau=0.9)
    rho = 0.15 + 0.01 * np.random.default_rng(1).standard_normal((nz, ny, nx))
    n = 8 * nx * ny * nz
    out, base = [], L.TorchAllocator
    for refuse in (lambda b, c: False, lambda b, c: b == n and c.count(n) == 4):  # after two densities and a snapshot
        monkeypatch.setattr(L, "TorchAllocator", refusing(L, base, refuse))
        s = L.Sim(p)
        s.lbm_init_density(rho)
        refused = list(s._alloc.refused)
        s.lbm_step(5)
        assert s.lbm_get_step() == 5
        out.append((s.lbm_get_f(), refused))
    assert out[0][1] == [] and out[1][1] == [n]
    assert np.max(np.abs(out[1][0] - out[0][0])) / 0.15 < 1e-13  # FP64: a few roundings of 2^-53 a step


def test_training_without_its_scratch(L, monkeypatch):
    sizes, batch = [4, 40, 24, 6], 20
    rng = np.random.default_rng(2)
    x, t = (rng.uniform(-1, 1, (batch, n)).astype(np.float32) for n in (sizes[0], sizes[-1]))
    w = np.concatenate([np.r_[rng.standard_normal(o * i) / np.sqrt(i), np.zeros(o)] for i, o in
                        zip(sizes[:-1], sizes[1:])]).astype(np.float32)
    out, base = [], L.TorchAllocator
    for refuse in (lambda b, c: False, lambda b, c: len(c) == 13):  # after the twelve buffers it needs
        monkeypatch.setattr(L, "TorchAllocator", refusing(L, base, refuse))
        m = L.MLP(sizes, batch)
        m.lbm_mlp_set_params(w)
        m.lbm_mlp_set_data(x, t)
        loss = m.lbm_mlp_train(10, 1e-3)
        out.append((m.lbm_mlp_get_params(), loss, len(m._alloc.refused)))
    assert [o[2] for o in out] == [0, 1]
    assert out[1][1] == pytest.approx(out[0][1], rel=1e-4)
    d = np.abs(out[1][0] - out[0][0])  # Adam's steps of 1e-3 follow FP32 gradients, off by 1e-7 of their scale
    assert np.quantile(d, 0.99) < 1e-4 and np.median(d) < 1e-6
