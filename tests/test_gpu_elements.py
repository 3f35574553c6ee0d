"""The element kernels at the sizes where their lane and block mapping can go wrong: one
element, fewer elements than a warp or a block, counts that are no multiple of either, blocks
of one warp and of four, the FP32 grid that walks the elements, hanging corners, every pressure
pin and a 4-byte-aligned FP32 output.  Bars as in the parity tests: relative L2 <= 1e-12 (FP64:
about 1e3 roundings of 1.1e-16 in the worst row), <= 1e-5 (FP32, 6e-8 likewise)."""
import os

import numpy as np
import pytest
import torch

import synth
from oracle import Mesh as OMesh, Oracle, Params as OParams

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def chns():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2009_06628_gb300 as chns
    if not os.path.exists(chns.LIB_PATH):
        from paper_2009_06628_gb300 import build
        build.build()
    chns.load()
    return chns


def leaves_of(dim, kind, level):
    if kind == "one":
        return np.zeros((1, 4), dtype=np.int32)
    if kind == "uniform":
        return synth.uniform_leaves(dim, level)
    return synth.sphere_band_leaves(dim, max(1, level - 3), level, [[0.4, 0.55, 0.6][:dim]], [0.27], 0.01)


CASES = [(2, "one", 1, 0, 1.0), (3, "one", 1, 2, 1.0), (2, "uniform", 1, 1, 1.0), (3, "uniform", 1, 0, 1.7),
         (2, "uniform", 3, 2, 0.9), (3, "band", 3, 1, 1.0), (2, "band", 6, 2, 1.3), (3, "band", 5, 0, 1.0),
         (3, "uniform", 5, 2, 1.0)]


@pytest.mark.parametrize("dim,kind,level,pin,hi", CASES)
def test_element_kernels(chns, dim, kind, level, pin, hi):
    leaves = leaves_of(dim, kind, level)
    om, gm = OMesh(dim, level, leaves, 0.0, hi), chns.Mesh(dim, level, leaves, 0.0, hi)
    if kind == "band":
        assert gm.H > 0 and gm.E % 32 != 0
    cfg = synth.config_params("drop3d" if dim == 3 else "drop2d")
    cfg.update(Fr=1.0, rho_ratio=20.0, eta_ratio=7.0, Cn=0.05, pin_pressure=pin)
    prm, oprm, o = chns.Params.make(**cfg), OParams(**cfg), Oracle(om)
    rng = np.random.default_rng(5)
    U = 0.1 * rng.standard_normal((om.N, dim + 3))
    U[:, dim + 1] = 1.3 * np.sin(3.0 * om.x.sum(axis=1)) + 1e-3 * rng.standard_normal(om.N)   # clipped in places
    Un = U + 1e-3 * rng.standard_normal(U.shape)
    Ut, Unt, x, w = (torch.tensor(a) for a in (U, Un, rng.standard_normal(U.shape), rng.standard_normal(U.shape)))
    d = lambda t: t.cuda()
    f = lambda t: t.cuda().float()
    rel = lambda a, b: float((a.cpu().double() - b).norm() / b.norm())
    assert rel(chns.residual(gm, prm, d(Ut), d(Unt)), o.residual(oprm, Ut, Unt)) <= 1e-12
    y = o.jvp(oprm, Ut, Unt, x)
    assert rel(chns.jvp(gm, prm, d(Ut), d(Unt), d(x)), y) <= 1e-12
    assert rel(chns.jvp(gm, prm, f(Ut), f(Unt), f(x)), y) <= 1e-5
    buf = torch.full((U.size + 1,), 7.0, dtype=torch.float32, device="cuda")
    out = buf[1:].view(U.shape)
    assert out.data_ptr() % 8 == 4
    assert rel(chns.jvp(gm, prm, f(Ut), f(Unt), f(x), out=out), y) <= 1e-5
    assert float(buf[0]) == 7.0
    gn, go, gc = chns.vjp(gm, prm, d(Ut), d(Unt), d(w))
    gno, goo, gco = o.vjp(oprm, Ut, Unt, w)
    assert rel(gn, gno) <= 1e-12 and rel(go, goo) <= 1e-12
    assert abs(float(gc.cpu()[0]) - float(gco)) <= 1e-11 * max(1.0, abs(float(gco)))
    g2, none, _ = chns.vjp(gm, prm, d(Ut), d(Unt), d(w), want_old=False, want_cn=False)
    assert none is None and rel(g2, gno) <= 1e-12


@pytest.mark.parametrize("dim,level,hi", [(2, 1, 1.0), (2, 2, 0.7), (2, 3, 1.0), (3, 1, 1.0), (3, 2, 1.4), (2, 6, 1.0)])
def test_q2_element_kernels(chns, dim, level, hi):
    """The Q2 kernels at element counts that are no multiple of a warp's 1, 2, 3 or 6 elements, blocks
    of one and of four warps, and a 4-byte-aligned FP32 output; bars as above."""
    from oracle import MeshQ2 as OMeshQ2
    om, gm = OMeshQ2(dim, level, 0.0, hi), chns.MeshQ2(dim, level, 0.0, hi)
    cfg = synth.config_params("drop3d" if dim == 3 else "drop2d")
    cfg.update(Fr=1.0, rho_ratio=20.0, eta_ratio=7.0, Cn=0.05)
    prm, oprm, o = chns.Params.make(**cfg), OParams(**cfg), Oracle(om)
    rng = np.random.default_rng(6)
    U = 0.1 * rng.standard_normal((om.N, dim + 3))
    U[:, dim + 1] = 1.3 * np.sin(3.0 * om.x.sum(axis=1))
    Un = U + 1e-3 * rng.standard_normal(U.shape)
    Ut, Unt, x, w = (torch.tensor(a) for a in (U, Un, rng.standard_normal(U.shape), rng.standard_normal(U.shape)))
    d = lambda t: t.cuda()
    f = lambda t: t.cuda().float()
    rel = lambda a, b: float((a.cpu().double() - b).norm() / b.norm())
    assert rel(chns.residual(gm, prm, d(Ut), d(Unt)), o.residual(oprm, Ut, Unt)) <= 1e-12
    y = o.jvp(oprm, Ut, Unt, x)
    assert rel(chns.jvp(gm, prm, d(Ut), d(Unt), d(x)), y) <= 1e-12
    assert rel(chns.jvp(gm, prm, f(Ut), f(Unt), f(x)), y) <= 1e-5
    out = torch.empty(U.size + 1, dtype=torch.float32, device="cuda")[1:].view(U.shape)
    assert rel(chns.jvp(gm, prm, f(Ut), f(Unt), f(x), out=out), y) <= 1e-5
    gn, go, gc = chns.vjp(gm, prm, d(Ut), d(Unt), d(w))
    gno, goo, gco = o.vjp(oprm, Ut, Unt, w)
    assert rel(gn, gno) <= 1e-12 and rel(go, goo) <= 1e-12
    assert abs(float(gc.cpu()[0]) - float(gco)) <= 1e-11 * max(1.0, abs(float(gco)))
