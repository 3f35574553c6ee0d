"""The plain adds of the colouring (scatter mode 1) where their turns can go wrong: one element, elements
with and without hanging corners in one warp, launches of a few elements, every pressure pin.
Against the atomics to rounding (FP64: 1e-13, FP32: 1e-5 relative, as between the modes elsewhere)
and the same bits from run to run."""
import os
import time

import numpy as np
import pytest
import torch

import synth

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


def setup(chns, dim, kind, level, pin):
    leaves = np.zeros((1, 4), dtype=np.int32) if kind == "one" else synth.uniform_leaves(dim, level) if kind == "uniform" else \
        synth.sphere_band_leaves(dim, max(1, level - 3), level, [[0.4, 0.55, 0.6][:dim]], [0.27], 0.01)
    gm = chns.Mesh(dim, level, leaves)
    cfg = synth.config_params("drop3d" if dim == 3 else "drop2d")
    cfg.update(Fr=1.0, rho_ratio=20.0, eta_ratio=7.0, Cn=0.05, pin_pressure=pin)
    rng = np.random.default_rng(5)
    U, V, X = (torch.tensor(0.1 * rng.standard_normal((gm.N, dim + 3)), device="cuda") for _ in range(3))
    return gm, chns.Params.make(**cfg), U, V, X


@pytest.mark.parametrize("dim,kind,level,pin", [(2, "one", 1, 0), (3, "one", 1, 1), (2, "uniform", 2, 2), (3, "uniform", 2, 1),
                                                (2, "band", 6, 1), (3, "band", 3, 0), (3, "band", 5, 2)])
def test_plain_adds(chns, dim, kind, level, pin):
    gm, prm, U, V, X = setup(chns, dim, kind, level, pin)
    assert kind != "band" or gm.H > 0
    run = lambda: (chns.residual(gm, prm, U, V), chns.jvp(gm, prm, U, V, X), *chns.vjp(gm, prm, U, V, X)[:2],
                   chns.jvp(gm, prm, U.float(), V.float(), X.float()))
    ref = run()
    gm.set_scatter(1)
    once, again = run(), run()
    for i, (r, a, b) in enumerate(zip(ref, once, again)):
        assert torch.equal(a, b), i
        assert float((a.double() - r.double()).norm()) <= (1e-5 if r.dtype == torch.float32 else 1e-13) * float(r.double().norm()), i


def test_colours_cost_their_launches(chns):
    """FP32 J x on 64^3 with 8 colours: scattered elements and 8 launches, but not the corners in turn
    (4.8 times the atomics with those, 2.6 without; bar 4)."""
    gm, prm, U, V, X = setup(chns, 3, "uniform", 6, 2)
    u, v, x = U.float(), V.float(), X.float()

    def best():
        out = 1e9
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(10):
                chns.jvp(gm, prm, u, v, x)
            torch.cuda.synchronize()
            out = min(out, time.perf_counter() - t)
        return out

    t0 = best()
    gm.set_scatter(1)
    assert best() <= 4.0 * t0
