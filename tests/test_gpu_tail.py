"""Which levels the one-block preconditioner kernel takes: meshes on both sides of its limits (rows per
thread, row width, entries, smoother degree), a V-cycle whose coarsest level is past the entry limit,
and a mesh that it must not slow down."""
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


def problem(chns, dim, lmin, level, band):
    leaves = synth.uniform_leaves(dim, level) if lmin == level else \
        synth.sphere_band_leaves(dim, lmin, level, [[0.5] * dim], [0.25], band)
    cfg = synth.config_params("drop3d" if dim == 3 else "drop2d")
    cfg.update(Cn=0.08, rho_ratio=3.0, eta_ratio=2.0, Fr=1.0, dt=1e-4)
    gm = chns.Mesh(dim, level, leaves)
    x = gm.node_x()
    U = np.zeros((gm.N, dim + 3))
    U[:, dim + 1] = synth.drop_phi(x, [[0.5] * dim], [0.25], cfg["Cn"], noise=1e-3, seed=3)
    U[:, :dim] = synth.fourier_velocity(x, 6, 4, 0.1)
    U[np.any((x <= 0.0) | (x >= 1.0), axis=1), :dim] = 0.0
    U = torch.tensor(U, device="cuda")
    prm = chns.Params.make(**cfg)
    chns.initial_mu(gm, prm, U)
    return gm, prm, U


@pytest.mark.parametrize("dim,lmin,level,band,rows", [(2, 4, 4, 0, 289), (2, 5, 5, 0, 1089), (2, 3, 6, 0.02, 733),
                                                      (2, 3, 7, 0.01, 1497), (2, 4, 7, 0.03, 2681), (2, 6, 6, 0, 4225),
                                                      (3, 3, 3, 0, 729), (3, 2, 3, 0.02, 301), (3, 3, 4, 0.01, 1049)])
def test_the_step_on_both_sides_of_the_limits(chns, dim, lmin, level, band, rows):
    """Every preconditioner gives the step of the nodal blocks alone: row-equilibrated residual <= 1e-11 of
    the first, 1e-9 in the state (as between the mixed and the FP64 step)."""
    gm, prm, U0 = problem(chns, dim, lmin, level, band)
    assert gm.N == rows
    kw = dict(rtol=1e-11, atol=1e-16, restart=256, max_krylov=6000, krylov_rtol=1e-6)
    ref, _ = chns.newton_step(gm, prm, chns.SolverOpts.make(precision=0, pc_type=0, **kw), U0)
    for pc, deg in ((1, 2), (1, 4), (1, 5), (1, 16), (3, 2), (3, 5), (4, 2), (1, 5)):
        U1, st = chns.newton_step(gm, prm, chns.SolverOpts.make(precision=1, pc_type=pc, pc_degree=deg, **kw), U0)
        assert float((U1 - ref).norm()) <= 1e-9 * float(ref.norm()), (pc, deg, st.as_dict())


def test_a_small_polynomial_costs_no_more_than_a_large_one(chns):
    """An application on 4,225 rows takes no longer than on 16,641 of the same kind (both are chains of
    launches, a third of what the smaller one took in one block; 1.5: noise)."""
    us = []
    for level in (6, 7):
        gm, prm, U0 = problem(chns, 2, level, level, 0)
        o = chns.SolverOpts.make(precision=1, pc_type=1, pc_degree=16, restart=30, max_krylov=60, max_newton=1, krylov_rtol=1e-12)
        runs = [chns.newton_step(gm, prm, o, U0, check=False)[1] for _ in range(5)]
        us.append(min(s.apply_ms / s.krylov_its for s in runs))
    assert us[0] <= 1.5 * us[1], us


def test_set_up_of_the_largest_degree(chns):
    """Degree 200 (the largest) gives the step of the nodal blocks, bar as above, and its set-up is not a
    chain of divisions: the residual and set-up of a small mesh take at most 1.4 times as long as with degree
    2 (1.8 with 0.6 us per degree)."""
    gm, prm, U0 = problem(chns, 2, 4, 4, 0)
    kw = dict(rtol=1e-11, atol=1e-16, restart=256, max_krylov=6000, krylov_rtol=1e-6)
    ref, _ = chns.newton_step(gm, prm, chns.SolverOpts.make(precision=0, pc_type=0, **kw), U0)
    U1, st = chns.newton_step(gm, prm, chns.SolverOpts.make(precision=1, pc_type=1, pc_degree=200, **kw), U0)
    assert float((U1 - ref).norm()) <= 1e-9 * float(ref.norm()), st.as_dict()

    def best(degree):
        o = chns.SolverOpts.make(precision=1, pc_type=1, pc_degree=degree, max_newton=0)
        out = 1e9
        for _ in range(20):
            torch.cuda.synchronize()
            t = time.perf_counter()
            chns.newton_step(gm, prm, o, U0, check=False)
            out = min(out, time.perf_counter() - t)
        return out

    assert best(200) <= 1.4 * best(2)
