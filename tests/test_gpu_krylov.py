"""The Gram-Schmidt kernels at the edges of their ranges: Arnoldi cycles of up to 256 columns (the
largest restart), and vector lengths of every split.  The adjoint solve with the FP64 block-Jacobi
alone reports the residual of its Givens recursion, and the J^T w kernel gives the true one: they
agree to 1 % (the solves stop at 1e-1 to 1e-6 of the right-hand side, where rounding is at
1e-9, by the oracle's Jacobian in a host restatement of the same recursion)."""
import ctypes
import os

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


def problem(chns, dim, leaves, level, **over):
    cfg = synth.config_params("drop3d" if dim == 3 else "drop2d")
    cfg.update(dict(Cn=0.08, rho_ratio=3.0, eta_ratio=2.0, Fr=1.0, dt=1e-4), **over)
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


def adjoint_claim(chns, gm, prm, U0, restart, its):
    """(reported, true, |g|, iterations) of an adjoint solve stopped after `its` iterations."""
    g = torch.tensor(synth.random_vectors(U0.numel(), 1, 5)[0], device="cuda").reshape(U0.shape)
    o = chns.SolverOpts.make(krylov_rtol=1e-6, restart=restart, max_krylov=its, pc_type=0)
    lam, go, st = torch.empty_like(g), torch.empty_like(g), chns.Stats()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    code = chns.load().chns_step_adjoint(gm.handle, ctypes.byref(prm), ctypes.byref(o), ptr(U0), ptr(U0), ptr(g), ptr(lam),
                                         ptr(go), None, ctypes.byref(st), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert chns.STATUS[code] in ("CHNS_OK", "CHNS_ENOCONV")     # short of the tolerance is fine here
    return st.res_final, float((chns.vjp(gm, prm, U0, U0, lam)[0] - g).norm()), float(g.norm()), st.krylov_its


@pytest.mark.parametrize("its", [100, 160, 255, 256, 300])
def test_adjoint_cycles_up_to_256_columns(chns, its):
    """21,125 values (2D, 64^2).  300: a full cycle of 256 columns and a restart."""
    gm, prm, U0 = problem(chns, 2, synth.uniform_leaves(2, 6), 6, pin_pressure=1)
    assert U0.numel() <= 32768
    claim, true, norm, done = adjoint_claim(chns, gm, prm, U0, 256, its)
    assert done == its
    assert 0.0 < claim < norm and abs(true - claim) <= 0.01 * claim, (true, claim)


@pytest.mark.parametrize("precision", [0, 1])
def test_newton_cycles_of_256_columns(chns, precision):
    """The Newton step, whose cluster decides by |w|^2 before and after a pass whether a second one
    follows, through several cycles of 256 columns per linear solve: the converged step is that of the
    pressure preconditioner's short solves (row-equilibrated residual <= 1e-11 of the first: 1e-9 in the
    state, as between the mixed and the FP64 step)."""
    gm, prm, U0 = problem(chns, 2, synth.uniform_leaves(2, 6), 6)
    kw = dict(precision=precision, rtol=1e-11, atol=1e-16, krylov_rtol=1e-6, restart=256, max_krylov=4000)
    U1, st = chns.newton_step(gm, prm, chns.SolverOpts.make(pc_type=0, **kw), U0)
    U2, _ = chns.newton_step(gm, prm, chns.SolverOpts.make(pc_type=1, pc_degree=16, **kw), U0)
    assert U0.numel() <= 32768 and max(st.as_dict()["krylov_hist"]) > 2 * 256
    assert float((U1 - U2).norm()) <= 1e-9 * float(U2.norm())


def test_breakdown_leaves_nothing_in_flight(chns):
    """The call synchronises its stream, also where it gives up in the middle of an Arnoldi cycle with
    the next operator application queued: velocities whose squares leave FP32 (not FP64) make the
    operator's result not finite."""
    gm, prm, U0 = problem(chns, 3, synth.uniform_leaves(3, 6), 6)
    U0[:, :3] *= 1e25
    opts = chns.SolverOpts.make(precision=1, pc_type=0, restart=30)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        out = torch.empty_like(U0)
        torch.cuda.synchronize()
        _, st = chns.newton_step(gm, prm, opts, U0, out, check=False)
        idle = s.query()
    torch.cuda.synchronize()
    assert chns.STATUS[st.reason] == "CHNS_EBREAKDOWN" and st.jvp_calls == 2
    assert idle


@pytest.mark.parametrize("dim,lmin,level,band,n,its", [
    (2, 4, 4, 0, 1445, 33), (2, 5, 5, 0, 5445, 70),                                # cluster, then 8 lanes per pair
    (2, 5, 7, 0.02, 13605, 40), (2, 6, 7, 0.06, 34105, 70),                        # 4 lanes; 2, odd, past the cluster
    (3, 4, 5, 0.01, 37518, 40), (3, 4, 5, 0.02, 46014, 70), (2, 7, 7, 0, 83205, 70),   # 2 lanes, 1 lane (even, odd)
    (2, 9, 9, 0, 1315845, 40)])                                                    # a kernel per column count, odd, two launches
def test_adjoint_over_the_splits(chns, dim, lmin, level, band, n, its):
    """Column counts on both sides of 8, 32 and 64, vectors of each split of the work, odd and even."""
    leaves = synth.uniform_leaves(dim, level) if lmin == level else \
        synth.sphere_band_leaves(dim, lmin, level, [[0.5] * dim], [0.2 if n == 37518 else 0.25], band)
    gm, prm, U0 = problem(chns, dim, leaves, level, pin_pressure=1)
    assert U0.numel() == n
    claim, true, norm, done = adjoint_claim(chns, gm, prm, U0, 256, its)
    assert done == its
    assert 0.0 < claim < norm and abs(true - claim) <= 0.01 * claim, (true, claim)
