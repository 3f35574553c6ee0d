"""The assembled preconditioners of the Newton step over the forms that take different routes: a
mesh whose whole polynomial or V-cycle runs in one block, mid-size levels with four lanes per row,
hanging rows, smoother degrees 2 (one pass) and above, both precisions, 2D and 3D, and the
Cahn-Hilliard block.  The preconditioner must not change the converged step (row-equilibrated
residual <= 1e-11 of the first: 1e-9 in the state, as between the mixed and the FP64 step), and
the pressure approximations must do their work: fewer GMRES iterations than plain block-Jacobi
(the Cahn-Hilliard block does not claim that on meshes of this size); each spec again after another
one (graphs and descriptions are rebuilt) takes the first one's iterations."""
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


def problem(chns, dim, leaves, level, cfg_name, **over):
    cfg = synth.config_params(cfg_name)
    cfg.update(over)
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


@pytest.mark.parametrize("dim,kind,level", [(2, "uniform", 3), (2, "band", 6), (3, "uniform", 2), (3, "band", 4),
                                            (3, "band", 5)])
def test_preconditioners_keep_the_step(chns, dim, kind, level):
    leaves = synth.uniform_leaves(dim, level) if kind == "uniform" else \
        synth.sphere_band_leaves(dim, 2, level, [[0.5] * dim], [0.25], 0.04)
    gm, prm, U0 = problem(chns, dim, leaves, level, "drop3d" if dim == 3 else "drop2d", Cn=0.05, rho_ratio=5.0,
                          eta_ratio=3.0, Fr=1.0)
    assert kind == "uniform" or gm.H > 0
    kw = dict(rtol=1e-11, atol=1e-16, restart=60, max_krylov=6000, max_newton=20)
    ref, s0 = chns.newton_step(gm, prm, chns.SolverOpts.make(precision=0, pc_type=0, krylov_rtol=1e-6, **kw), U0)
    rel = lambda a: float((a - ref).norm() / ref.norm())
    first = {}
    for pc, deg in ((1, 2), (1, 16), (2, 8), (3, 2), (3, 3), (4, 2), (4, 5), (1, 16), (4, 2)):
        for prec in (1, 0):
            o = chns.SolverOpts.make(precision=prec, pc_type=pc, pc_degree=deg, krylov_rtol=1e-4, **kw)
            U1, st = chns.newton_step(gm, prm, o, U0)
            assert st.reason == 0 and rel(U1) <= 1e-9, (pc, deg, prec, rel(U1))
            if pc in (1, 3) and gm.N > 100:
                assert st.krylov_its < s0.krylov_its, (pc, deg, prec, st.krylov_its, s0.krylov_its)
            key = (pc, deg, prec)
            assert abs(first.setdefault(key, st.krylov_its) - st.krylov_its) <= 2, key


def test_not_finite_coefficients_are_reported(chns):
    gm, prm, U0 = problem(chns, 2, synth.uniform_leaves(2, 3), 3, "drop2d")
    U0[5, 3] = float("nan")
    for pc in (1, 3):
        with pytest.raises(chns.ChnsError) as e:
            chns.newton_step(gm, prm, chns.SolverOpts.make(precision=1, pc_type=pc, pc_degree=4), U0)
        assert e.value.name == "CHNS_ENAN" and "bound" in str(e.value)


@pytest.mark.parametrize("dim,level,hi", [(2, 1, 1.0), (2, 4, 0.8), (3, 1, 1.0), (3, 3, 1.5)])
def test_nodal_blocks_give_the_diagonal_of_the_jacobian(chns, dim, level, hi):
    """Without hanging points the nodal blocks are exact, and the first norm a step reports is
    ||R / |diag J|| with J's identity rows: both from the oracle.  FP64 blocks: 1e-11 (1e3
    roundings over the quotient of two sums); FP32 blocks: 1e-4 (the same count at 6e-8)."""
    from oracle import Mesh as OMesh, Oracle, Params as OParams
    leaves = synth.uniform_leaves(dim, level)
    om, gm = OMesh(dim, level, leaves, 0.0, hi), chns.Mesh(dim, level, leaves, 0.0, hi)
    cfg = synth.config_params("drop3d" if dim == 3 else "drop2d")
    cfg.update(Fr=1.0, rho_ratio=20.0, eta_ratio=7.0, Cn=0.05)
    prm, oprm, o = chns.Params.make(**cfg), OParams(**cfg), Oracle(om)
    rng = np.random.default_rng(11)
    U = 0.1 * rng.standard_normal((om.N, dim + 3))
    U[:, dim + 1] = 1.2 * np.sin(4.0 * om.x.sum(axis=1))
    Ut = torch.tensor(U)
    dg = np.abs(np.asarray(o.jacobian(oprm, Ut, Ut).diagonal())).reshape(U.shape)
    want = float(np.linalg.norm(o.residual(oprm, Ut, Ut).numpy() / dg))
    for prec, tol in ((0, 1e-11), (1, 1e-4)):
        opts = chns.SolverOpts.make(precision=prec, pc_type=0, max_newton=0)
        _, st = chns.newton_step(gm, prm, opts, Ut.cuda(), check=False)
        assert abs(st.res0 - want) <= tol * want, (prec, st.res0, want)


@pytest.mark.parametrize("dim,level,restart,its", [(2, 2, 256, 40), (3, 2, 256, 70), (3, 2, 33, 70), (3, 5, 64, 45)])
def test_arnoldi_over_column_counts(chns, dim, level, restart, its):
    """The Gram-Schmidt kernels over their column counts (every count to 32, further chunks), an odd
    vector length (2D: 125 values) and one- and four-warp blocks, through the adjoint solve with the
    FP64 block-Jacobi alone (the FP32 polynomials are linear only up to their rounding): the
    residual that the Givens recursion reports is the true one, J^T lambda - g by the J^T w kernel,
    to 1 % (rounding is four orders below it)."""
    import ctypes
    gm, prm, U0 = problem(chns, dim, synth.uniform_leaves(dim, level), level, "drop3d" if dim == 3 else "drop2d", Cn=0.08,
                          rho_ratio=3.0, eta_ratio=2.0, Fr=1.0, dt=1e-4, pin_pressure=1)
    g = torch.tensor(synth.random_vectors(U0.numel(), 1, 5)[0], device="cuda").reshape(U0.shape)
    o = chns.SolverOpts.make(krylov_rtol=1e-6, restart=restart, max_krylov=its, pc_type=0)
    lam, go, gc, st = torch.empty_like(g), torch.empty_like(g), torch.zeros(1, dtype=torch.float64, device="cuda"), chns.Stats()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    code = chns.load().chns_step_adjoint(gm.handle, ctypes.byref(prm), ctypes.byref(o), ptr(U0), ptr(U0), ptr(g), ptr(lam),
                                         ptr(go), ptr(gc), ctypes.byref(st),
                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert chns.STATUS[code] in ("CHNS_OK", "CHNS_ENOCONV")     # short of the tolerance is fine here
    gn, gold, gcn = chns.vjp(gm, prm, U0, U0, lam)
    true = float((gn - g).norm())
    assert 0.0 < st.res_final < float(g.norm()) and abs(true - st.res_final) <= 0.01 * st.res_final, (true, st.as_dict())
    assert float((go + gold).norm()) <= 1e-12 * float(gold.norm()) and abs(float(gc + gcn)) <= 1e-11 * abs(float(gcn))


@pytest.mark.parametrize("dim,lmin,level,its", [(2, 4, 4, 40), (2, 5, 5, 9), (2, 4, 7, 40), (3, 3, 3, 70), (3, 2, 4, 33),
                                                (2, 5, 7, 40), (3, 4, 4, 40)])
def test_arnoldi_over_vector_lengths(chns, dim, lmin, level, its):
    """Vectors of 1,445 to 29,478 values, odd and even: one cluster with one and two entry pairs per
    thread, and past its range two-warp blocks.  The claim and its bound are those of the test over
    column counts: the reported residual is the true one to 1 %."""
    import ctypes
    leaves = synth.uniform_leaves(dim, level) if lmin == level else \
        synth.sphere_band_leaves(dim, lmin, level, [[0.5] * dim], [0.25], 0.04)
    gm, prm, U0 = problem(chns, dim, leaves, level, "drop3d" if dim == 3 else "drop2d", Cn=0.08, rho_ratio=3.0, eta_ratio=2.0,
                          Fr=1.0, dt=1e-4, pin_pressure=1)
    g = torch.tensor(synth.random_vectors(U0.numel(), 1, 5)[0], device="cuda").reshape(U0.shape)
    o = chns.SolverOpts.make(krylov_rtol=1e-6, restart=256, max_krylov=its, pc_type=0)
    lam, go, st = torch.empty_like(g), torch.empty_like(g), chns.Stats()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    code = chns.load().chns_step_adjoint(gm.handle, ctypes.byref(prm), ctypes.byref(o), ptr(U0), ptr(U0), ptr(g), ptr(lam),
                                         ptr(go), None, ctypes.byref(st), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert chns.STATUS[code] in ("CHNS_OK", "CHNS_ENOCONV")
    true = float((chns.vjp(gm, prm, U0, U0, lam)[0] - g).norm())
    assert 0.0 < st.res_final < float(g.norm()) and abs(true - st.res_final) <= 0.01 * st.res_final, (true, st.as_dict())
