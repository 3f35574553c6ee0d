"""The mass-matrix solves and the mass and energy sums where their lane and block mapping can go
wrong: one element, fewer elements than a block, counts that are no multiple of one, more blocks
than the grid holds at once, hanging corners, boxes that are not the unit box, with and without
gravity.  The solves stop at a residual of 1e-14 |rhs|; what is left in the true residual besides
is the rounding of the right-hand side and of the matrix product, about 1e3 roundings of 1.1e-16 in
the worst row: bar 1e-12 (with |M| |x| beside |rhs| where the level differences make x large).  The
sums round like sqrt(their terms): 1e-13 of the sum of magnitudes for the mass, 1e-12 for the
energy's parts (cubes of rounded values; no cancellation, every part is positive here)."""
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


CASES = [(2, "one", 1, 1.0), (3, "one", 1, 1.0), (2, "uniform", 1, 2.5), (3, "uniform", 2, 1.0), (2, "band", 7, 0.7),
         (3, "band", 5, 1.9), (3, "uniform", 5, 1.0)]


@pytest.mark.parametrize("dim,kind,level,hi", CASES)
def test_mass_solves_and_sums(chns, dim, kind, level, hi):
    if kind == "one":
        leaves = np.zeros((1, 4), dtype=np.int32)
    elif kind == "uniform":
        leaves = synth.uniform_leaves(dim, level)
    else:
        leaves = synth.sphere_band_leaves(dim, level - 3, level, [[0.4, 0.55, 0.6][:dim]], [0.27], 0.01)
    om, gm = OMesh(dim, level, leaves, 0.0, hi), chns.Mesh(dim, level, leaves, 0.0, hi)
    o = Oracle(om)
    if kind == "band":
        assert gm.H > 0
    rng = np.random.default_rng(11)
    U = torch.tensor(0.3 * rng.standard_normal((om.N, dim + 3)))
    U[:, dim + 1] = 1.2 * torch.sin(2.0 * torch.tensor(om.x).sum(1)) + 0.05 * U[:, 0]   # clipped in places
    M = o.mass_matrix().tocsr()
    for Fr in (1.0, 1e30):
        cfg = synth.config_params("drop3d" if dim == 3 else "drop2d")
        cfg.update(Fr=Fr, rho_ratio=9.0, Cn=0.05)
        prm, oprm = chns.Params.make(**cfg), OParams(**cfg)
        for a, b in zip(chns.energy(gm, prm, U.cuda()), o.energy(oprm, U)):
            assert abs(a - b) <= 1e-12 * abs(b) + 1e-40
    m = M @ np.ones(om.N)
    assert abs(chns.mass(gm, U.cuda()) - o.mass(U)) <= 1e-13 * float(np.abs(m * U[:, dim + 1].numpy()).sum())
    out = U.cuda()
    chns.initial_mu(gm, prm, out)
    mu, b = out[:, dim + 2].cpu().numpy(), o.mu_rhs(U[:, dim + 1], cfg["Cn"]).numpy()
    scale = np.linalg.norm(b) + np.linalg.norm(abs(M) @ abs(mu))
    assert np.linalg.norm(M @ mu - b) <= 1e-12 * scale
    assert torch.equal(out[:, : dim + 2].cpu(), U[:, : dim + 2])
    x0 = rng.standard_normal(om.N)
    rhs = M @ x0
    x = chns.mass_solve(gm, torch.tensor(rhs).cuda()).cpu().numpy()
    assert np.linalg.norm(M @ x - rhs) <= 1e-12 * (np.linalg.norm(rhs) + np.linalg.norm(abs(M) @ abs(x)))
    assert not chns.mass_solve(gm, torch.zeros(om.N, dtype=torch.float64, device="cuda")).any()
