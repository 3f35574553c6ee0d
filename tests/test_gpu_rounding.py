"""Rounding that acts on every entry alike: interpolated constants, and the scales of the Q1 exchange."""
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


def params(chns, dim, **over):
    cfg = synth.config_params("drop3d" if dim == 3 else "drop2d")
    cfg.update(dict(Fr=0.0, rho_ratio=7.0, eta_ratio=3.0), **over)
    return chns.Params.make(**cfg)


@pytest.mark.parametrize("dim,order", [(2, 1), (3, 1), (2, 2), (3, 2)])
def test_a_constant_has_no_derivative(chns, dim, order):
    """A uniform phase at rest (no gravity) has zero rows for v, p and phi, without rounding: its gradients
    are differences of equal numbers and nothing else drives it.  (As a sum of products the derivative of
    0.3 rounds to 1e-17.)"""
    gm = chns.MeshQ2(dim, 3) if order == 2 else chns.Mesh(dim, 3, synth.uniform_leaves(dim, 3))
    U = torch.zeros((gm.N, dim + 3), dtype=torch.float64, device="cuda")
    U[:, dim + 1] = 0.3
    U[:, dim + 2] = 0.3 ** 3 - 0.3
    R = chns.residual(gm, params(chns, dim), U, U)
    assert not R[:, : dim + 2].any()
    assert float(R[:, dim + 2].abs().max()) <= 1e-16      # psi'(0.3) and its nodal value, each rounded


@pytest.mark.parametrize("dim", [2, 3])
def test_fp32_mass_terms_have_no_bias(chns, dim):
    """-(N, dmu) of a random dmu: the part of the FP32 error along the result is that of the scales alone (the
    other roundings differ from entry to entry: below 1e-9 over these meshes).  f fc is f^2 to 2.3e-8 in both
    dimensions; with f in both places 2D is at -8.1e-8.  Bar 4e-8."""
    level = 8 if dim == 2 else 5
    gm = chns.Mesh(dim, level, synth.uniform_leaves(dim, level))
    prm = params(chns, dim)
    U = torch.zeros((gm.N, dim + 3), dtype=torch.float64, device="cuda")
    x = torch.zeros_like(U)
    x[:, dim + 2] = torch.tensor(synth.random_vectors(gm.N, 1, 9)[0], device="cuda").float().double()
    e = chns.jvp(gm, prm, U, U, x)[:, dim + 2]
    d = chns.jvp(gm, prm, U.float(), U.float(), x.float())[:, dim + 2].double() - e
    assert abs(float((d * e).sum() / (e * e).sum())) <= 4e-8
