"""The block eigen-solver of the Rayleigh-Ritz step (csrc/small_eig_block.cuh) through the
reduced problem, at block sizes p on both sides of its warps and of its shared-memory range.
The samples are B_j = w_j (D - z_j I), D = Q diag(d) Q^-1 with 20 known values d within 0.45
of the contour's centre: the trapezoid rule reproduces D - z there up to 0.45^32 = 8e-12, so
the reduced problem's eigenvalues inside the contour are the d, to 1e-9 of their size (that
error times the conditioning of Q, ~50). A block of p >= 31 vectors finds all of them;
smaller blocks report none with a small residual that is not one."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def problem():
    import paper_1906_03938_gb300 as bem
    mesh = synth.icosphere(1)
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    z, w = ctx.set_contour("circle", 4.0, 1.0, 1.0, 32)
    r = np.random.RandomState(3)
    d = 4.0 + 0.45 * np.sqrt(r.rand(20)) * np.exp(2j * np.pi * r.rand(20))
    Q = np.linalg.qr(r.randn(20, 20) + 1j * r.randn(20, 20))[0] @ (np.eye(20) + 0.1 * r.randn(20, 20))
    D = Q @ np.diag(d) @ np.linalg.inv(Q)
    B = np.stack([wj * (D - zj * np.eye(20)) for zj, wj in zip(z, w)])
    yield ctx, torch.from_numpy(B).to("cuda:0"), d
    ctx.close()


@pytest.mark.parametrize("p", [1, 2, 31, 32, 33, 63, 64, 65, 96, 150])
def test_ritz_values_are_the_known_eigenvalues(problem, p):
    ctx, B, d = problem
    lam, Y, res, its = ctx.solve_reduced(B, 4.0 + 1e-3j, p=p, max_iter=100, tol=1e-11)
    good = lam[(res <= 1e-10) & (np.abs(lam - 4.0) < 0.9)]
    dist = np.abs(good[:, None] - d[None, :])
    assert all(row.min() <= 1e-9 * 4.0 for row in dist)
    if p >= 31:
        assert sorted({int(row.argmin()) for row in dist}) == list(range(20))
