"""The block eigen-solver of the Rayleigh-Ritz step (csrc/small_eig_block.cuh) at its smallest sizes:
p = 1 (nothing to rotate), 2 (no Hessenberg step), 3 and 5. The samples are B_j = w_j (D - z_j I), D
nu x nu with known eigenvalues within 0.45 of the centre of a 32-node contour of radius 1, which the
trapezoid rule reproduces up to 0.45^32 = 8e-12; nu is the half of the block that the iteration waits
for, so all of them must come out, to 1e-9 of their size."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu, p", [(1, 1), (1, 2), (2, 3), (3, 5)])
def test_all_eigenvalues_come_out(nu, p):
    import paper_1906_03938_gb300 as bem
    mesh = synth.icosphere(1)
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    z, w = ctx.set_contour("circle", 4.0, 1.0, 1.0, 32)
    r = np.random.RandomState(7)
    d = 4.0 + 0.45 * np.sqrt(r.rand(nu)) * np.exp(2j * np.pi * r.rand(nu))
    Q = np.linalg.qr(r.randn(nu, nu) + 1j * r.randn(nu, nu))[0] @ (np.eye(nu) + 0.1 * r.randn(nu, nu))
    D = Q @ np.diag(d) @ np.linalg.inv(Q)
    B = torch.from_numpy(np.stack([wj * (D - zj * np.eye(nu)) for zj, wj in zip(z, w)])).to("cuda:0")
    lam, Y, res, its = ctx.solve_reduced(B, 4.0 + 1e-3j, p=p, max_iter=200, tol=1e-11)
    ctx.close()
    dist = np.abs(d[:, None] - lam[None, :])
    assert np.all(dist.min(1) <= 4e-9)
    assert np.all(res[dist.argmin(1)] <= 1e-10)
