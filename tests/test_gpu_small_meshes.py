"""FP64 projections and residuals on meshes of a few panels, on both sides of the sizes from which the
expansion over the wavenumbers (csrc/expand64.cu) takes the place of the direct and the double-FP32
forms, against the oracle. Bar: 1e-11 of the largest entry, the FP64 paths' bar throughout."""
import numpy as np
import pytest
import torch

import synth
from oracle import assembly as oasm

pytestmark = pytest.mark.gpu


def _columns(a):
    t = torch.empty((a.shape[1], a.shape[0]), dtype=torch.complex128, device="cuda:0")
    return t.copy_(torch.from_numpy(np.ascontiguousarray(a.T))).t()


@pytest.mark.parametrize("op", [(1.0, 0.0), (0.5 + 0.2j, 1.0 - 0.3j)])
@pytest.mark.parametrize("near", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 39, 40, 41, 48, 64])
def test_against_the_oracle(n, near, op):
    import paper_1906_03938_gb300 as bem
    full = synth.cube_sphere(3, (1.0, 0.8, 0.55))
    mesh = synth.Mesh("part", full.xyz, full.tri[:n])
    nu = min(n, 5)
    V = synth.complex_gaussian(n, nu, 3)
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_operator(*op)
    ctx.set_near_field(near)
    z, w = ctx.set_contour("circle", 4.0, 0.8, 0.8, 6)
    B, Y = (t.cpu().numpy() for t in ctx.project(_columns(V), bem.PREC_FP64, AV=True))
    lam = z[:nu]
    R = [ctx.residual_arith(lam, _columns(V), arith=a)[1].cpu().numpy() for a in (0, 1)]
    ctx.check()
    ctx.close()
    for j in range(6):
        AV = oasm.matrix(mesh, z[j], near=bool(near), op=op) @ V
        ref = w[j] * (V.conj().T @ AV)
        assert np.max(np.abs(Y[j] - AV)) < 1e-11 * np.max(np.abs(AV))
        assert np.max(np.abs(B[j] - ref)) < 1e-11 * np.max(np.abs(ref))
        if j < nu:
            for a in (0, 1):
                assert np.max(np.abs(R[a][:, j] - AV[:, j])) < 1e-11 * np.max(np.abs(AV[:, j]))
