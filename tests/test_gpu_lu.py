"""The dense LU's sub-panel and substitution kernels (csrc/dense32.cu) through the inverse
power step, whose one solve is u' = S^{-1} b: sizes around the 32-row blocks and the 256-row
panels against the oracle's FP64 step, and sizes above the sub-panel cluster's and the
one-launch substitution's rows against the matrix-free solve. Bar: 1e-3 in direction per
column, the inverse power step's bar (FP32 factors of a well-conditioned sum)."""
import numpy as np
import pytest
import torch

import synth
from oracle import assembly as oasm, rr as orr

pytestmark = pytest.mark.gpu
SPEC = ("circle", 4.5, 1.0, 1.0, 8)


def _ctx(xyz, tri):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    ctx.set_mesh(xyz, tri)
    return bem, ctx, *ctx.set_contour(*SPEC)


def _misaligned(a, b):
    """Largest sine of the angle between the columns of a and b."""
    dot = np.abs(np.sum(np.conj(a) * b, 0)) / (np.linalg.norm(a, axis=0) * np.linalg.norm(b, axis=0))
    return np.sqrt(np.max(np.maximum(0.0, 1.0 - dot ** 2)))


@pytest.mark.parametrize("n, nu", [(1, 1), (12, 3), (31, 1), (32, 2), (33, 2), (63, 3), (64, 1),
                                   (255, 2), (257, 5), (289, 33)])
def test_small_sizes_match_the_oracle(n, nu):
    mesh = synth.cube_sphere(5, (1.0, 0.8, 0.55))
    mesh = synth.Mesh("part", mesh.xyz, mesh.tri[:n])
    bem, ctx, z, w = _ctx(mesh.xyz, mesh.tri)
    V0 = synth.complex_gaussian(n, nu, 4)
    V = bem.fortran(torch.from_numpy(V0).to("cuda:0"))
    ctx.inverse_power(V, 1, 4.5 + 0.3j)
    ctx.close()
    B = np.stack([w[j] * oasm.matrix(mesh, z[j]) for j in range(len(z))])
    assert _misaligned(V.cpu().numpy(), orr.inverse_power(B, z, 4.5 + 0.3j, V0, 1)) < 1e-3


@pytest.mark.parametrize("m", [25, 38])   # 7500 and 17328 panels
def test_large_sizes_match_the_matrix_free_solve(m):
    mesh = synth.cube_sphere(m, (1.0, 0.8, 0.55))
    bem, ctx, z, w = _ctx(mesh.xyz, mesh.tri)
    V0 = torch.from_numpy(synth.complex_gaussian(mesh.n, 3, 4)).to("cuda:0")
    V, W = bem.fortran(V0), bem.fortran(V0.clone())
    ctx.inverse_power(V, 1, 4.5 + 0.3j)
    ctx.inverse_power_mf(W, 1, 4.5 + 0.3j, tol=2e-5, max_iter=2000)
    ctx.close()
    assert _misaligned(V.cpu().numpy(), W.cpu().numpy()) < 1e-3
