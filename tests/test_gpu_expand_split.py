"""The expanded FP64 products on the tensor core (csrc/split64.cu, split64_batch): projections
wide enough for it against the same columns a few at a time, which take the FP64 products
(sizes around the 128-row, 32-column and 16-deep tiles; operators, near field, strides), and one
problem whose moments come in two parts against the oracle.

Bars: both forms sum n products of entries good to a few eps; 1e-13 of the largest entry is a
hundred times the root of the longest sum's error and the accuracy the series keeps. The oracle:
1e-11, the FP64 paths' bar throughout."""
import numpy as np
import pytest
import torch

import synth
from oracle import assembly as oasm

pytestmark = pytest.mark.gpu
OPS = {"single": (1.0, 0.0), "neumann": (0.0, 1.0), "robin": (0.5 + 0.2j, 1.0 - 0.3j)}


def _ctx(mesh, op, near):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_operator(*OPS[op])
    ctx.set_near_field(near)
    return bem, ctx


def _strided(a, ld):
    buf = torch.zeros((a.shape[1], ld), dtype=torch.complex128, device="cuda:0")
    buf[:, :a.shape[0]] = torch.from_numpy(a.T.copy())
    return buf.t()[:a.shape[0]]


@pytest.mark.parametrize("op", list(OPS))
@pytest.mark.parametrize("m, nu, near, pad", [(5, 32, 0, 0), (5, 33, 1, 3), (6, 97, 0, 1), (7, 64, 1, 0)])
def test_against_narrow(op, m, nu, near, pad):
    mesh = synth.cube_sphere(m, (1.0, 0.8, 0.55))
    bem, ctx = _ctx(mesh, op, near)
    N = 8
    ctx.set_contour("ellipse", 5.0, 0.8, 0.4, N)
    V = synth.complex_gaussian(mesh.n, nu, 3) * np.logspace(0, -6, nu)
    B, Y = ctx.project(_strided(V, mesh.n + pad), bem.PREC_FP64, AV=True)
    for c0 in range(0, nu, 4):
        sub = _strided(V[:, c0:c0 + 4], mesh.n)
        _, Y1 = ctx.project(sub, bem.PREC_FP64, AV=True)
        for c in range(Y1[0].shape[1]):
            a, b = Y[:, :, c0 + c], Y1[:, :, c]
            assert float((a - b).abs().max()) < 1e-13 * float(b.abs().max()), (c0, c)
    ctx.close()


def test_two_parts():
    mesh = synth.cube_sphere(11, (1.0, 0.8, 0.55))
    bem, ctx = _ctx(mesh, "robin", 0)
    lam = np.array([4.0 + 0.1j, 5.6 - 0.02j])
    X = synth.complex_gaussian(mesh.n, 2, 5)
    _, R, _ = ctx.residual_arith(lam, _strided(X, mesh.n), arith=0)
    ctx.close()
    for c in range(2):
        want = oasm.matrix(mesh, lam[c], near=False, op=OPS["robin"]) @ X[:, c]
        assert np.max(np.abs(R[:, c].cpu().numpy() - want)) < 1e-11 * np.max(np.abs(want))


def test_not_finite():
    mesh = synth.cube_sphere(5, (1.0, 0.8, 0.55))
    bem, ctx = _ctx(mesh, "single", 0)
    ctx.set_contour("ellipse", 5.0, 0.8, 0.4, 8)
    V = synth.complex_gaussian(mesh.n, 40, 3)
    V[17, 5] = np.nan
    _, Y = ctx.project(_strided(V, mesh.n), bem.PREC_FP64, AV=True)
    ctx.close()
    bad = torch.isnan(Y).any(dim=1).any(dim=0)
    assert bool(bad[5]) and not bool(bad[:5].any()) and not bool(bad[6:].any())
