"""The expanded FP64 products (csrc/expand64.cu) against the oracle: projections and residuals
over operators, contours (complex centre, flat ellipse, real interval), ragged sizes around
the product tiles' 32 rows, 8 and 32 columns, near field on and off, strided inputs, and
values too far apart for the expansion (the direct form runs). Bar: 1e-11 of the largest
entry, the FP64 paths' bar throughout."""
import numpy as np
import pytest
import torch

import synth
from oracle import assembly as oasm

pytestmark = pytest.mark.gpu
OPS = {"single": (1.0, 0.0), "neumann": (0.0, 1.0), "robin": (0.5 + 0.2j, 1.0 - 0.3j)}
CONTOURS = {"circle": ("circle", 4.0 + 0.3j, 1.0, 1.0, 16), "flat": ("ellipse", 6.5, 1.5, 0.4, 23),
            "wide": ("circle", 3.0, 2.4, 2.4, 64), "interval": ("chebyshev", 5.0, 0.8, 0.8, 12),
            "far": ("circle", 40.0, 35.0, 35.0, 6)}


def _ctx(mesh, op, near):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_operator(*OPS[op])
    ctx.set_near_field(near)
    return bem, ctx


def _strided(a, ld):
    """Column-major copy with leading dimension ld."""
    buf = torch.zeros((a.shape[1], ld), dtype=torch.complex128, device="cuda:0")
    buf[:, :a.shape[0]] = torch.from_numpy(a.T.copy())
    return buf.t()[:a.shape[0]]


def _err(got, ref):
    return np.max(np.abs(got - ref)) / np.max(np.abs(ref))


@pytest.mark.parametrize("op", list(OPS))
@pytest.mark.parametrize("contour", list(CONTOURS))
@pytest.mark.parametrize("m, nu, near, pad", [(1, 1, 0, 0), (2, 9, 1, 5), (3, 33, 0, 1), (4, 8, 1, 0)])
def test_projection(op, contour, m, nu, near, pad):
    mesh = synth.cube_sphere(m, (1.0, 0.8, 0.55))
    bem, ctx = _ctx(mesh, op, near)
    kind, c, a, b, N = CONTOURS[contour]
    z, w = ctx.set_contour(kind, c, a, b, N)
    V = synth.complex_gaussian(mesh.n, nu, 11)
    B, Y = ctx.project(_strided(V, mesh.n + pad), bem.PREC_FP64, AV=True)
    B0 = ctx.project(_strided(V, mesh.n + pad), bem.PREC_FP64)
    ctx.check()
    ctx.close()
    assert torch.equal(B, B0)
    for j in range(N):
        A = oasm.matrix(mesh, z[j], near=bool(near), op=OPS[op])
        assert _err(Y[j].cpu().numpy(), A @ V) < 1e-11, j
        assert _err(B[j].cpu().numpy(), w[j] * (V.conj().T @ (A @ V))) < 1e-11, j


@pytest.mark.parametrize("op", list(OPS))
@pytest.mark.parametrize("m, k, spread, near", [(1, 1, 0.0, 0), (3, 1, 0.0, 1), (3, 8, 0.8, 0),
                                                (4, 9, 0.8, 1), (3, 3, 30.0, 0)])
def test_residuals(op, m, k, spread, near):
    mesh = synth.cube_sphere(m, (1.0, 0.8, 0.55))
    bem, ctx = _ctx(mesh, op, near)
    r = np.random.RandomState(k)
    lam = 35.0 * (spread > 1) + 4.0 + spread * r.uniform(-1, 1, k) + 0.05j * r.uniform(-1, 1, k)
    X = synth.complex_gaussian(mesh.n, k, 5)
    rel, R, Rd = ctx.residual_arith(lam, _strided(X, mesh.n + 3), arith=0, deriv=True)
    rel0 = ctx.residual(lam, _strided(X, mesh.n))
    ctx.close()
    for c in range(k):
        want = oasm.matrix(mesh, lam[c], near=bool(near), op=OPS[op]) @ X[:, c]
        want_d = oasm.matrix(mesh, lam[c], deriv=1, near=bool(near), op=OPS[op]) @ X[:, c]
        assert _err(R[:, c].cpu().numpy(), want) < 1e-11
        assert _err(Rd[:, c].cpu().numpy(), want_d) < 1e-11
        norm = np.linalg.norm(want) / np.linalg.norm(X[:, c])
        assert abs(rel[c] - norm) < 1e-11 * norm and abs(rel0[c] - norm) < 1e-11 * norm


@pytest.mark.parametrize("k", [0.4, 7.0 + 0.5j, 24.0 - 1.0j, 60.0])
def test_self_entries(k):
    """One panel: the residual is the self entry (series below |k| rho = 2, angular sum above)."""
    mesh = synth.cube_grid(4)
    mesh = synth.Mesh("one", mesh.xyz, mesh.tri[:1])
    _, ctx = _ctx(mesh, "single", 0)
    _, R, Rd = ctx.residual_arith([k], _strided(np.ones((1, 1), dtype=complex), 1), arith=0, deriv=True)
    ctx.close()
    for got, d in ((R, 0), (Rd, 1)):
        assert _err(got.cpu().numpy(), oasm.matrix(mesh, k, deriv=d, op=OPS["single"])) < 1e-11
