"""The FP64 expansion (csrc/expand64.cu) and the mesh's reach R, which scales its fixed-point phases.

A vertex that no panel has changes nothing, to the bit. For two bodies far apart the rows of the
first, with a vector that vanishes on the second, are those of the first alone. Bar: 64 eps of the
largest entry: an entry carries a few eps from its phase (k r <= 25) and root, the sums of 80 terms
that many halves of eps in the worst case."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


def _columns(a):
    t = torch.empty((a.shape[1], a.shape[0]), dtype=torch.complex128, device="cuda:0")
    return t.copy_(torch.from_numpy(np.ascontiguousarray(a.T))).t()


def _context(xyz, tri):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    ctx.set_mesh(xyz, tri)
    return bem, ctx


@pytest.mark.parametrize("m", [1, 8])
@pytest.mark.parametrize("where", [1e2, 1e6, 1e12])
def test_vertex_without_panels(m, where):
    mesh = synth.icosphere(2)
    lam = 9.0 + 0.1 * np.arange(m)
    X, V = (_columns(synth.complex_gaussian(mesh.n, k, k)) for k in (m, 12))
    out = []
    for xyz in (mesh.xyz, np.concatenate([mesh.xyz, [[where, -where, 0.0]]])):
        bem, ctx = _context(xyz, mesh.tri)
        ctx.set_contour("circle", 9.0, 0.8, 0.8, 16)
        out.append(ctx.residual_arith(lam, X, arith=0, deriv=True)[1:] +
                   ctx.project(V, bem.PREC_FP64, AV=True))
        ctx.check()
        ctx.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("m", [1, 8])
@pytest.mark.parametrize("apart", [5.0, 1e3, 1e4, 1e6])
def test_two_bodies(m, apart):
    mesh = synth.icosphere(1)
    n = mesh.n
    X = synth.complex_gaussian(n, m, 1)
    out = []
    for bodies in (1, 2):
        xyz = np.concatenate([mesh.xyz + [apart * b, 0.0, 0.0] for b in range(bodies)])
        tri = np.concatenate([mesh.tri + len(mesh.xyz) * b for b in range(bodies)])
        bem, ctx = _context(xyz, tri)
        Xb = _columns(np.concatenate([X] + [np.zeros_like(X)] * (bodies - 1)))
        R, Rd = ctx.residual_arith(np.full(m, 9.0), Xb, arith=0, deriv=True)[1:]
        out.append((R[:n], Rd[:n]))
        ctx.close()
    for a, b in zip(*out):
        assert float((a - b).abs().max()) < 64 * EPS * float(a.abs().max())
