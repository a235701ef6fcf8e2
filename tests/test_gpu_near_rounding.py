"""The near-field corrections in the FP64 expansion (csrc/near.cu) on a contour that reaches far below the
real axis, where the coefficients of the slots' products grow to e^{a R / 2} of the result (a = 1.6,
R = 2): with and without the near field the far products are the same numbers, so their difference is
the corrections' sum C V and what its addition rounds. C V is formed in binary128 (or 64-bit extended).
Bar: e^{a R / 2} units of 2^-53 of ||Y||: each slot's product takes the corrections by one addition,
0.4 units rms. Corrections added one by one cost 3 times the bar."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _gauss8():
    x = np.polynomial.legendre.leggauss(8)[0].astype(LD)
    for _ in range(5):
        p0, p1 = np.ones_like(x), x
        for k in range(2, 9):
            p0, p1 = p1, ((2 * k - 1) * x * p1 - (k - 1) * p0) / k
        dp = 8 * (x * p1 - p0) / (x * x - 1)
        x = x - p1 / dp
    return (x + 1) / 2, 1 / ((1 - x * x) * dp * dp)


def _corrections(mesh, ptr, cols, k):
    """(A_near - A_7) of every pair at wavenumber k."""
    pi = LD(4) * np.arctan(LD(1))
    v = mesh.xyz.astype(LD)[mesh.tri]
    c = np.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    area = np.sqrt((c * c).sum(1)) / 2
    i = np.repeat(np.arange(mesh.n), np.diff(ptr))
    x, t, ar = v.mean(1)[i], v[cols], area[cols]
    at = np.argmin(((t - x[:, None]) ** 2).sum(-1).astype(float), 1)
    e = np.arange(len(i))
    a, b, d = t[e, at], t[e, (at + 1) % 3], t[e, (at + 2) % 3]
    g, w = _gauss8()
    s = np.repeat(g, 8)
    y = a[:, None] + s[:, None] * (b - a)[:, None] + (s * np.tile(g, 8))[:, None] * (d - b)[:, None]
    wn = (np.repeat(w, 8) * np.tile(w, 8) * s)[None] * 2 * ar[:, None]
    r15 = np.sqrt(LD(15))
    bary, w7 = [(LD(1) / 3,) * 3], [LD(9) / 40]
    for al, ww in (((6 - r15) / 21, (155 - r15) / 1200), ((6 + r15) / 21, (155 + r15) / 1200)):
        for p in ((al, al, 1 - 2 * al), (al, 1 - 2 * al, al), (1 - 2 * al, al, al)):
            bary.append(p)
            w7.append(ww)
    y = np.concatenate([y, np.stack([sum(p[m] * t[:, m] for m in range(3)) for p in bary], 1)], 1)
    wn = np.concatenate([wn, -np.stack([ww * ar for ww in w7], 1)], 1) / (4 * pi)
    r = np.sqrt(((y - x[:, None]) ** 2).sum(-1))
    kr, ki = LD(k.real), LD(k.imag)
    f = wn / r * np.exp(-ki * r)
    return i, (f * np.cos(kr * r)).sum(1) + 1j * (f * np.sin(kr * r)).sum(1)


def test_corrections_cost_one_rounding():
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(5, (1.0, 0.7, 0.5))
    V = synth.complex_gaussian(mesh.n, 20, 9)
    Vd = bem.fortran(torch.from_numpy(V).to("cuda:0"))
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    Y = []
    for near in (0, 1):
        ctx.set_near_field(near)
        z, w = ctx.set_contour("circle", 3.0, 1.6, 1.6, 8)
        Y.append(ctx.project(Vd, bem.PREC_FP64, AV=True)[1].cpu().numpy().astype(np.clongdouble))
    ptr, cols = ctx.near_pairs()
    ctx.close()
    for j in (0, 3, 5, 6):
        i, C = _corrections(mesh, ptr, cols, complex(z[j]))
        CV = np.zeros((mesh.n, 20), np.clongdouble)
        np.add.at(CV, i, C[:, None] * V[cols])
        err = np.linalg.norm((Y[1][j] - Y[0][j] - CV).astype(complex)) / np.linalg.norm(Y[1][j].astype(complex))
        assert err < np.exp(1.6) * 2.0 ** -53, j
