"""FP64 products at wavenumbers far from the real axis (csrc/expand64.cu): the entries of A(k) grow by
e^{|Im k| R} over the mesh, and with them the coefficients of the expansion over the wavenumbers,
whose rounding then shows in the near entries. Bar: 64 eps of (|A| |x|)_i, component by component, for
vectors of four neighbouring panels: an entry carries a few eps from its phase (k r <= 15) and root in
either code, a sum of four terms two more. Contours inside the expansion's range, at its end and
beyond, where the direct form runs."""
import numpy as np
import pytest
import torch

import synth
from oracle import assembly as oasm

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


def _columns(a):
    t = torch.empty((a.shape[1], a.shape[0]), dtype=torch.complex128, device="cuda:0")
    return t.copy_(torch.from_numpy(np.ascontiguousarray(a.T))).t()


@pytest.mark.parametrize("op", [(1.0, 0.0), (0.5 + 0.2j, 1.0 - 0.3j)])
@pytest.mark.parametrize("radius", [0.8, 2.0, 2.1, 2.8, 3.4])
def test_local_vectors(op, radius):
    import paper_1906_03938_gb300 as bem
    mesh = synth.icosphere(1)
    r = np.random.RandomState(0)
    c = mesh.xyz[mesh.tri].mean(1)
    V = np.zeros((mesh.n, 12), complex)
    for k in range(12):
        V[np.argsort(np.linalg.norm(c - c[6 * k], axis=1))[:4], k] = r.randn(4) + 1j * r.randn(4)
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_operator(*op)
    z, w = ctx.set_contour("circle", 4.0, radius, radius, 16)
    Y = ctx.project(_columns(V), bem.PREC_FP64, AV=True)[1].cpu().numpy()
    R = ctx.residual_arith(z[:12], _columns(V), arith=0)[1].cpu().numpy()
    ctx.check()
    ctx.close()
    for j in range(16):
        A = oasm.matrix(mesh, z[j], op=op)
        bar = 64 * EPS * (np.abs(A) @ np.abs(V))
        assert np.all(np.abs(Y[j] - A @ V) <= bar), j
        if j < 12:
            assert np.all(np.abs(R[:, j] - A @ V[:, j]) <= bar[:, j]), j
