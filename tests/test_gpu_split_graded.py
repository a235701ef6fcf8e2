"""The split products (csrc/split64.cu) on columns whose entries span 14 orders of magnitude. An operand
is cut at 2^-55 of the largest entry of its column (or row), each of a component's two real terms at
both operands, so a sum of K terms is off by up to 2.1 K 2^-53 max|a| max|b| beside its rounding: the
bars below are this bound with the data's own maxima, against binary128 (or 64-bit extended) sums. A
sum of small entries beside a large one that meets zeros has fewer bits than an FP64 sum: only this
bound is promised."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _columns(a):
    t = torch.empty((a.shape[1], a.shape[0]), dtype=torch.complex128, device="cuda:0")
    return t.copy_(torch.from_numpy(np.ascontiguousarray(a.T))).t()


def _graded(n, nu, seed):
    """Gaussian columns, entries times 1 .. 1e-14 in another order in every column."""
    r = np.random.RandomState(seed)
    g = 10.0 ** (-14.0 * np.arange(n) / (n - 1))
    return synth.complex_gaussian(n, nu, seed) * np.stack([r.permutation(g) for _ in range(nu)], 1)


def _amax(a):
    return np.maximum(np.abs(a.real), np.abs(a.imag)).max(0)


@pytest.mark.parametrize("n, nu", [(4096, 64), (1000, 140)])
def test_orthonormal_basis(n, nu):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    V = _graded(n, nu, 3)
    Qd = _columns(V)
    R = ctx.cholqr2(Qd, want_R=True).cpu().numpy()
    ctx.close()
    Q = Qd.cpu().numpy()
    m = _amax(Q)
    bar = (2.1 * n * np.outer(m, m) + 16) * U        # the second pass's Gram matrix
    bar = bar + 2 * 2.1 * nu * U                     # its product, rows of norm at most one
    assert np.all(np.abs(Q.conj().T @ Q - np.eye(nu)) <= bar + 16 * U)
    norm = np.linalg.norm(V, axis=0)
    assert np.all(np.abs(V - Q @ R).max(0) <= (4.2 * nu + 16) * U * norm)


def test_projection():
    """B_j = w_j V^H Y_j from the returned Y_j: n nu^2 N = 2^21."""
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(8, (1.0, 0.8, 0.55))
    V = _graded(mesh.n, 16, 4)
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    z, w = ctx.set_contour("circle", 5.0, 0.8, 0.8, 12)
    B, Y = (t.cpu().numpy() for t in ctx.project(_columns(V), bem.PREC_FP64, AV=True))
    ctx.check()
    ctx.close()
    Vh = V.conj().T.astype(np.clongdouble)
    for j in range(12):
        ref = np.clongdouble(w[j]) * (Vh @ Y[j].astype(np.clongdouble))
        bar = abs(w[j]) * 2 * 2.1 * mesh.n * U * np.outer(_amax(V), _amax(Y[j])) + 8 * U * np.abs(ref)
        assert np.all(np.abs(B[j].astype(np.clongdouble) - ref) <= bar), j


def test_residuals():
    """A(lam) x for graded x, against the oracle's matrix (its sums' own bound beside)."""
    import paper_1906_03938_gb300 as bem
    from oracle import assembly as oasm
    mesh = synth.cube_sphere(10, (1.0, 0.8, 0.55))
    X = _graded(mesh.n, 8, 5)
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    R = ctx.residual_arith(np.full(8, 5.0), _columns(X), arith=0)[1].cpu().numpy()
    ctx.close()
    A = oasm.matrix(mesh, 5.0)
    bar = 2 * 2 * 2.1 * mesh.n * U * np.outer(np.abs(A).max(1), np.abs(X).max(0))
    assert np.all(np.abs(R - A @ X) <= bar)
