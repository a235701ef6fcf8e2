"""CholeskyQR2 of bases of condition 3 .. 1000. Wider than 128 columns the FP32 first factor accepts
them but does not leave them orthonormal enough for the near-identity factor: the last pass is a near one
all the same. Q^H Q - I is summed in binary128 (or 64-bit extended). Bar 4 eps: the last pass rounds
the entries of Q once (2.8 units of 2^-53 in an entry of Q^H Q at most), its factor and its Gram matrix
once each (3 units); the digits' cuts are random and a fraction of a unit.
A basis that FP32 refuses, and one with a NaN or a zero column, as before."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


def _basis(n, nu, cond):
    g = torch.Generator(device="cuda:0").manual_seed(n)
    rand = lambda *s: torch.randn(*s, dtype=torch.complex128, device="cuda:0", generator=g)
    U, W = torch.linalg.qr(rand(n, nu))[0], torch.linalg.qr(rand(nu, nu))[0]
    s = torch.logspace(0.0, -np.log10(cond), nu, dtype=torch.float64, device="cuda:0")
    return ((U * s) @ W).t().contiguous().t()


@pytest.mark.parametrize("cond", [10.0, 30.0, 100.0, 1000.0, 1e5])
@pytest.mark.parametrize("n, nu", [(400, 140), (600, 200), (1100, 256)])
def test_orthonormal(n, nu, cond):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    V = _basis(n, nu, cond)
    Q = V.clone()
    ctx.cholqr2(Q, want_R=False)
    ctx.close()
    cols = np.random.RandomState(0).permutation(nu)[:32]   # (all of narrower bases)
    q = Q.cpu().numpy().astype(np.clongdouble)
    err = np.abs(q.conj().T @ q[:, cols] - np.eye(nu)[:, cols])
    assert float(err.max()) <= 4 * EPS
    R = Q.mH @ V
    assert float((V - Q @ R).abs().max()) < 64 * EPS   # ||V|| = 1: the span is V's
    low = R.tril(-1)
    assert float(low.abs().max()) < 64 * EPS           # and R is triangular: Q is V's QR factor


@pytest.mark.parametrize("cond", [3.0, 30.0, 60.0, 100.0, 150.0])
@pytest.mark.parametrize("n, nu", [(40, 5), (300, 17), (500, 32), (500, 33), (1000, 63), (3072, 64)])
def test_both_steps_of_narrow_bases(n, nu, cond):
    """nu <= 64: one cluster forms the near-identity factor; for 1e-5 < ||G - I|| <= 5e-4 in two steps."""
    test_orthonormal(n, nu, cond)


@pytest.mark.parametrize("n, nu", [(400, 140), (1100, 256)])
def test_refused(n, nu):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    V = _basis(n, nu, 100.0)
    for kind in ("nan", "zero", "equal"):
        W = V.clone()
        if kind == "nan":
            W[n // 2, nu - 1] = float("nan")
        elif kind == "zero":
            W[:, nu - 1] = 0.0
        else:
            W[:, nu - 1] = W[:, 0]
        with pytest.raises(bem.BemError):
            ctx.cholqr2(W, want_R=False)
    ctx.close()
