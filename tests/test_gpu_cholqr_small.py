"""CholeskyQR2 of narrow bases (nu <= 64), whose factors are formed by one cluster each
(csrc/cholqr.cu, cq_factor_kernel), at the edges of the 32-wide tiles and of its eight blocks'
rows, on each of its routes: columns close to the first (distance d, condition ~1/d) take the
FP32 first pass with one second-order step, with two, and the FP64 passes alone.

Bars as for the wide bases: Q^H Q - I and V - Q Q^H V (relative to V's columns) below 64 eps."""
import pytest
import torch

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


def _basis(n, nu, distance):
    g = torch.Generator(device="cuda:0").manual_seed(17 * n + nu)
    V = torch.randn((nu, n), dtype=torch.complex128, device="cuda:0", generator=g).t()
    V[:, 1:] = V[:, 1:] * distance + V[:, :1] * (0.0 if distance == 1.0 else 1.0)
    return V


def _check(V0, Q):
    Vn = V0 / torch.linalg.vector_norm(V0, dim=0)
    eye = torch.eye(Q.shape[1], dtype=Q.dtype, device=Q.device)
    assert float((Q.mH @ Q - eye).abs().max()) < 64 * EPS
    assert float(torch.linalg.vector_norm(Vn - Q @ (Q.mH @ Vn), dim=0).max()) < 64 * EPS


@pytest.mark.parametrize("distance", [1.0, 1e-1, 1e-2, 1e-3, 1e-5])
@pytest.mark.parametrize("n, nu", [(1, 1), (2, 1), (9, 2), (320, 16), (65, 31), (131, 32), (140, 33),
                                   (1452, 47), (200, 64), (4097, 64), (20000, 40)])
def test_routes(n, nu, distance):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    V0 = _basis(n, nu, distance)
    Q = V0.clone()
    ctx.cholqr2(Q, want_R=False)
    _check(V0, Q)
    ctx.close()


@pytest.mark.parametrize("n, nu", [(100, 20), (300, 64)])
def test_refused(n, nu):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    V0 = _basis(n, nu, 1.0)
    for bad in ("nan", "zero", "equal"):
        W = V0.clone()
        if bad == "nan":
            W[n // 3, nu // 2] = float("nan")
        elif bad == "zero":
            W[:, nu // 2] = 0.0
        else:
            W[:, nu // 2] = W[:, 0]
        with pytest.raises(bem.BemError):
            ctx.cholqr2(W, want_R=False)
    Q = V0.clone()
    ctx.cholqr2(Q, want_R=False)
    _check(V0, Q)
    ctx.close()
