"""CholeskyQR2 on its two sets of kernels: the split products on the tensor core
(csrc/split64.cu, from n nu^2 = 2^23) and the FP64 pipe below, with the FP32 first factor in one
or two diagonal blocks (nu > 128). Sizes around the 16-, 32- and 128-wide tiles and the 64- and
128-row flushes; columns of one sign (the digits' sums at their largest), columns scaled by
1e30 .. 1e35 (a spread of 1e7 or squares beyond FP32's range squared are refused), strided
storage, ill-conditioned bases (the FP64 passes take over) and non-finite or deficient ones
(an error).

Bars: Q^H Q - I and V - Q Q^H V (relative to V's columns) below 64 eps: each entry is a dot product
of unit vectors whose terms carry eps / 2 each, ten times the root of the longest sum's random
error being far below; Q against Householder QR below 1e-13 for a well-conditioned basis."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


def _basis(n, nu, seed, pad=0):
    g = torch.Generator(device="cuda:0").manual_seed(seed)
    buf = torch.zeros((nu, n + pad), dtype=torch.complex128, device="cuda:0")
    buf[:, :n] = torch.randn((nu, n), dtype=torch.complex128, device="cuda:0", generator=g)
    return buf.t()[:n]


def _check(V0, Q, exact=True):
    scale = torch.linalg.vector_norm(V0, dim=0)
    Vn = V0 / scale
    eye = torch.eye(Q.shape[1], dtype=Q.dtype, device=Q.device)
    assert float((Q.mH @ Q - eye).abs().max()) < 64 * EPS
    assert float(torch.linalg.vector_norm(Vn - Q @ (Q.mH @ Vn), dim=0).max()) < 64 * EPS
    if exact:
        H, R = torch.linalg.qr(Vn)
        H = H * torch.sgn(torch.diagonal(R))
        assert float((Q - H).abs().max()) < 1e-13


SIZES = [(4096, 256, 0), (4113, 255, 3), (7000, 200, 0), (16400, 129, 1), (16385, 128, 0),
         (66000, 64, 0), (262144, 32, 0), (300, 130, 2), (1000, 200, 0), (700, 256, 1), (600, 128, 0)]


@pytest.mark.parametrize("n, nu, pad", SIZES)
def test_orthonormal_basis(n, nu, pad):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    V0 = _basis(n, nu, n)
    Q = _basis(n, nu, n, pad)
    ctx.cholqr2(Q, want_R=False)
    _check(V0, Q)
    ctx.close()


@pytest.mark.parametrize("kind", ["one_sign", "scaled", "ill"])
@pytest.mark.parametrize("n, nu", [(8192, 200), (500, 150)])
def test_hard_bases(kind, n, nu):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    V0 = _basis(n, nu, 9)
    k = torch.arange(nu, device=V0.device)
    if kind == "one_sign":      # a large common part: every digit of a column alike
        V0 = V0 + 3.0 * (1.0 + 0.5j) * (k % 2 == 0)
    elif kind == "scaled":
        V0 = V0 * 10.0 ** (30.0 + 5.0 * (k * 37 % nu) / nu)
    else:                       # columns nearly parallel to the first, condition ~1e5
        V0 = V0 * 1e-5 + V0[:, :1]
    Q = V0.clone()   # column-major, as V0
    ctx.cholqr2(Q, want_R=False)
    _check(V0, Q, exact=kind != "ill")
    ctx.close()


@pytest.mark.parametrize("n, nu", [(5000, 256), (400, 140)])
def test_factor_and_errors(n, nu):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    V0 = _basis(n, nu, 4)
    Q = V0.clone()   # column-major, as V0
    R = ctx.cholqr2(Q, want_R=True)
    assert float((V0 - Q @ R).abs().max()) < 64 * EPS * float(torch.linalg.vector_norm(V0, dim=0).max())
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
    Q = V0.clone()   # column-major, as V0          # the context is usable after an error
    ctx.cholqr2(Q, want_R=False)
    _check(V0, Q)
    ctx.close()
