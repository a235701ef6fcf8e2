"""The bounded waits of the FP64 products on the tensor core (csrc/split64.cu). With no poll allowed
every wait gives up at once; with a few, some give up while copies and tensor-core products are in
flight, which the blocks let land (those waits keep their full bound) before they leave. The calls
report BEM_ETIMEOUT and the context stays usable."""
import numpy as np
import pytest
import torch

import synth
from oracle import contour as ocon, rr as orr

pytestmark = pytest.mark.gpu
N, NU = 16, 64


def _timed_out(bem, call, certain):
    try:
        call()
    except bem.BemError as e:
        assert e.status == bem.STATUS_CODES["BEM_ETIMEOUT"], str(e)
        assert "wait-timeout" in str(e)
    else:
        assert not certain


@pytest.mark.parametrize("polls", [0, 1, 8])
def test_fp64_projection(polls):
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(8, (1.0, 0.8, 0.55))
    V = synth.complex_gaussian(mesh.n, NU, 5)
    Vd = bem.fortran(torch.from_numpy(V).to("cuda:0"))
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    z, w = ctx.set_contour("circle", 5.0, 0.8, 0.8, N)
    ctx.set_wait_limit(polls)

    def project():
        ctx.project(Vd, bem.PREC_FP64)
        ctx.check()

    for _ in range(3):
        _timed_out(bem, project, polls == 0)
    ctx.set_wait_limit(1 << 24)
    B = ctx.project(Vd, bem.PREC_FP64).cpu().numpy()
    ctx.check()
    ctx.close()
    ref = w[:, None, None] * orr.project(mesh, z, V)[0]
    assert np.max(np.abs(B - ref)) < 1e-11 * np.max(np.abs(ref))   # the FP64 paths' bar


@pytest.mark.parametrize("polls", [0, 1, 8])
@pytest.mark.parametrize("n, nu", [(4096, 64), (16385, 129)])
@pytest.mark.parametrize("want_R", [False, True])
def test_cholqr2(polls, n, nu, want_R):
    import paper_1906_03938_gb300 as bem
    g = torch.Generator(device="cuda:0").manual_seed(n)
    V0 = torch.randn((nu, n), dtype=torch.complex128, device="cuda:0", generator=g).t()
    ctx = bem.Context(0)
    ctx.set_wait_limit(polls)
    for _ in range(3):
        Q = V0.clone()
        _timed_out(bem, lambda: ctx.cholqr2(Q, want_R=want_R), polls == 0)
    ctx.set_wait_limit(1 << 24)
    Q = V0.clone()
    ctx.cholqr2(Q, want_R=want_R)
    ctx.close()
    eye = torch.eye(nu, dtype=Q.dtype, device=Q.device)
    assert float((Q.mH @ Q - eye).abs().max()) < 64 * 2.0 ** -52   # as tests/test_gpu_split64.py


@pytest.mark.parametrize("polls", [0, 1, 8])
@pytest.mark.parametrize("deriv", [False, True])
def test_residual(polls, deriv):
    """1200 panels, 8 vectors: the expansion's products are split ones (n^2 S 28 > 1.5e7)."""
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(10, (1.0, 0.8, 0.55))
    X = bem.fortran(torch.from_numpy(synth.complex_gaussian(mesh.n, 8, 6)).to("cuda:0"))
    lam = 5.0 + 0.1 * np.arange(8) + 0.01j
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ref = ctx.residual_arith(lam, X, arith=0, deriv=deriv)[0]
    ctx.set_wait_limit(polls)
    for _ in range(3):
        _timed_out(bem, lambda: ctx.residual_arith(lam, X, arith=0, deriv=deriv), polls == 0)
    ctx.check()   # the timeout was this call's to report: nothing is left of it
    ctx.set_wait_limit(1 << 24)
    assert np.array_equal(ctx.residual_arith(lam, X, arith=0, deriv=deriv)[0], ref)
    ctx.close()


@pytest.mark.parametrize("m, arith", [(1, 1), (1, 0)])
def test_residual_without_waits_leaves_other_calls_timeouts(m, arith):
    """108 panels and one vector: no split products. The timeout that a projection
    recorded is the check's to report, not the residual's."""
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(3, (1.0, 0.8, 0.55))
    X = bem.fortran(torch.from_numpy(synth.complex_gaussian(mesh.n, 16, 6)).to("cuda:0"))
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_contour("circle", 5.0, 0.8, 0.8, N)
    ref = ctx.residual_arith([5.0], X[:, :m], arith=arith)[0]
    ctx.set_wait_limit(0)
    ctx.project(X, bem.PREC_MIXED)
    ctx.set_wait_limit(1 << 24)
    assert np.array_equal(ctx.residual_arith([5.0], X[:, :m], arith=arith)[0], ref)
    with pytest.raises(bem.BemError) as e:
        ctx.check()
    assert e.value.status == bem.STATUS_CODES["BEM_ETIMEOUT"]
    ctx.check()
    ctx.close()
