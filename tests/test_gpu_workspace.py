"""Calls whose faster form finds no room for its workspace (bem_set_workspace_limit, a limit kept
on the host): they take the form that needs less, with results inside the same bars, or return
BEM_ENOMEM where there is none. The limits lie below, between and above the sizes that the FP64
projection's two workspaces take here (products 12 MB, V^H Y ~50 MB, expansion ~410 MB). Bars:
1e-11 of the largest entry against the oracle, the FP64 paths' bar throughout."""
import numpy as np
import pytest
import torch

import synth
from oracle import contour as ocon, rr as orr

pytestmark = pytest.mark.gpu
N, NU = 16, 64
Y_BYTES = N * 768 * NU * 16


@pytest.fixture(scope="module")
def problem():
    mesh = synth.cube_sphere(8, (1.0, 0.8, 0.55))
    V = synth.complex_gaussian(mesh.n, NU, 5)
    z, w = ocon.from_spec(synth.ContourSpec("circle", 5.0 + 0j, 0.8, 0.8), N)
    P, Y = orr.project(mesh, z, V)
    return mesh, V, w[:, None, None] * P, np.stack(Y)


def _context(mesh):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_contour("circle", 5.0, 0.8, 0.8, N)
    return bem, ctx


def _err(got, ref):
    return np.max(np.abs(got.cpu().numpy() - ref)) / np.max(np.abs(ref))


@pytest.mark.parametrize("limit", [Y_BYTES - 1, Y_BYTES, 40 << 20, 100 << 20, 400 << 20, 2 << 30, 0])
@pytest.mark.parametrize("av", [False, True])
@pytest.mark.parametrize("held", [0, 30 << 20])
def test_fp64_projection_takes_the_form_that_fits(problem, limit, av, held):
    mesh, V, B, Y = problem
    bem, ctx = _context(mesh)
    Vd = bem.fortran(torch.from_numpy(V).to("cuda:0"))
    if held:   # a buffer that a refused growth gives up
        ctx.set_contour("circle", 5.0, 0.8, 0.8, held // (mesh.n * NU * 16))
        ctx.set_workspace_limit(held)
        ctx.project(Vd, bem.PREC_FP64)
        ctx.set_contour("circle", 5.0, 0.8, 0.8, N)
    ctx.set_workspace_limit(limit)
    if limit == Y_BYTES - 1 and not av and not held:
        with pytest.raises(bem.BemError) as e:
            ctx.project(Vd, bem.PREC_FP64)
        assert e.value.status == bem.STATUS_CODES["BEM_ENOMEM"]
        ctx.set_workspace_limit(0)
    for _ in range(2):   # the buffer as found, then as kept
        out = ctx.project(Vd, bem.PREC_FP64, AV=av)
        ctx.check()
        assert _err(out[0] if av else out, B) < 1e-11
        if av:
            assert _err(out[1], Y) < 1e-11
    ctx.close()


@pytest.mark.parametrize("limit", [1 << 20, 8 << 20, 64 << 20])
def test_cholqr2_and_residual_take_the_form_that_fits(problem, limit):
    mesh, V, B, Y = problem
    bem, ctx = _context(mesh)
    ctx.set_workspace_limit(limit)
    X = bem.fortran(torch.from_numpy(V[:, :8].copy()).to("cuda:0"))
    lam = 5.0 + 0.1 * np.arange(8) + 0.01j
    res, R = ctx.residual_arith(lam, X, arith=0)[:2]
    ctx.set_workspace_limit(0)
    res0, R0 = ctx.residual_arith(lam, X, arith=0)[:2]
    assert _err(R, R0.cpu().numpy()) < 1e-11 and np.allclose(res, res0, rtol=1e-11)
    V0 = bem.fortran(torch.from_numpy(synth.complex_gaussian(4096, 64, 2)).to("cuda:0"))
    Q = V0.clone()
    _, fresh = _context(mesh)
    fresh.set_workspace_limit(limit)
    if limit == 1 << 20:   # less than the partial Gram matrices take in any form
        with pytest.raises(bem.BemError) as e:
            fresh.cholqr2(Q, want_R=False)
        assert e.value.status == bem.STATUS_CODES["BEM_ENOMEM"]
        fresh.set_workspace_limit(0)
    fresh.cholqr2(Q, want_R=False)
    fresh.close()
    eye = torch.eye(64, dtype=Q.dtype, device=Q.device)
    assert float((Q.mH @ Q - eye).abs().max()) < 64 * 2.0 ** -52
    ctx.close()


@pytest.mark.parametrize("near", [0, 1])
def test_recorded_mixed_projections_survive_fp64_calls(near):
    """A recorded batch, or a captured projection with near field, holds the addresses of the
    context's scratch and near-field buffers. Residuals into the caller's buffer and FP64
    projections with AV given need neither: the recording stays valid and its results the same."""
    mesh = synth.cube_sphere(7, (1.0, 0.8, 0.55))
    bem, ctx = _context(mesh)
    ctx.set_near_field(near)
    V = bem.fortran(torch.from_numpy(synth.complex_gaussian(mesh.n, 16, 3)).to("cuda:0"))
    if near:
        B = torch.empty((N, 16, 16), dtype=torch.complex128, device="cuda:0")
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            ctx.project(V, bem.PREC_MIXED, Bhat=B)
            s.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=s):
                ctx.project(V, bem.PREC_MIXED, Bhat=B)

        def run():
            graph.replay()
            torch.cuda.synchronize()
            return [B]
    else:
        batch = bem.Batch([ctx], [V])
        run = batch.run
    first = [b.clone() for b in run()]
    X = bem.fortran(torch.from_numpy(synth.complex_gaussian(mesh.n, 64, 4)).to("cuda:0"))
    ctx.project(X, bem.PREC_FP64, AV=True)
    ctx.residual_arith(5.0 + 0.01 * np.arange(64), X, arith=0)
    again = run()
    torch.cuda.synchronize()
    ctx.check()
    for a, b in zip(first, again):
        assert torch.equal(a, b)
    ctx.close()
