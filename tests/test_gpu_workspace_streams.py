"""The FP64 forms' workspace between calls that shared nothing before they had one: a captured
projection replays after calls that need a larger workspace, and calls on two streams that are not
ordered by the caller take turns. Results are compared bit for bit with those of calls one by one."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _context():
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(8, (1.0, 0.8, 0.55))
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_contour("circle", 5.0, 0.8, 0.8, 16)
    return bem, ctx, mesh.n


def _basis(bem, n, nu, seed):
    return bem.fortran(torch.from_numpy(synth.complex_gaussian(n, nu, seed)).to("cuda:0"))


@pytest.mark.parametrize("near", [0, 1])
@pytest.mark.parametrize("av", [False, True])
def test_captured_projection_outlives_larger_workspaces(near, av):
    bem, ctx, n = _context()
    ctx.set_near_field(near)
    V = _basis(bem, n, 32, 1)
    B = torch.empty((16, 32, 32), dtype=torch.complex128, device="cuda:0")
    Y = torch.empty((16, 32, n), dtype=torch.complex128, device="cuda:0") if av else False
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        ctx.project(V, bem.PREC_FP64, Bhat=B, AV=Y)
        s.synchronize()
        expected = [B.clone()] + ([Y.clone()] if av else [])
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            ctx.project(V, bem.PREC_FP64, Bhat=B, AV=Y)
    big = _basis(bem, n, 128, 2)
    lam = 5.0 + 0.01 * np.arange(128)
    for _ in range(2):
        ctx.project(big, bem.PREC_FP64, AV=True)
        ctx.residual_arith(lam, big, arith=0)
        B.zero_()
        graph.replay()
        torch.cuda.synchronize()
        ctx.check()
        assert all(torch.equal(a, b) for a, b in zip(expected, [B, Y]))
    ctx.close()


def test_captured_cholqr2_outlives_larger_workspaces():
    """Split products at both sizes (n nu^2 > 2^23). The room for partial Gram matrices is that of the
    longest basis whatever n."""
    bem, ctx, _ = _context()
    ctx.set_async(True)
    V = _basis(bem, 3072, 64, 1)
    Q = V.clone()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        ctx.cholqr2(Q, want_R=False)
        s.synchronize()
        expected = Q.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            ctx.cholqr2(Q, want_R=False)
    for _ in range(2):
        big = _basis(bem, 32768, 64, 2)
        ctx.cholqr2(big, want_R=False)
        Q.copy_(V)
        graph.replay()
        torch.cuda.synchronize()
        ctx.check()
        assert torch.equal(Q, expected)
    ctx.close()


def test_calls_on_two_streams():
    bem, ctx, n = _context()
    Vs = [_basis(bem, n, nu, 3 + nu) for nu in (48, 64)]
    lam = 5.0 + 0.1 * np.arange(48) + 0.01j
    alone = [[t.clone() for t in ctx.project(V, bem.PREC_FP64, AV=True)] for V in Vs]
    _, R0, _ = ctx.residual_arith(lam, Vs[0], arith=0)
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(3):
        with torch.cuda.stream(a):
            first = ctx.project(Vs[0], bem.PREC_FP64, AV=True)
        with torch.cuda.stream(b):
            second = ctx.project(Vs[1], bem.PREC_FP64, AV=True)
        with torch.cuda.stream(a):
            _, R, _ = ctx.residual_arith(lam, Vs[0], arith=0)
        torch.cuda.synchronize()
        ctx.check()
        assert torch.equal(R, R0)
        for got, want in zip([first, second], alone):
            assert all(torch.equal(x, y) for x, y in zip(got, want))
    ctx.close()
