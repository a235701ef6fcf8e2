"""Nodes of the low-rank far field compressed and applied as a group: bit for bit the result
of one node at a time (which timing every leaf kernel implies), for node counts and basis
widths on both sides of the panel widths, both operator kinds, and a mesh too small for any
far block."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m, nu, N, op", [(8, 5, 1, (1.0, 0.0)), (8, 64, 7, (1.0, 0.0)),
                                          (8, 65, 4, (0.5, 1.0)), (6, 129, 3, (1.0, 0.0)),
                                          (1, 4, 5, (1.0, 0.0))])
def test_group_equals_single_nodes(m, nu, N, op):
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(m, (1.0, 0.7, 0.5))
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_operator(*op)
    ctx.set_contour("circle", 5.0, 1.0, 1.0, N)
    ctx.set_hmatrix(leaf=16)
    V = bem.fortran(torch.from_numpy(synth.complex_gaussian(mesh.n, nu, 2)).to("cuda:0"))
    B, Y = ctx.project(V, bem.PREC_HMATRIX, AV=True)
    stats = ctx.hmatrix_stats()
    ctx.set_timing(True)
    B1, Y1 = ctx.project(V, bem.PREC_HMATRIX, AV=True)
    assert len(ctx.kernel_times()) == N
    assert ctx.hmatrix_stats() == stats
    ctx.check()
    assert torch.equal(B, B1) and torch.equal(Y, Y1)
    ctx.close()
