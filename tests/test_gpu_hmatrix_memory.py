"""The compressed projection with little memory (bem_set_workspace_limit): what has room for one node
at a time (bem_set_timing takes the nodes so) is not refused because a group of nodes has none,
whichever buffer it is that does not fit, and the results are the same."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _project(bem, mesh, V, near, rmax, limit, single):
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_contour("circle", 5.0, 1.0, 1.0, 8)
    ctx.set_near_field(near)
    ctx.set_hmatrix(leaf=16, rmax=rmax)
    ctx.set_timing(single)
    ctx.set_workspace_limit(limit)
    try:
        B = ctx.project(V, bem.PREC_HMATRIX)
        ctx.check()
        return B
    except bem.BemError as e:
        assert e.status == bem.STATUS_CODES["BEM_ENOMEM"]
        return None
    finally:
        ctx.close()


@pytest.mark.parametrize("nu, near, rmax", [(8, 1, 48), (64, 0, 16), (250, 0, 12)])
def test_group_without_room_runs_node_by_node(nu, near, rmax):
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(14, (1.0, 0.7, 0.5))
    V = bem.fortran(torch.from_numpy(synth.complex_gaussian(mesh.n, nu, 2)).to("cuda:0"))
    ref = _project(bem, mesh, V, near, rmax, 0, False)
    fits = 0
    for k in range(26):
        limit = int((1 << 19) * 1.35 ** k)
        one = _project(bem, mesh, V, near, rmax, limit, True)
        group = _project(bem, mesh, V, near, rmax, limit, False)
        assert (one is None) == (group is None), limit
        if group is not None:
            fits += 1
            assert torch.equal(group, ref) and torch.equal(one, ref)
    assert 0 < fits < 26
