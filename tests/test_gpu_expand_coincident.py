"""A panel given twice, whose centroid is one of its twin's quadrature points to the last bit (vertices
of small whole numbers: 3 fl(1/3) = 1). The single layer is infinite there and its k-derivative is not:
the expansion has non-finite values where the direct form has them and the direct form's elsewhere
(1e-11 of the largest entry, the FP64 paths' bar)."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [4, 11])   # 194 panels: FP64 products; 1454: split products
@pytest.mark.parametrize("op", [(1.0, 0.0), (0.0, 1.0), (0.7 + 0.2j, 1.0)])
def test_derivative_at_coinciding_points(m, op):
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(m, (1.0, 0.8, 0.55))
    xyz = np.concatenate([mesh.xyz, [[0.0, 0.0, 0.0], [3.0, 0.0, 0.0], [0.0, 3.0, 0.0]]])
    twin = np.array([[0, 1, 2]] * 2, dtype=mesh.tri.dtype) + len(mesh.xyz)
    tri = np.concatenate([mesh.tri, twin])
    X = bem.fortran(torch.from_numpy(synth.complex_gaussian(len(tri), 8, 6)).to("cuda:0"))
    lam = 5.0 + 0.05 * np.arange(8) + 0.01j
    out = []
    for limit in (0, 1 << 20):   # expanded, direct
        ctx = bem.Context(0)
        ctx.set_mesh(xyz, tri)
        ctx.set_operator(*op)
        ctx.set_workspace_limit(limit)
        launches = ctx.launches
        _, R, Rd = ctx.residual_arith(lam, X, arith=0, deriv=True)
        out.append((R.cpu().numpy(), Rd.cpu().numpy(), ctx.launches - launches))
        ctx.close()
    assert out[0][2] != out[1][2]   # two different forms
    for got, ref in zip(out[0][:2], out[1][:2]):
        ok = np.isfinite(ref)
        assert np.array_equal(np.isfinite(got), ok)
        assert np.max(np.abs(got[ok] - ref[ok])) < 1e-11 * np.max(np.abs(ref[ok]))
    finite = [np.isfinite(a[-2:]).any() for a in out[1][:2]]
    assert finite == [False, op[1] == 0]
