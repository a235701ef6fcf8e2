"""The sparse product of the near corrections (csrc/near.cu, near_spmm32_kernel) at the edges of
its 8-row blocks, of its groups of 4 (or, above 128 columns, 2) nodes and of its 32-wide column
groups: mixed projections with the near field against FP64 ones, column by column.
Bar: 1e-4 of the largest entry, the mixed path's bar throughout."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m, nu, N", [(1, 5, 2), (2, 31, 5), (3, 33, 4), (4, 65, 3), (5, 129, 7), (5, 256, 6)])
def test_against_fp64(m, nu, N):
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(m, (1.0, 0.8, 0.55))
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_near_field(1)
    ctx.set_contour("circle", 4.0, 0.8, 0.8, N)
    V = torch.from_numpy(synth.complex_gaussian(mesh.n, nu, 7).T.copy()).to("cuda:0").t()
    _, Y = ctx.project(V, bem.PREC_MIXED, AV=True)
    _, Z = ctx.project(V, bem.PREC_FP64, AV=True)
    ctx.close()
    for j in range(N):
        assert float((Y[j] - Z[j]).abs().max()) < 1e-4 * float(Z[j].abs().max()), j
