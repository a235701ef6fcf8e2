"""Panel data for panel counts around the geometry kernel's blocks of 32 panels and the packed
array's rows of 16 (csrc/geometry.cu): mixed and FP64 projections with the near field against the
oracle. Bars: 1e-11 (FP64) and 1e-4 (mixed) of the largest entry, those of the two paths
throughout."""
import numpy as np
import pytest
import torch

import synth
from oracle import assembly as oasm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 64, 65])
def test_panel_counts(n):
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(3, (1.0, 0.8, 0.55))
    mesh = synth.Mesh("part", mesh.xyz, np.ascontiguousarray(mesh.tri[:n]))
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_near_field(1)
    z, _ = ctx.set_contour("circle", 4.0, 0.8, 0.8, 2)
    V = np.eye(n, dtype=complex)
    Vd = torch.from_numpy(V).to("cuda:0")
    _, Y = ctx.project(Vd.t(), bem.PREC_FP64, AV=True)
    _, Z = ctx.project(Vd.t(), bem.PREC_MIXED, AV=True)
    ctx.check()
    ctx.close()
    for j in range(2):
        want = oasm.matrix(mesh, z[j], near=True, op=(1.0, 0.0))
        top = np.max(np.abs(want))
        assert np.max(np.abs(Y[j].cpu().numpy() - want)) < 1e-11 * top
        assert np.max(np.abs(Z[j].cpu().numpy() - want)) < 1e-4 * top
