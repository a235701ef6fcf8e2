"""The near-pair scan (csrc/near.cu) on meshes of every scale: the criterion is scale-invariant and a
power of two changes no rounding in FP64, so the pairs are those of the mesh of size one. Beyond
1e19 and below 1e-22 the squared distances leave FP32's range and the exact test decides. (Below
~2^-270 a mesh is refused: its areas vanish in FP64.)"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _pairs(xyz, tri):
    import paper_1906_03938_gb300 as bem
    ctx = bem.Context(0)
    ctx.set_mesh(xyz, tri)
    ctx.set_near_field(1)
    out = ctx.near_pairs()
    ctx.close()
    return out


@pytest.mark.parametrize("power", [-200, -130, -110, -80, -70, -60, -50, -40, 40, 55, 60, 62, 63, 64, 66, 80, 120, 200])
def test_pairs_do_not_depend_on_the_scale(power):
    mesh = synth.cube_sphere(5, (1.0, 0.8, 0.55))
    ptr, cols = _pairs(mesh.xyz, mesh.tri)
    assert 0 < len(cols) < mesh.n * (mesh.n - 1)
    p, c = _pairs(mesh.xyz * 2.0 ** power, mesh.tri)
    assert np.array_equal(p, ptr) and np.array_equal(c, cols)
