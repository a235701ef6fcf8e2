"""The near-pair scan (csrc/near.cu) against the criterion evaluated in NumPy with the same
step-by-step rounding: the pair lists are equal, element by element. Sizes at the edges of a
block's 32 rows and the 256 staged columns; a mesh far from the origin, where FP32
coordinates decide few pairs and the exact test decides the rest."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _pairs(xyz, tri):
    v = xyz[tri]
    c = (v[:, 0] + v[:, 1] + v[:, 2]) / 3.0
    norm = lambda d: np.sqrt((d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2])
    h = np.maximum(np.maximum(norm(v[:, 1] - v[:, 0]), norm(v[:, 2] - v[:, 0])), norm(v[:, 2] - v[:, 1]))
    near = norm(c[:, None] - c[None, :]) < 2.0 * np.maximum(h[:, None], h[None, :])
    np.fill_diagonal(near, False)
    return near


@pytest.mark.parametrize("n", [1, 12, 31, 32, 33, 255, 256, 257, 300])
@pytest.mark.parametrize("shift", [0.0, 3.0e4])
def test_pairs_equal_the_criterion(n, shift):
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(5, (1.0, 0.8, 0.55))
    xyz, tri = mesh.xyz + shift, mesh.tri[:n]
    ctx = bem.Context(0)
    ctx.set_mesh(xyz, tri)
    ctx.set_near_field(1)
    ptr, cols = ctx.near_pairs()
    ctx.close()
    ref = _pairs(xyz, tri)
    assert np.array_equal(ptr, np.concatenate([[0], np.cumsum(ref.sum(1))]))
    assert np.array_equal(cols, np.nonzero(ref)[1])
