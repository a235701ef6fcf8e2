"""The fixed-point moments (csrc/expand64.cu) against the oracle where their scales and ranges
change: bodies of very small and very large size (roots outside the FP32 range of the starting
value, weights far from 1), a phase of many turns, a wavenumber below zero, values off the real
axis (a real centre within a term, a complex one beyond). Bar: 1e-11 of the largest entry, the
FP64 paths' bar throughout; at c r turns of phase FP64 itself keeps 2 pi c r 2^-53."""
import numpy as np
import pytest
import torch

import synth
from oracle import assembly as oasm

pytestmark = pytest.mark.gpu
OPS = {"single": (1.0, 0.0), "neumann": (0.0, 1.0), "robin": (0.5 + 0.2j, 1.0 - 0.3j)}


@pytest.mark.parametrize("op", list(OPS))
@pytest.mark.parametrize("scale, k0, im", [(1.0, 5.0, 0.0), (1e-6, 5.0, 0.0), (1e-17, 5.0, 0.0), (1e6, 5.0, 0.0),
                                           (1e17, 5.0, 0.0), (1.0, 900.0, 0.0), (1.0, -6.0, 0.0), (1.0, 0.0, 0.0),
                                           (1.0, 5.0, 1e-3), (1.0, 5.0, 2.0)])
def test_ranges(op, scale, k0, im):
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(3, (1.0, 0.8, 0.55))
    mesh = synth.Mesh("scaled", mesh.xyz * scale, mesh.tri)
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_operator(*OPS[op])
    lam = (np.array([k0 - 0.2, k0, k0 + 0.3]) + 1j * im * np.array([1.0, 1.1, 0.9])) / scale
    X = synth.complex_gaussian(mesh.n, 3, 5)
    _, R, _ = ctx.residual_arith(lam, torch.from_numpy(X.T.copy()).to("cuda:0").t(), arith=0)
    ctx.close()
    for c in range(3):
        want = oasm.matrix(mesh, lam[c], near=False, op=OPS[op]) @ X[:, c]
        assert np.max(np.abs(R[:, c].cpu().numpy() - want)) < 1e-11 * np.max(np.abs(want)), c
