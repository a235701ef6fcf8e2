"""bem_residual_arith with arith 1 on both of its routes (csrc/residual.cu, expand_beats_ff):
the double-FP32 kernel for few columns or values too far apart, the shared FP64 evaluation for many
columns or near fields; against arith 0 one column at a time. Bar: 1e-11 of the largest component,
the double-FP32 residual's bar throughout."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
OPS = {"single": (1.0, 0.0), "robin": (0.5 + 0.2j, 1.0 - 0.3j)}


@pytest.mark.parametrize("op, m, k, spread, near, deriv", [
    ("single", 5, 12, 0.8, 1, False), ("single", 5, 12, 0.8, 1, True), ("single", 8, 24, 0.8, 0, False),
    ("single", 8, 2, 0.8, 0, False), ("single", 3, 1, 0.0, 1, False), ("single", 6, 9, 25.0, 1, False),
    ("robin", 5, 7, 0.8, 1, True), ("robin", 5, 7, 0.8, 0, False)])
def test_arith1(op, m, k, spread, near, deriv):
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(m, (1.0, 0.8, 0.55))
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_operator(*OPS[op])
    ctx.set_near_field(near)
    r = np.random.RandomState(k)
    lam = max(5.0, 1.1 * spread) + spread * r.uniform(-1, 1, k) + 0.01j * r.uniform(-1, 1, k)
    X = torch.from_numpy(synth.complex_gaussian(mesh.n, k, 5).T.copy()).to("cuda:0").t()
    rel, R, Rd = ctx.residual_arith(lam, X, arith=1, deriv=deriv)
    for c in range(k):
        rel0, R0, Rd0 = ctx.residual_arith(lam[c:c + 1], X[:, c:c + 1].t().contiguous().t(), arith=0,
                                           deriv=deriv)
        assert float((R[:, c] - R0[:, 0]).abs().max()) < 1e-11 * float(R0.abs().max())
        assert abs(rel[c] - rel0[0]) < 1e-10 * rel0[0]
        if deriv:
            assert float((Rd[:, c] - Rd0[:, 0]).abs().max()) < 1e-11 * float(Rd0.abs().max())
    ctx.close()
