"""The FP64 self entries (csrc/selfterm.cuh) on both sides of |k| rho = 2, where the series over the
moments gives way to the sum over the angular nodes, and with both kinds among the wavenumbers of one
call: against the oracle's self integral, 64 eps of the entry (96 terms of one sign at k = 0, whose
sum carries some eps in either code). The k-derivative against the oracle by a six-point difference
of step h = 1e-2 / k: its error is below (k rho h / k)^6 / 140 of the entry over h, ~1e-12, and the
rounding 1e-15 / h ~ 1e-12 of it; bar 1e-10 of |A| / h's scale, rho |A|."""
import numpy as np
import pytest
import torch

import synth
from oracle import assembly as oasm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op", [(1.0, 0.0), (0.5 + 0.2j, 1.0 - 0.3j)])
@pytest.mark.parametrize("ks", [(0.5, 2.0), (2.0, 12.0), (8.0, 60.0), (3.0, 3.0)])
def test_self_entries(op, ks):
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(2, (1.0, 0.8, 0.2))
    n = mesh.n
    lam = np.linspace(*ks, n) * np.exp(0.05j * np.sin(np.arange(n)))
    ctx = bem.Context(0)
    ctx.set_mesh(mesh.xyz, mesh.tri)
    ctx.set_operator(*op)
    X = torch.eye(n, dtype=torch.complex128, device="cuda:0").t()
    _, R, Rd = ctx.residual_arith(lam, X, arith=0, deriv=True)
    ctx.close()
    got, dgot = torch.diagonal(R).cpu().numpy(), torch.diagonal(Rd).cpu().numpy()
    v = mesh.xyz[mesh.tri]
    rho = np.linalg.norm(v - v.mean(1, keepdims=True), axis=2).max(1)
    diag = lambda k, l: oasm.matrix(mesh, k, op=op)[l, l]
    for l in range(0, n, 5):
        ref = diag(lam[l], l)
        assert abs(got[l] - ref) <= 64 * 2.0 ** -52 * abs(ref), l
        h = 1e-2 / max(1.0, abs(lam[l]))
        d = sum(c * (diag(lam[l] + s * h, l) - diag(lam[l] - s * h, l))
                for s, c in ((1, 3 / 4), (2, -3 / 20), (3, 1 / 60))) / h
        assert abs(dgot[l] - d) <= 1e-10 * abs(ref) * max(rho[l], 1.0), l
