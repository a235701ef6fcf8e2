"""FP64 products by the expansion (csrc/expand64.cu) against binary128 (or 64-bit extended) entries, for
the single layer, the double layer alone and Robin's combination: the error of ||A X|| is no larger than
the direct forms leave on the same inputs, which run where the workspace limit leaves the expansion no
room. Both errors are root mean squares over the nodes and 8 vectors of 192 entries, sums of some 1e5
roundings; 3 % for their chance."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
LD = np.longdouble
OPS = {"single": (1.0, 0.0), "neumann": (0.0, 1.0), "robin": (0.5 + 0.2j, 1.0 - 0.3j)}


class Exact:
    """Off-diagonal entries by the 7-point rule; the diagonal is taken from the code under test (a
    closed form of its own, see test_gpu_self_term)."""

    def __init__(self, mesh, op):
        self.cg, self.ch = (np.clongdouble(c) for c in op)
        v = mesh.xyz.astype(LD)[mesh.tri]
        n = np.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
        two = np.sqrt((n * n).sum(1))
        r15 = np.sqrt(LD(15))
        bary, w = [(LD(1) / 3,) * 3], [LD(9) / 40]
        for a, ww in (((6 - r15) / 21, (155 - r15) / 1200), ((6 + r15) / 21, (155 + r15) / 1200)):
            for p in ((a, a, 1 - 2 * a), (a, 1 - 2 * a, a), (1 - 2 * a, a, a)):
                bary.append(p)
                w.append(ww)
        y = np.stack([sum(p[m] * v[:, m] for m in range(3)) for p in bary], 1)
        d = y[None] - v.mean(1)[:, None, None]
        r = np.sqrt((d * d).sum(-1))
        e = np.arange(mesh.n)
        r[e, e] = 1
        wr = np.stack([ww * two / 2 for ww in w], 1)[None] / (16 * np.arctan(LD(1))) / r
        wr[e, e] = 0
        self.r, self.g, self.h = r, wr, wr * (d * (n / two[:, None])[None, :, None]).sum(-1) / r ** 2

    def matrix(self, k):
        kr, ki = LD(complex(k).real), LD(complex(k).imag)
        ph = np.exp(-ki * self.r) * (np.cos(kr * self.r) + 1j * np.sin(kr * self.r))
        f = self.cg * self.g + self.ch * self.h * (1j * (kr + 1j * ki) * self.r - 1)
        return (f * ph).sum(-1)


def _columns(a):
    t = torch.empty((a.shape[1], a.shape[0]), dtype=torch.complex128, device="cuda:0")
    return t.copy_(torch.from_numpy(np.ascontiguousarray(a.T))).t()


def _err(got, ref):
    return float(np.linalg.norm((got - ref).astype(complex)) / np.linalg.norm(ref.astype(complex)))


@pytest.mark.parametrize("op", list(OPS))
@pytest.mark.parametrize("k", [4.0, 8.0])
def test_no_further_off_than_the_direct_forms(op, k):
    import paper_1906_03938_gb300 as bem
    mesh = synth.cube_sphere(4, (1.0, 0.7, 0.5))
    n = mesh.n
    X = synth.complex_gaussian(n, 8, 3)
    lam = k + np.array([0.005j, -0.005j] * 4)
    eye = _columns(np.eye(n))
    exact = Exact(mesh, OPS[op])
    nodes, AX, off = (1, 3, 6), {}, []
    for limit in (0, 4096):
        ctx = bem.Context(0)
        ctx.set_workspace_limit(limit)
        ctx.set_mesh(mesh.xyz, mesh.tri)
        ctx.set_operator(*OPS[op])
        z, w = ctx.set_contour("circle", k, 0.9, 0.9, 8)
        if not AX:
            for q in [z[j] for j in nodes] + list(lam[:2]):
                d = torch.diagonal(ctx.residual_arith(np.full(n, q), eye, arith=0)[1]).cpu().numpy()
                AX[q] = (exact.matrix(q) + np.diag(d.astype(np.clongdouble))) @ X.astype(np.clongdouble)
        before = ctx.launches
        Y = ctx.project(_columns(X), bem.PREC_FP64, AV=True)[1].cpu().numpy()
        R = ctx.residual_arith(lam, _columns(X), arith=0)[1].cpu().numpy()
        off.append((np.sqrt(np.mean([_err(Y[j], AX[z[j]]) ** 2 for j in nodes])),
                    np.sqrt(np.mean([_err(R[:, c], AX[lam[c]][:, c]) ** 2 for c in range(8)])),
                    ctx.launches - before))
        ctx.close()
    assert off[0][2] > off[1][2]   # the expansion takes more launches: both forms ran
    assert off[0][0] <= 1.03 * off[1][0] and off[0][1] <= 1.03 * off[1][1]
