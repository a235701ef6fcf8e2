"""The FP64 complex product (csrc/reduced.cu, zgemm_kernel) through bem_ritz_vectors, X = V Y: sizes
at the edges of its 16 x 16 tiles and 32-deep chunks, and of the split over k (few tiles, k from 128).
Bar: 8 k eps of |V| |Y| entrywise (k products of two complex numbers, each sum in any order)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, nu, k", [(1, 1, 1), (16, 15, 17), (17, 16, 16), (33, 31, 5), (40, 32, 33),
                                      (130, 127, 2), (128, 128, 3), (257, 200, 48), (3000, 33, 7)])
def test_product(n, nu, k):
    import paper_1906_03938_gb300 as bem
    g = torch.Generator(device="cuda:0").manual_seed(n)
    tri = torch.tensor([[0, 1, 2]] * n, dtype=torch.int32).numpy()   # the mesh only sets n
    xyz = torch.tensor([[0.0, 0, 0], [1, 0, 0], [0, 1, 0]], dtype=torch.float64).numpy()
    ctx = bem.Context(0)
    ctx.set_mesh(xyz, tri)
    V = torch.randn((nu, n), dtype=torch.complex128, device="cuda:0", generator=g).t()
    Y = torch.randn((k, nu), dtype=torch.complex128, device="cuda:0", generator=g).t()
    X = ctx.ritz_vectors(V, Y)
    ctx.close()
    err = (X - V @ Y).abs()
    assert bool((err <= 8 * nu * 2.0 ** -52 * (V.abs() @ Y.abs())).all())
