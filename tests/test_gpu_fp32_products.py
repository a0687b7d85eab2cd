"""The FP32 products: rounding against FP64, and sizes at the limits of a launch."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# Relative errors (2-norm) of the Hessian with 32 slices at most, added in FP32, on these inputs were, in this order, 1.07e-7, 0.90e-7,
# 1.22e-7, 0.79e-7, 1.88e-7, 1.49e-7; however the contraction is cut, it must not be further off.  (A fixed seed: the factor 1.1 is
# for the difference between one random stream and another.)
@pytest.mark.parametrize("kind,d,n,bound", [("relu", 64, 65536, 1.07e-7), ("relu", 147, 50173, 0.90e-7), ("normal", 64, 65536, 1.22e-7),
                                            ("relu", 1024, 8192, 0.79e-7), ("normal", 1024, 8192, 1.88e-7), ("normal", 700, 16384, 1.49e-7)])
def test_hessian_rounding(kind, d, n, bound):
    import paper_2208_11580_b200 as m
    g = torch.Generator(device="cuda").manual_seed(d * 7 + n)
    X = torch.zeros(d, (n + 3) // 4 * 4, device="cuda")[:, :n]
    x = torch.randn(d, n, device="cuda", generator=g)
    X.copy_(x.relu() if kind == "relu" else x)
    H = torch.zeros(d, (d + 3) // 4 * 4, device="cuda")[:, :d]
    m.obc_hessian(X, H, prec=m.PREC_FP32)
    want = 2 * X.double() @ X.double().T
    assert float((H.double() - want).norm() / want.norm()) <= 1.1 * bound


def test_cross_product_of_more_columns_than_a_grid_dimension_has_tiles():
    import paper_2208_11580_b200 as m
    r, d, n = 2, 65535 * 128 + 130, 4
    g = torch.Generator(device="cuda").manual_seed(1)
    Y, X = torch.randn(r, n, device="cuda", generator=g), torch.randn(d, n, device="cuda", generator=g)
    G = torch.zeros(r, (d + 3) // 4 * 4, device="cuda")[:, :d]
    m.obc_cross_gram(Y, X, G, prec=m.PREC_FP32)
    want = Y.double() @ X.double().T
    # four products and their sum, each rounded once, of the size of the row norms' product
    assert float((G - want).abs().max()) <= 8 * 2.0 ** -24 * float(Y.double().norm(dim=1).max() * X.double().norm(dim=1).max())
