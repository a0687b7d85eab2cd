"""Hessian, cross products and dense refit at the edges of their tiles and slices (either FP32 tile, ragged rows, short and odd
contractions, several parts of the contraction), against FP64 products on the GPU.  Tolerances relative to the largest entry:
FP32 sums of at most 2048 products before the partial sums (2e-5), split BF16 values (16 significant bits, 3e-5), TF32 (2e-3)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = {0: 2e-5, 1: 2e-3, 2: 3e-5}


def matrix(rows, cols, g):
    m = torch.zeros(rows, (cols + 3) // 4 * 4, device="cuda")[:, :cols]
    m.copy_(torch.randn(rows, cols, device="cuda", generator=g) + 0.3)
    return m


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("d,n", [(2, 3), (63, 31), (64, 129), (65, 4097), (147, 2053), (257, 640), (640, 33), (641, 5000), (1025, 300), (2305, 1030)])
def test_hessian_tiles(d, n, prec):
    import paper_2208_11580_b200 as obc
    g = torch.Generator(device="cuda").manual_seed(d + n)
    X, H = matrix(d, n, g), matrix(d, d, g)
    before = H.clone()
    obc.obc_hessian(X, H, accumulate=True, prec=prec)
    want = 2 * X.double() @ X.double().T
    low = torch.tril(torch.ones(d, d, device="cuda", dtype=torch.bool))
    assert ((H.double() - before.double() - want)[low].abs().max() <= TOL[prec] * want.abs().max() + 1e-6)
    obc.obc_hessian(X, H, prec=prec)
    assert torch.equal(H, H.T)
    assert (H.double() - want).abs().max() <= TOL[prec] * want.abs().max()


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("r,d,n", [(2, 3, 5), (65, 64, 257), (37, 300, 2051), (130, 129, 8200), (1500, 1100, 515)])
def test_cross_and_refit_tiles(r, d, n, prec):
    import paper_2208_11580_b200 as obc
    g = torch.Generator(device="cuda").manual_seed(r + d + n)
    Y, X, G = matrix(r, n, g), matrix(d, n, g), matrix(r, d, g)
    before = G.clone()
    obc.obc_cross_gram(Y, X, G, accumulate=True, prec=prec)
    want = Y.double() @ X.double().T
    assert (G.double() - before.double() - want).abs().max() <= TOL[prec] * want.abs().max() + 1e-6
    S = matrix(d, d, g)
    S.copy_(S + S.T)
    W = matrix(r, d, g)
    obc.obc_refit(G, S, W, prec=prec)
    want = 2 * G.double() @ S.double()
    scale = (2 * G.double().abs() @ S.double().abs()).max()
    assert (W.double() - want).abs().max() <= TOL[prec] * scale
