"""The FP32 estimates that screen the candidates of a step, where they could lead away from the FP64 scores: weights far beyond the grid (the
integer nearest to w / scale does not fit 32 bits), weights that lie on the grid exactly (all scores 0: the lowest column goes first), grids
whose zero point is no integer."""
import numpy as np
import pytest
import torch

import obc_synth
import oracle
from parity import check_rows

pytestmark = pytest.mark.gpu


def _quantize(W, H, scale, zero, bits, threads, symmetric):
    import paper_2208_11580_b200 as obc
    rows, d = W.shape
    Wd, Hd = torch.from_numpy(W).cuda(), torch.from_numpy(H).cuda()
    sc, ze = torch.from_numpy(scale).cuda(), torch.from_numpy(zero).cuda()
    Wq, loss = torch.zeros(rows, d, device="cuda"), torch.zeros(rows, d, device="cuda")
    codes, order = torch.zeros(rows, d, dtype=torch.int32, device="cuda"), torch.zeros(rows, d, dtype=torch.int32, device="cuda")
    status = torch.full((rows,), -7, dtype=torch.int32, device="cuda")
    obc.obc_quantize(Wd, Hd, sc, ze, bits, symmetric, Wq, codes, status, loss=loss, qorder=order, opts=obc.engine_opts(obc.ENGINE_BLOCKED, threads, 0))
    torch.cuda.synchronize()
    assert int(status.abs().sum()) == 0
    return order.cpu().numpy(), loss.cpu().numpy(), Wq.cpu().numpy(), codes.cpu().numpy()


def _hinv(d):
    _, X = obc_synth.make_small(1, d, 2 * d + 40, d, "relu")
    Hinv, info = oracle.inverse(oracle.hessian(X), obc_synth.DAMP_REL)
    assert info == 0
    return Hinv.astype(np.float32)


@pytest.mark.parametrize("sign", [-1, 1])
@pytest.mark.parametrize("threads,d", [(128, 64), (128, 320), (256, 512), (512, 640)])
def test_weights_far_beyond_the_grid(threads, d, sign):
    sc, maxq, ze = np.float32(0.1), 65534, np.float32(32767)
    # a weight next to +-2^32 scales, whose quotient is 2e-3 away from an integer at most (but not 0) and whose low 32 bits are a code
    w = np.float32(sign * (2.0 ** 32 - 30000 * np.arange(1, 200)[::-1] / 200 * 32) * 0.1)
    t = w.astype(np.float64) / np.float64(sc)
    far = np.abs(t - np.rint(t))
    low = np.rint(t) - sign * 2.0 ** 32
    ok = (np.abs(low) < 32000) & (far > 1e-5)
    g = np.random.default_rng(d)
    W = (g.standard_normal((2, d)) * 100).astype(np.float32)
    W[:, d // 3] = w[ok][np.argmin(far[ok])]
    order, loss, _, _ = _quantize(W, _hinv(d), np.full(2, sc), np.full(2, ze), 16, threads, True)
    assert np.all(order[:, 0] != d // 3)               # the worst of all scores
    first = 16                                         # (compared while the row is as it was: that weight has not been taken)
    at = [int(np.argmax(order[r] == d // 3)) for r in range(2)]
    assert min(at) >= first
    check_rows(_hinv(d), W, order, loss, mode="quant", scale=np.full(2, np.float64(sc)), zero=np.full(2, np.float64(ze)), maxq=maxq, steps=first)


@pytest.mark.parametrize("threads,d", [(128, 64), (128, 320), (256, 512), (512, 640)])
def test_weights_on_the_grid(threads, d):
    # w = scale * a power of two: the FP64 distance to the grid is 0, w / scale through the reciprocal is not
    cand = (0.3 + 0.01 * np.arange(200)).astype(np.float32)
    sc = next(s for s in cand if np.float64(s) * (1.0 / np.float64(s)) != 1.0)
    g = np.random.default_rng(d)
    W = (sc * np.array([1, -1, 2, -2, 4, -4], np.float32)[g.integers(0, 6, (2, d))]).astype(np.float32)
    H = (np.diag(g.uniform(1e-4, 1e-3, d)) + 1e-5).astype(np.float32)
    order, loss, Wq, codes = _quantize(W, H, np.full(2, sc), np.full(2, np.float32(7)), 4, threads, True)
    assert np.array_equal(order, np.tile(np.arange(d), (2, 1))) and np.all(loss == 0.0)
    assert np.array_equal(Wq, W) and np.array_equal(codes, np.rint(W / sc).astype(np.int64) + 7)


@pytest.mark.parametrize("zero", [7.25, 7.5, 7.000001, 1e-12])
@pytest.mark.parametrize("threads,d", [(128, 64), (128, 300), (512, 516)])
def test_zero_point_that_is_no_integer(threads, d, zero):
    W, H = obc_synth.make_small(2, d, 2 * d + 40, d, "relu")[0].astype(np.float32), _hinv(d)
    if zero < 1:                                       # (a grid of positive values)
        W = np.abs(W)
    sc, ze = (np.abs(W).max(axis=1) / (7 if zero > 1 else 15)).astype(np.float32), np.full(2, zero, np.float32)
    order, loss, Wq, codes = _quantize(W, H, sc, ze, 4, threads, False)
    check_rows(H, W, order, loss, gpu_w=Wq, mode="quant", scale=sc.astype(np.float64), zero=ze.astype(np.float64), maxq=15, gpu_codes=codes)
