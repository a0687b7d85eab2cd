"""Block pruning without a weight trace, the form that ships: without the trace's barrier in every step, and (blocks of 4) with the members of
a block eliminated together where the kernel can.  Order and block losses against the oracle along the GPU's order."""
import numpy as np
import pytest
import torch

import obc_synth
import oracle
from parity import REL_TOL

pytestmark = pytest.mark.gpu


def _layer(d, rows):
    W, X = obc_synth.make_small(rows, d, 2 * d + 40, d, "relu")
    Hinv, info = oracle.inverse(oracle.hessian(X), obc_synth.DAMP_REL)
    assert info == 0
    ld = (d + 3) // 4 * 4
    Hd, Wd = torch.zeros(d, ld, device="cuda")[:, :d], torch.zeros(rows, ld, device="cuda")[:, :d]
    Hd.copy_(torch.from_numpy(Hinv.astype(np.float32)))
    Wd.copy_(torch.from_numpy(W.astype(np.float32)))
    return Wd, Hd


def _run(Wd, Hd, c, threads, pending):
    import paper_2208_11580_b200 as obc
    rows, d = Wd.shape
    order = torch.full((rows, d), -7, dtype=torch.int32, device="cuda")
    loss = torch.full((rows, d), -7.0, device="cuda")
    status = torch.full((rows,), -7, dtype=torch.int32, device="cuda")
    obc.obc_prune_blocks(Wd, Hd, order, loss, status, block=c, opts=obc.engine_opts(obc.ENGINE_BLOCKED, threads, pending))
    torch.cuda.synchronize()
    return order.cpu().numpy(), loss.cpu().numpy().astype(np.float64), status.cpu().numpy()


def _check(Wd, Hd, c, threads, pending):
    rows, d = Wd.shape
    o, l, st = _run(Wd, Hd, c, threads, pending)
    assert np.all(st == 0)
    blocks = o[:, ::c] // c
    assert np.array_equal(np.sort(blocks, axis=1), np.tile(np.arange(d // c), (rows, 1)))
    assert np.array_equal(o, (blocks[:, :, None] * c + np.arange(c)).reshape(rows, d))
    assert np.all(l.reshape(rows, -1, c)[:, :, 1:] == 0.0)
    res = oracle.run_rows_blocks(Hd.cpu().numpy().astype(np.float64), Wd.cpu().numpy(), c, forced_blocks=blocks)
    assert np.all(res["status"] == 0)
    assert not ((res["best_block"] != blocks) & (res["forced_gap"] > 1e-6)).any()
    L = res["loss"][:, ::c]
    floor = 1e-7 * np.abs(L).max(axis=1, keepdims=True)
    assert (np.abs(l[:, ::c] - L) / (np.abs(L) + floor)).max() <= REL_TOL


@pytest.mark.parametrize("threads,d,pending", [(0, 64, 0), (128, 320, 0), (128, 600, 8), (256, 600, 0), (256, 1000, 16), (512, 600, 0), (512, 1000, 24)])
def test_blocks_of_8(threads, d, pending):
    _check(*_layer(d, 3), 8, threads, pending)


@pytest.mark.parametrize("threads,d,pending", [(512, 12, 0), (512, 320, 16), (512, 640, 0), (0, 740, 0), (0, 740, 12), (512, 1000, 20), (0, 1152, 0), (512, 1152, 12),
                                               (0, 2040, 0), (0, 2060, 0), (128, 600, 0), (256, 1000, 16)])
def test_blocks_of_4(threads, d, pending):
    _check(*_layer(d, 2 if d > 1500 else 3), 4, threads, pending)


@pytest.mark.parametrize("d", [640, 1152])
def test_block_that_is_not_positive_definite(d):
    """such a block is never chosen and is reported when nothing else is left, as in the single steps that a weight trace asks for"""
    import paper_2208_11580_b200 as obc
    g = np.random.default_rng(d)
    H = g.standard_normal((d, d)) * 1e-3
    H = H + H.T + np.eye(d)
    at = 4 * (d // 8)
    H[at:at + 4, :] = H[:, at:at + 4] = 0.0
    H[at:at + 4, at:at + 4] = np.eye(4)
    H[at, at + 1] = H[at + 1, at] = 2.0                        # minor 1 - 4 < 0
    Hd = torch.from_numpy(H.astype(np.float32)).cuda()
    Wd = torch.from_numpy(g.standard_normal((2, d)).astype(np.float32)).cuda()
    o, l, st = _run(Wd, Hd, 4, 512, 0)
    assert np.all(st == 1 + d - 4) and np.all(o[:, -4:] == -1) and np.all(np.isinf(l[:, -4:])) and not np.any(o[:, :-4] // 4 == at // 4)
    order, loss = torch.zeros(2, d, dtype=torch.int32, device="cuda"), torch.zeros(2, d, device="cuda")
    status, trace = torch.zeros(2, dtype=torch.int32, device="cuda"), torch.zeros(2, d + 1, d, device="cuda")
    obc.obc_prune_blocks(Wd, Hd, order, loss, status, block=4, w_trace=trace, opts=obc.engine_opts(obc.ENGINE_BLOCKED, 512, 0))
    torch.cuda.synchronize()
    assert np.array_equal(status.cpu().numpy(), st) and (order.cpu().numpy() == o).mean() > 0.99
