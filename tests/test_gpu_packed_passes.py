"""Rows of 128 and 256 threads: passes over the triangle by mma.sync on packed FP16 planes, at the edges of their tiles (16 x 64), of
their groups of 16 vectors, with an odd number of vectors, and with a diagonal that is too wide for the planes (which takes the TF32
form).  Compared with the oracle along the GPU's order; tolerances as in every engine test (check_rows)."""
import numpy as np
import pytest
import torch

import obc_synth
import oracle
from parity import check_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("threads,d,pending", [(128, 145, 1), (128, 193, 7), (128, 260, 16), (128, 321, 17), (128, 513, 33), (128, 700, 0),
                                               (256, 304, 15), (256, 417, 32), (256, 705, 0), (256, 1090, 47)])
def test_passes_against_oracle(threads, d, pending, wide):
    import paper_2208_11580_b200 as obc
    W, X = obc_synth.make_small(3, d, 2 * d + 40, d, "relu")
    Hinv, info = oracle.inverse(oracle.hessian(X), obc_synth.DAMP_REL)
    assert info == 0
    # columns in other units: w s, s Hinv s have the same scores and picks
    s = 10.0 ** (-5.0 * np.random.default_rng(d).random(d)) if wide else np.ones(d)
    ld = (d + 3) // 4 * 4
    Hd, Wd = torch.zeros(d, ld, device="cuda")[:, :d], torch.zeros(3, ld, device="cuda")[:, :d]
    Hd.copy_(torch.from_numpy((Hinv * s[:, None] * s[None, :]).astype(np.float32)))
    Wd.copy_(torch.from_numpy((W * s).astype(np.float32)))
    order = torch.full((3, d), -7, dtype=torch.int32, device="cuda")
    loss = torch.zeros(3, d, device="cuda")
    status = torch.full((3,), -7, dtype=torch.int32, device="cuda")
    obc.obc_prune_trace(Wd, Hd, order, loss, status, opts=obc.engine_opts(obc.ENGINE_BLOCKED, threads, pending))
    torch.cuda.synchronize()
    assert int(status.abs().sum()) == 0
    check_rows(Hd.cpu().numpy(), Wd.cpu().numpy(), order.cpu().numpy(), loss.cpu().numpy())
