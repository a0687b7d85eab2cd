"""Replays whose last part runs on chip: from the number of slots where a replay alone moves there, reached with and without a rest of a group
of four, against the weight trace that the same order leaves."""
import numpy as np
import pytest
import torch

import obc_synth
import oracle
from parity import REL_TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads,d", [(128, 129), (128, 160), (128, 250), (256, 229), (256, 256), (256, 330), (512, 270), (512, 452), (0, 161)])
def test_replay_against_trace(threads, d):
    import paper_2208_11580_b200 as obc
    rows, ld = 6, (d + 3) // 4 * 4
    W, X = obc_synth.make_small(rows, d, 2 * d + 40, d, "relu")
    Hinv, info = oracle.inverse(oracle.hessian(X), obc_synth.DAMP_REL)
    assert info == 0
    Hd, Wd = torch.zeros(d, ld, device="cuda")[:, :d], torch.zeros(rows, ld, device="cuda")[:, :d]
    Hd.copy_(torch.from_numpy(Hinv.astype(np.float32)))
    Wd.copy_(torch.from_numpy(W.astype(np.float32)))
    opts = obc.engine_opts(obc.ENGINE_BLOCKED, threads, 0)
    order, loss = torch.zeros(rows, d, dtype=torch.int32, device="cuda"), torch.zeros(rows, d, device="cuda")
    status, trace = torch.zeros(rows, dtype=torch.int32, device="cuda"), torch.zeros(rows, d + 1, d, device="cuda")
    obc.obc_prune_trace(Wd, Hd, order, loss, status, w_trace=trace, opts=opts)
    left = [d - 1, d // 2, 130, 65, 3, 0]                      # slots left at the end of each row's replay
    counts = torch.tensor([d - min(n, d) for n in left], dtype=torch.int32, device="cuda")
    Wo = torch.full((rows, ld), 7.0, device="cuda")[:, :d]
    obc.obc_prune_apply(Wd, Hd, order, counts, Wo, status, opts=opts)
    torch.cuda.synchronize()
    assert int(status.abs().sum()) == 0
    want = torch.stack([trace[r, int(counts[r])] for r in range(rows)]).cpu().numpy()
    got, scale = Wo.cpu().numpy(), np.abs(Wd.cpu().numpy()).max(axis=1, keepdims=True)
    assert np.array_equal(got == 0.0, want == 0.0)
    assert (np.abs(got - want) / np.maximum(np.abs(want), scale)).max() <= 2 * REL_TOL      # (each is within REL_TOL of the exact weights)
