"""Rows of 512 threads: passes over the triangle on tcgen05, at the edges of their tiles (128 x 64), of their groups of 16 vectors
and of the number of vectors kept in shared memory, and with a diagonal that spans more than the FP16 planes' common power
of two covers (every slot has a power of its own there).  Compared with the oracle along the GPU's order; tolerances as in
every engine test (check_rows): FP32 matrix, so picks beyond a 1e-6 margin, losses and weights within 1e-4."""
import numpy as np
import pytest
import torch

import obc_synth
import oracle
from parity import check_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("d,pending", [(260, 0), (319, 1), (384, 16), (385, 17), (513, 33), (641, 0), (1090, 40)])
def test_passes_against_oracle(d, pending, wide):
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
    obc.obc_prune_trace(Wd, Hd, order, loss, status, opts=obc.engine_opts(obc.ENGINE_BLOCKED, 512, pending))
    torch.cuda.synchronize()
    assert int(status.abs().sum()) == 0
    check_rows(Hd.cpu().numpy(), Wd.cpu().numpy(), order.cpu().numpy(), loss.cpu().numpy())


def test_diagonal_that_collapses_before_the_pass():
    """Two slots with diagonal 2^41 and correlation 1 - 2^-20: once the first is eliminated the other has 2^22 left, within 2^24 of the
    rest (about 1), but its entry of the pending vector is still 2^20.5.  A common power of two for that entry would lose the
    others' (about 2^-21); the products of the two are what the survivor's column is made of."""
    import paper_2208_11580_b200 as obc
    d, T, eps = 300, 2.0 ** 41, 2.0 ** -20
    rng = np.random.default_rng(3)
    _, X = obc_synth.make_small(1, d - 2, 3 * d, 9, "relu")
    A, info = oracle.inverse(oracle.hessian(X), obc_synth.DAMP_REL)
    assert info == 0
    Hinv = np.zeros((d, d))
    Hinv[2:, 2:] = A / np.diag(A).mean()
    Hinv[:2, :2] = T * np.array([[1, 1 - eps], [1 - eps, 1]])
    u = rng.standard_normal(d - 2)
    u *= 0.2 * np.sqrt(T * eps * np.linalg.eigvalsh(Hinv[2:, 2:])[0]) / np.linalg.norm(u)
    Hinv[0, 2:] = Hinv[2:, 0] = u
    Hinv[1, 2:] = Hinv[2:, 1] = -u
    W = rng.standard_normal((2, d))
    W[:, 0], W[:, 1] = 0.0, 1400.0                  # the first goes at once, the second in the middle of the row
    Hd, Wd = torch.from_numpy(Hinv.astype(np.float32)).cuda(), torch.from_numpy(W.astype(np.float32)).cuda()
    order = torch.full((2, d), -7, dtype=torch.int32, device="cuda")
    loss, status = torch.zeros(2, d, device="cuda"), torch.full((2,), -7, dtype=torch.int32, device="cuda")
    obc.obc_prune_trace(Wd, Hd, order, loss, status, opts=obc.engine_opts(obc.ENGINE_BLOCKED, 512, 0))
    torch.cuda.synchronize()
    assert int(status.abs().sum()) == 0
    P = order.cpu().numpy()
    assert (P[:, 0] == 0).all() and (np.argwhere(P == 1)[:, 1] > 48).all()
    check_rows(Hd.cpu().numpy(), Wd.cpu().numpy(), P, loss.cpu().numpy())
