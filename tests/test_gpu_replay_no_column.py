"""A replay whose order holds an entry that names no column (-1, as a row that failed leaves it, or one beyond the row) within the count: the
row stops there and is reported, in the part on chip, with vectors pending, and inside a group of four; the other rows, and the memory in
front of and behind the outputs, are as without it."""
import numpy as np
import pytest
import torch

import obc_synth
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads,d,at", [
    (128, 64, 0), (128, 64, 9), (128, 128, 40), (256, 64, 17), (256, 256, 70), (0, 100, 3),      # wholly on chip
    (128, 300, 290), (256, 500, 480), (512, 500, 496),                                           # on chip, reached from passes
    (128, 300, 0), (128, 300, 8), (128, 300, 13), (256, 500, 6), (256, 500, 130), (512, 500, 5), (512, 500, 64), (0, 700, 2)])
@pytest.mark.parametrize("entry", [-1, 1 << 20])
def test_entry_that_names_no_column(threads, d, at, entry):
    import paper_2208_11580_b200 as obc
    rows, ld = 4, (d + 3) // 4 * 4
    W, X = obc_synth.make_small(rows, d, 2 * d + 40, d, "relu")
    Hinv, info = oracle.inverse(oracle.hessian(X), obc_synth.DAMP_REL)
    assert info == 0
    Hd, Wd = torch.zeros(d, ld, device="cuda")[:, :d], torch.zeros(rows, ld, device="cuda")[:, :d]
    Hd.copy_(torch.from_numpy(Hinv.astype(np.float32)))
    Wd.copy_(torch.from_numpy(W.astype(np.float32)))
    opts = obc.engine_opts(obc.ENGINE_BLOCKED, threads, 0)
    order = torch.from_numpy(np.stack([np.random.default_rng(d + r).permutation(d) for r in range(rows)]).astype(np.int32)).cuda()
    bad = [0, 2]
    broken = order.clone()
    broken[bad, at:] = entry
    counts = torch.full((rows,), min(d, at + 9), dtype=torch.int32, device="cuda")

    def fill(dtype, value, cols):                       # outputs inside a larger buffer
        b = torch.full((rows + 2, cols), value, dtype=dtype, device="cuda")
        return b, b[1:-1, :d]

    def outputs(o, quantize):
        Wb, Wo = fill(torch.float32, 77.0, ld)
        cb, codes = fill(torch.int32, 77, d)
        status = torch.full((rows,), -7, dtype=torch.int32, device="cuda")
        if quantize:
            scale, zero = torch.zeros(rows, device="cuda"), torch.zeros(rows, device="cuda")
            obc.obc_quantize(Wd, Hd, scale, zero, 4, True, Wo, codes, status, prune_order=o, prune_counts=counts, opts=opts)
        else:
            obc.obc_prune_apply(Wd, Hd, o, counts, Wo, status, opts=opts)
        torch.cuda.synchronize()
        return Wb.cpu().numpy(), cb.cpu().numpy(), status.cpu().numpy()

    for quantize in (False, True):
        W0, c0, s0 = outputs(order, quantize)
        W1, c1, s1 = outputs(broken, quantize)
        assert np.all(s0 == 0)
        assert np.array_equal(s1, np.where(np.isin(np.arange(rows), bad), 1 + at, 0))
        for b in (W1, c1):
            assert np.all(b[[0, -1]] == 77) and np.all(b[:, d:] == 77)
        good = [1 + r for r in range(rows) if r not in bad]
        assert np.array_equal(W0[good], W1[good]) and np.array_equal(c0[good], c1[good])
        o = order.cpu().numpy()
        for r in bad:                                   # what was eliminated before the entry is zero, the rest are weights
            kept = np.ones(d, bool)
            kept[o[r, :at]] = False
            assert np.all(W1[1 + r, :d][~kept] == 0.0) and np.all(np.isfinite(W1[1 + r, :d][kept])) and np.all(W1[1 + r, :d][kept] != 0.0)
            if quantize:
                assert np.all(c1[1 + r, :d] == -1)
