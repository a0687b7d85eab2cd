"""The end of a row on chip (one slot per thread, eight updates deferred, compaction when 32 slots or a quarter are gone) at the sizes where it
can go wrong: fewer slots than deferred updates, one more or less than a warp, than the compaction's count, than the threads, and
rows that reach it from deferred steps.  Compared with the oracle along the GPU's order; tolerances as in every engine test."""
import numpy as np
import pytest
import torch

import obc_synth
import oracle
from parity import check_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads,d", [(128, 2), (128, 7), (128, 8), (128, 9), (128, 31), (128, 33), (128, 40), (128, 127), (128, 128), (128, 131),
                                       (256, 16), (256, 255), (256, 256), (256, 259), (512, 24), (512, 300)])
def test_end_of_a_row(threads, d):
    import paper_2208_11580_b200 as obc
    rows, ld = 3, (d + 3) // 4 * 4
    W, X = obc_synth.make_small(rows, d, 3 * d + 40, d, "relu")
    Hinv, info = oracle.inverse(oracle.hessian(X), obc_synth.DAMP_REL)
    assert info == 0
    Hd, Wd = torch.zeros(d, ld, device="cuda")[:, :d], torch.zeros(rows, ld, device="cuda")[:, :d]
    Hd.copy_(torch.from_numpy(Hinv.astype(np.float32)))
    Wd.copy_(torch.from_numpy(W.astype(np.float32)))
    Hh, Wh, opts = Hd.cpu().numpy(), Wd.cpu().numpy(), obc.engine_opts(obc.ENGINE_BLOCKED, threads, 0)
    i32 = lambda v=-7: torch.full((rows, d), v, dtype=torch.int32, device="cuda")
    f32 = lambda: torch.zeros(rows, ld, device="cuda")[:, :d]
    order, loss, status = i32(), torch.zeros(rows, d, device="cuda"), torch.full((rows,), -7, dtype=torch.int32, device="cuda")
    trace = torch.zeros(rows, d + 1, d, device="cuda")
    obc.obc_prune_trace(Wd, Hd, order, loss, status, w_trace=trace, opts=opts)
    torch.cuda.synchronize()
    assert int(status.abs().sum()) == 0
    check_rows(Hh, Wh, order.cpu().numpy(), loss.cpu().numpy(), gpu_trace=trace.cpu().numpy())
    scale, zero, Wq, codes = torch.zeros(rows, device="cuda"), torch.zeros(rows, device="cuda"), f32(), i32()
    maxq = obc.obc_minmax_grid(Wd, 4, False, scale, zero)
    obc.obc_quantize(Wd, Hd, scale, zero, 4, False, Wq, codes, status, loss=loss, qorder=order, opts=opts)
    torch.cuda.synchronize()
    assert int(status.abs().sum()) == 0
    check_rows(Hh, Wh, order.cpu().numpy(), loss.cpu().numpy(), gpu_w=Wq.cpu().numpy(), mode="quant", scale=scale.cpu().numpy().astype(np.float64),
               zero=zero.cpu().numpy().astype(np.float64), maxq=maxq, gpu_codes=codes.cpu().numpy())
    if d % 4 == 0:
        Wn, mask = f32(), torch.full((rows, d), 9, dtype=torch.uint8, device="cuda")
        obc.obc_prune_nm(Wd, Hd, 2, 4, Wn, status, order=order, loss=loss, mask=mask, opts=opts)
        torch.cuda.synchronize()
        assert int(status.abs().sum()) == 0
        check_rows(Hh, Wh, order.cpu().numpy(), loss.cpu().numpy(), gpu_w=Wn.cpu().numpy(), steps=d // 2, nm=(2, 4))
