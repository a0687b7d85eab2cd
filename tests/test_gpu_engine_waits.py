"""Bounded waits that run out on purpose: the pipeline of a pass on tcgen05, the 256 x 256 tiles of the Hessian and the cross product.
Nothing hangs and nothing faults: the products of a pass give up at a given tile, as after a wait that expired, and the block abandons
the pass; the other kernels take a limit of -1 (every wait expires at once) or a few polls.  The call returns, the failure is reported, and the next ordinary call is right."""
import ctypes
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu
OBC_ERR_TIMEOUT = 6
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    import paper_2208_11580_b200 as m
    m.load_library()
    out = str(tmp_path_factory.mktemp("shim") / "wait_limit_shim.so")
    pkg = os.path.dirname(m.library_path())
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-O1", "-o", out, os.path.join(HERE, "wait_limit_shim.cpp"), "-I", os.path.join(pkg, "csrc"),
                           "-I", os.path.join(os.path.dirname(pkg), "include"), "-I", "/usr/local/cuda/include", m.library_path()])
    return m, ctypes.CDLL(out)


def pointer(t):
    return ctypes.c_void_p(t.data_ptr())


def spd(d, g):
    X = torch.randn(d, 2 * d, device="cuda", generator=g, dtype=torch.float64)
    H = X @ X.T
    H.diagonal().add_(0.01 * H.diagonal().mean())
    return torch.cholesky_inverse(torch.linalg.cholesky(H))


# a few tiles / rows handed over between blocks / pending vectors in global memory, the smallest rings
@pytest.mark.parametrize("rows,d", [(5, 600), (1, 261), (161, 520), (3, 4200)])
def test_pass_that_runs_out_of_time(shim, rows, d):
    m, lib = shim
    g = torch.Generator(device="cuda").manual_seed(d)
    inv = spd(d, g)
    Hinv, W = ((inv + inv.T) / 2).float().contiguous(), torch.randn(rows, (d + 3) // 4 * 4, device="cuda", generator=g)
    if d % 4:
        pad = torch.zeros(d, W.shape[1], device="cuda")
        pad[:, :d] = Hinv
        Hinv = pad
    ws = torch.empty(m.obc_workspace_bytes(m.OP_PRUNE_TRACE, rows, d), dtype=torch.uint8, device="cuda")

    def call(stop):
        order = torch.full((rows, d), -7, dtype=torch.int32, device="cuda")
        loss, st = torch.zeros(rows, d, device="cuda"), torch.full((rows,), -7, dtype=torch.int32, device="cuda")
        rc = lib.shim_prune_trace(pointer(W), W.shape[1], rows, d, pointer(Hinv), Hinv.shape[1], pointer(order), pointer(loss), pointer(st), pointer(ws),
                                  ctypes.c_size_t(ws.numel()), 512, stop, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        torch.cuda.synchronize()
        return order, loss, st

    want = call(0)
    assert int(want[2].abs().sum()) == 0
    tiles = sum(-(-(d - 48 - 64 * c) // 128) for c in range(d // 64))      # about those of the first pass
    for stop in (1, 2, 3, 4, 5, 6, 8, 11, tiles // 2, tiles - 2, tiles - 1, tiles, 10 ** 6):
        order, loss, st = call(max(stop, 1))
        late = st == -OBC_ERR_TIMEOUT
        assert bool((late | (st == 0)).all())
        if stop == 1:
            assert bool(late.all())
        if stop == 10 ** 6:
            assert not bool(late.any())
        assert torch.equal(order[~late], want[0][~late]) and torch.equal(loss[~late], want[1][~late])
        assert bool((order[late][:, -1] == -1).all()) and bool(torch.isinf(loss[late][:, -1]).all())      # what was not produced
        assert torch.equal(torch.where(order[late] == -1, want[0][late], order[late]), want[0][late])         # what was, before
        again = call(0)
        assert all(torch.equal(a, b) for a, b in zip(again, want))


def test_large_hessian_tiles_that_run_out_of_time():
    import paper_2208_11580_b200 as m
    d, n = 2304, 1500
    X = torch.randn(d, n, device="cuda")
    H, info = torch.zeros(d, d, device="cuda"), torch.full((1,), -1, dtype=torch.int32, device="cuda")
    want = 2 * X.double() @ X.double().T
    for limit in (-1, 0, 3, 0):
        m.obc_hessian(X, H, prec=m.PREC_BF16X3, info=info, wait_limit=limit)
        late = int(info.item())
        assert late == {-1: OBC_ERR_TIMEOUT, 0: 0}.get(limit, late)
        assert bool(torch.isnan(H).all()) if late else float((H.double() - want).abs().max() / want.abs().max()) <= 3e-5


def test_large_cross_product_tiles_that_run_out_of_time():
    import paper_2208_11580_b200 as m
    r, d, n = 1536, 2048, 1500
    Y, X = torch.randn(r, n, device="cuda"), torch.randn(d, n, device="cuda")
    G, info = torch.zeros(r, d, device="cuda"), torch.full((1,), -1, dtype=torch.int32, device="cuda")
    want = Y.double() @ X.double().T
    for limit in (-1, 0, 3, 0):
        m.obc_cross_gram(Y, X, G, prec=m.PREC_BF16X3, info=info, wait_limit=limit)
        late = int(info.item())
        assert late == {-1: OBC_ERR_TIMEOUT, 0: 0}.get(limit, late)
        assert bool(torch.isnan(G).all()) if late else float((G.double() - want).abs().max() / want.abs().max()) <= 3e-5


def test_selection_that_runs_out_of_time_is_reported_downstream(shim):
    m, lib = shim
    rows, d = 300, 96
    g = torch.Generator(device="cuda").manual_seed(4)
    inv = spd(d, g)
    Hinv, W = ((inv + inv.T) / 2).float().contiguous(), torch.randn(rows, d, device="cuda", generator=g)
    order, loss = torch.zeros(rows, d, dtype=torch.int32, device="cuda"), torch.zeros(rows, d, device="cuda")
    st = torch.zeros(rows, dtype=torch.int32, device="cuda")
    trace = torch.zeros(rows, d + 1, d, device="cuda")
    m.obc_prune_trace(W, Hinv, order, loss, st, w_trace=trace)
    counts, mask = torch.zeros(rows, dtype=torch.int32, device="cuda"), torch.full((rows, d), 7, dtype=torch.uint8, device="cuda")
    ws = torch.empty(m.obc_workspace_bytes(m.OP_SELECT, rows, d), dtype=torch.uint8, device="cuda")

    def select(limit):
        rc = lib.shim_select(pointer(loss), pointer(order), rows, d, ctypes.c_longlong(rows * d // 2), pointer(counts), pointer(mask), pointer(ws), limit,
                             ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0

    select(-1)
    assert bool((counts == -OBC_ERR_TIMEOUT).all())
    counts[::3] = 5                                 # the other rows are ordinary ones
    late = counts == -OBC_ERR_TIMEOUT
    out = torch.zeros(rows, d, device="cuda")
    for kw in (dict(), dict(w_trace=trace, trace_steps=d), dict(opts=m.engine_opts(m.ENGINE_STREAMING))):
        st.zero_()
        m.obc_prune_apply(W, Hinv, order, counts, out, st, **kw)
        assert torch.equal(st, torch.where(late, -OBC_ERR_TIMEOUT, 0).int())
        assert torch.equal(out[late], W[late]) and bool(((out == 0).sum(1)[~late] == 5).all())
    scale, zero, codes = torch.zeros(rows, device="cuda"), torch.zeros(rows, device="cuda"), torch.zeros(rows, d, dtype=torch.int32, device="cuda")
    m.obc_quantize(W, Hinv, scale, zero, 4, True, out, codes, st, prune_order=order, prune_counts=counts)
    assert torch.equal(st, torch.where(late, -OBC_ERR_TIMEOUT, 0).int())
    counts.fill_(-3)                                # any other negative count prunes nothing, as ever
    m.obc_prune_apply(W, Hinv, order, counts, out, st)
    assert int(st.abs().sum()) == 0 and torch.equal(out, W)
    select(0)                                       # and the next selection is right
    want = (torch.zeros_like(counts), torch.zeros_like(mask))
    m.obc_select_global_mask(loss, order, rows * d // 2, *want)
    assert torch.equal(counts, want[0]) and torch.equal(mask, want[1]) and int(counts.sum()) == rows * d // 2
