"""The longest rows the engine takes (d_col 4097 to 5120: twelve slots per thread, up to 40 pending vectors in global memory, the
smallest operand and tile rings), eliminated to the end, every mode.  A row of this length takes minutes on the CPU oracle, so
the reference is the same method in FP64 torch on the GPU (`fp64_rows`, FP64 updates applied 64 at a time), which is pinned to the
oracle here; it runs along the engine's order like the oracle does in check_rows, with the same tolerances."""
import numpy as np
import pytest
import torch

import obc_synth
import oracle
import parity
from parity import check_rows, record_stats, REL_TOL


def fp64_rows(Hinv, W, steps=None, mode="prune", scale=None, zero=None, maxq=0, flags=0, forced=None, active0=None, want_trace=False, nm=None):
    """oracle.run_rows (without flags and active0) for all rows at once, in FP64 torch."""
    assert flags == 0 and active0 is None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    t = lambda x: torch.tensor(np.asarray(x, dtype=np.float64), device=dev)
    H0, w = t(Hinv), t(W)
    R, d = w.shape
    steps = d if steps is None else steps
    quant = mode == "quant"
    if quant:
        sc, ze = t(np.broadcast_to(scale, (R,)))[:, None], t(np.broadcast_to(zero, (R,)))[:, None]
    H = H0.repeat(R, 1, 1)
    dg = H0.diagonal().repeat(R, 1)
    alive = torch.ones(R, d, dtype=torch.bool, device=dev)
    B, nb = 64, 0
    Z = torch.zeros(R, B, d, dtype=torch.float64, device=dev)
    rows = torch.arange(R, device=dev)
    out = torch.zeros_like(w)
    codes = torch.full((R, d), -1, dtype=torch.int32, device=dev)
    res = {k: torch.zeros(R, steps, dtype=torch.float64, device=dev) for k in ("loss", "margin", "forced_gap", "pivot_diag", "round_dist")}
    res.update({k: torch.zeros(R, steps, dtype=torch.int64, device=dev) for k in ("order", "best")})
    trace = torch.zeros(R, steps + 1, d, dtype=torch.float64, device=dev) if want_trace else None
    if want_trace:
        trace[:, 0] = w
    if nm is not None:
        lost = torch.zeros(R, d // nm[1], dtype=torch.int64, device=dev)
    if forced is not None:
        forced = torch.as_tensor(np.ascontiguousarray(forced, dtype=np.int64), device=dev)
    for s in range(steps):
        q, c = torch.zeros_like(w), torch.full_like(w, -1.0)
        if quant:
            c = torch.clamp(torch.round(w / sc) + ze, 0, maxq)
            q = sc * (c - ze)
        allowed = alive if nm is None else alive & (lost < nm[1] - nm[0]).repeat_interleave(nm[1], 1)
        score = torch.where(allowed, (q - w).square() / dg, torch.inf)
        two = torch.topk(score, min(2, d), dim=1, largest=False)
        p = two.indices[:, 0] if forced is None else forced[:, s]
        sp, sb = score[rows, p], two.values[:, 0]
        res["best"][:, s], res["order"][:, s], res["loss"][:, s] = two.indices[:, 0], p, sp
        res["forced_gap"][:, s] = (sp - sb) / sp.clamp_min(1e-300)
        res["margin"][:, s] = torch.where(torch.isfinite(two.values[:, -1]), (two.values[:, -1] - sb) / two.values[:, -1].clamp_min(1e-300), 1.0)
        dpp = dg[rows, p]
        res["pivot_diag"][:, s] = dpp
        if quant:
            x = (w / sc)[rows, p]
            res["round_dist"][:, s] = ((x - x.floor()).abs() - 0.5).abs()
        codes[rows, p], out[rows, p] = c[rows, p].int(), q[rows, p]
        col = H[rows, p]
        if nb:
            col = col - torch.bmm(Z[rows, :nb, p].unsqueeze(1), Z[:, :nb])[:, 0]
        w = w - ((w - q)[rows, p] / dpp)[:, None] * col
        dg = dg - col.square() / dpp[:, None]
        alive[rows, p] = False
        if nm is not None:
            lost[rows, p // nm[1]] += 1
        Z[:, nb] = torch.where(alive, col * dpp.rsqrt()[:, None], 0.0)
        nb += 1
        if nb == B and s + 1 < steps:
            H.baddbmm_(Z.transpose(1, 2), Z, alpha=-1.0)
            nb = 0
        if want_trace:
            trace[:, s + 1] = torch.where(alive, w, out)
    res.update(w=torch.where(alive, w, out), codes=codes, w_trace=trace, status=torch.zeros(R, dtype=torch.int32))
    return {k: None if v is None else v.cpu().numpy() for k, v in res.items()}


@pytest.mark.parametrize("mode", ["prune", "quant", "nm"])
def test_the_reference_is_the_oracle(mode):
    d = 152
    W, X = obc_synth.make_small(3, d, 3 * d, 5, "relu")
    Hinv, info = oracle.inverse(oracle.hessian(X), obc_synth.DAMP_REL)
    kw = dict(mode="quant", scale=np.abs(W).max(1) / 7, zero=7.0, maxq=14) if mode == "quant" else dict(nm=(2, 4), steps=d // 2) if mode == "nm" else {}
    for forced in (False, True):
        if forced:                                  # another order than the greedy one
            kw["forced"] = np.stack([np.roll(a["order"][r], 3) for r in range(3)])
        if forced and mode == "nm":
            break
        a = oracle.run_rows(Hinv, W, want_trace=True, **kw)
        b = fp64_rows(Hinv, W, want_trace=True, **kw)
        assert np.array_equal(a["order"], b["order"]) and np.array_equal(a["best"], b["best"]) and np.array_equal(a["codes"], b["codes"])
        for k in ("loss", "forced_gap", "margin", "pivot_diag", "w", "w_trace") + (("round_dist",) if mode == "quant" else ()):
            assert np.allclose(a[k], b[k], rtol=1e-9, atol=1e-9 * max(1.0, np.abs(W).max())), k


def layer(rows, d, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(d, 2 * d + 96, device="cuda", generator=g, dtype=torch.float64).relu_()
    H = 2.0 * X @ X.T
    H.diagonal().add_(obc_synth.DAMP_REL * H.diagonal().mean())
    inv = torch.cholesky_inverse(torch.linalg.cholesky(H))
    ld = (d + 3) // 4 * 4
    Hinv, W = torch.zeros(d, ld, device="cuda")[:, :d], torch.zeros(rows, ld, device="cuda")[:, :d]
    Hinv.copy_((inv + inv.T) * 0.5)
    W.copy_(torch.randn(rows, d, device="cuda", generator=g) * (2.0 / d) ** 0.5)
    return Hinv, W


def buffers(rows, d):
    i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device="cuda")
    return i32(rows, d), torch.zeros(rows, d, device="cuda"), i32(rows)


@pytest.fixture
def gpu_reference(monkeypatch):
    monkeypatch.setattr(parity.oracle, "run_rows", fp64_rows)


@pytest.mark.gpu
@pytest.mark.parametrize("rows,d,bits,symmetric", [(128, 4608, 4, True), (3, 4097, 4, False), (6, 5119, 8, True)])
def test_obq(gpu_reference, rows, d, bits, symmetric):
    import paper_2208_11580_b200 as m
    Hinv, W = layer(rows, d, d)
    order, loss, st = buffers(rows, d)
    codes, Wq = torch.zeros_like(order), torch.zeros(rows, (d + 3) // 4 * 4, device="cuda")[:, :d]
    scale, zero = torch.zeros(rows, device="cuda"), torch.zeros(rows, device="cuda")
    maxq = m.obc_minmax_grid(W, bits, symmetric, scale, zero)
    grid = dict(mode="quant", scale=scale.cpu().numpy().astype(np.float64), zero=zero.cpu().numpy().astype(np.float64), maxq=maxq)
    free = fp64_rows(Hinv.cpu().numpy(), W.cpu().numpy(), **grid)["order"]
    for pending in (0, 16):                         # few updates per pass: other roundings, so other ties
        m.obc_quantize(W, Hinv, scale, zero, bits, symmetric, Wq, codes, st, loss=loss, qorder=order, opts=m.engine_opts(m.ENGINE_BLOCKED, 0, pending))
        torch.cuda.synchronize()
        assert int(st.abs().sum()) == 0
        P = order.cpu().numpy()
        s = check_rows(Hinv.cpu().numpy(), W.cpu().numpy(), P, loss.cpu().numpy(), gpu_w=Wq.cpu().numpy(), gpu_codes=codes.cpu().numpy(), **grid)
        part = (P != free).any(axis=1)              # rows that leave the order of FP64 -- at a tie, as check_rows has shown
        s.update(rows=rows, rows_that_part=int(part.sum()), first_parting=[int(x) for x in (P != free)[part].argmax(axis=1)],
                 gap_there=[float(s["oracle"]["forced_gap"][r, (P[r] != free[r]).argmax()]) for r in np.flatnonzero(part)])
        record_stats(f"OBQ {rows} x {d}, {bits} bits, max_pending {pending}", s)
        assert s["codes_differ"] == 0


@pytest.mark.gpu
def test_prune_trace_and_replay(gpu_reference):
    import paper_2208_11580_b200 as m
    rows, d = 2, 5000
    Hinv, W = layer(rows, d, d)
    order, loss, st = buffers(rows, d)
    trace = torch.zeros(rows, d + 1, d, device="cuda")
    m.obc_prune_trace(W, Hinv, order, loss, st, w_trace=trace)
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0
    s = check_rows(Hinv.cpu().numpy(), W.cpu().numpy(), order.cpu().numpy(), loss.cpu().numpy(), gpu_trace=trace.cpu().numpy())
    counts = torch.tensor([4321, 1234], dtype=torch.int32, device="cuda")
    out = torch.zeros(rows, d, device="cuda")
    m.obc_prune_apply(W, Hinv, order, counts, out, st)
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0
    for r, c in enumerate(counts.tolist()):
        want, top = s["oracle"]["w_trace"][r, c], float(W[r].abs().max())
        assert (np.abs(out[r].cpu().numpy() - want) / np.maximum(np.abs(want), top)).max() <= REL_TOL


@pytest.mark.gpu
def test_row_shares(gpu_reference):
    import paper_2208_11580_b200 as m
    d = 4608
    rows = torch.cuda.get_device_properties(0).multi_processor_count + 9
    Hinv, W = layer(rows, d, 1)
    order, loss, st = buffers(rows, d)
    m.obc_prune_trace(W, Hinv, order, loss, st)
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0
    some = [0, 1, 2, rows // 3, rows // 2, rows - 2, rows - 1]
    check_rows(Hinv.cpu().numpy(), W[some].cpu().numpy(), order[some].cpu().numpy(), loss[some].cpu().numpy())


@pytest.mark.gpu
def test_nm_and_blocks(gpu_reference):
    import paper_2208_11580_b200 as m
    rows, d = 3, 4608
    Hinv, W = layer(rows, d, 2)
    order, loss, st = buffers(rows, d)
    out = torch.zeros(rows, d, device="cuda")
    m.obc_prune_nm(W, Hinv, 2, 4, out, st, order=order, loss=loss)
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0
    check_rows(Hinv.cpu().numpy(), W.cpu().numpy(), order.cpu().numpy(), loss.cpu().numpy(), gpu_w=out.cpu().numpy(), steps=d // 2, nm=(2, 4))
    m.obc_prune_blocks(W, Hinv, order, loss, st, block=4)
    torch.cuda.synchronize()
    assert int(st.abs().sum()) == 0
    P, L = order.cpu().numpy(), loss.cpu().numpy().astype(np.float64)
    assert np.array_equal(P[:, ::4] % 4, np.zeros((rows, d // 4))) and np.array_equal(P[:, 3::4], P[:, ::4] + 3)
    want = fp64_rows(Hinv.cpu().numpy(), W.cpu().numpy(), forced=P)["loss"].reshape(rows, -1, 4).sum(-1)      # a block's score: the sum of its members' losses
    assert (np.abs(L[:, ::4] - want) <= REL_TOL * (want + 1e-7 * want.max(axis=1, keepdims=True))).all()
