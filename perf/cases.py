"""Performance cases of the layer solver: what a compression run asks of it, layer by layer.

Every case is one pass through the package's public entry points on inputs that live on the GPU.  The shapes are those
of the repository's own workloads (convolutions unfolded to d_col = 9 x channels, BERT-base linear layers) and of the
other layers that the same networks have.  Kinds:

  layer    calibration inputs in hand: Hessian, inverse, pruning trace, global mask, final weights (and, with `bits`,
           the layer's OBQ codes on the same inverse): the whole of one small layer
  prune    inverse Hessian in hand: pruning trace, a global mask and the final weights for each sparsity
  quant    inverse Hessian in hand: OBQ of every row on a min-max grid
  compound inverse Hessian in hand: pruning trace, global mask, replay of the pruning and OBQ of the survivors
  nm       inverse Hessian in hand: N:M pruning
  blocks   inverse Hessian in hand: block pruning, global mask, final weights by forced-order replay
  hessian  one more chunk of the calibration axis is added to a layer's Hessian
  refit    sequential compression: Hessian and inverse of the compressed model's inputs, cross products with the dense
           outputs, refitted dense weights
  levels   loss traces in hand: the global masks of several sparsity levels (a model database stores many of them)

A program prepares a layer's inverse Hessian once and solves several compression problems on it, so the kinds from
`prune` to `blocks` start from it.  It is computed here with torch in FP64, so that the inputs depend on the seed alone.
"""
import math

import torch
import torch.nn.functional as F

import paper_2208_11580_b200 as obc

DAMP = 0.01                       # relative dampening of the Hessian, as in every workload of the repository
PREC = {"fp32": obc.PREC_FP32, "tf32": obc.PREC_TF32, "bf16x3": obc.PREC_BF16X3}


def listed():
    return [
        # A tiny linear layer from its inputs to a 50 % mask and 4-bit codes, Hessian in the default precision: all
        # latency and launches.
        {"name": "tiny_linear_layer", "kind": "layer", "d_row": 32, "d_col": 64, "n": 1024, "acts": "correlated", "prec": "fp32",
         "sparsity": 0.5, "bits": 4, "symmetric": True},
        # An early ResNet-18 3x3 convolution (64 -> 64) pruned to 60 % from its inputs: fewer rows than SMs.
        {"name": "conv64_prune_layer", "kind": "layer", "d_row": 64, "d_col": 576, "n": 16384, "acts": "relu_conv", "prec": "bf16x3",
         "sparsity": 0.6, "bits": 0, "symmetric": False},
        # A ResNet-50 bottleneck 3x3 convolution (256 -> 256), OBQ to 4 bits on an asymmetric grid.
        {"name": "conv256_quant4", "kind": "quant", "d_row": 256, "d_col": 2304, "n": 32768, "acts": "abs_conv", "bits": 4,
         "symmetric": False, "outliers": False},
        # BERT-base FFN up-projection: 50 % pruning and 8-bit codes for the rest (many short rows).
        {"name": "ffn_up_compound", "kind": "compound", "d_row": 3072, "d_col": 768, "n": 65536, "acts": "layernorm", "sparsity": 0.5,
         "bits": 8, "symmetric": True},
        # BERT-base FFN down-projection: full pruning trace with the weight trace kept, three of a model database's levels.
        {"name": "ffn_down_prune", "kind": "prune", "d_row": 768, "d_col": 3072, "n": 65536, "acts": "gelu", "trace": True,
         "sparsity": 0.2, "sparsity_step": 0.1, "masks": 3},
        # A last-block ResNet 3x3 convolution (512 -> 512, the longest rows of these networks): one GPU's share of its
        # rows when the layer is split over four.
        {"name": "conv512_quant4_share", "kind": "quant", "d_row": 128, "d_col": 4608, "n": 16384, "acts": "abs_conv", "bits": 4,
         "symmetric": True, "outliers": False},
        # A BERT-base attention projection pruned 2:4.
        {"name": "attention_2to4", "kind": "nm", "d_row": 768, "d_col": 768, "n": 16384, "acts": "layernorm", "n_keep": 2, "m_block": 4},
        # A ResNet-18 3x3 convolution (128 -> 128) pruned in blocks of 4 to 50 %, final weights by replay.
        {"name": "conv128_blocks4", "kind": "blocks", "d_row": 128, "d_col": 1152, "n": 16384, "acts": "relu_conv", "block": 4, "sparsity": 0.5},
        # The largest calibration set: 128 sequences of 512 tokens into the 3072 x 3072 Hessian.
        {"name": "hessian_ffn_down", "kind": "hessian", "d_col": 3072, "n": 65536, "acts": "gelu", "prec": "bf16x3"},
        # The ResNet stem (7x7x3 patches): ragged d_col, a long calibration axis (4 images, the last one cut), default
        # precision.
        {"name": "hessian_stem", "kind": "hessian", "d_col": 147, "n": 50173, "acts": "correlated", "prec": "fp32"},
        # The ResNet-50 classifier (2048 -> 1000) refitted to a compressed model's inputs.
        {"name": "classifier_refit", "kind": "refit", "d_row": 1000, "d_col": 2048, "n": 8192, "acts": "relu", "prec": "bf16x3"},
        # Nine masks, 10 % to 90 %, from the traces of the BERT-base FFN up-projection.
        {"name": "ffn_up_levels", "kind": "levels", "d_row": 3072, "d_col": 768, "sparsity": 0.1, "sparsity_step": 0.1, "masks": 9},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _engine_rows(rng, d, most=3072):
    """A number of rows whose elimination costs no more than the largest listed layer's (work grows as rows * d^3)."""
    return _log_int(rng, 16, max(17, min(most, int(0.3 * 768 * (3072 / d) ** 3))))


def draw(rng):
    kind = rng.choice(["layer", "prune", "quant", "quant", "compound", "nm", "blocks", "hessian", "hessian", "refit", "levels"])
    acts = rng.choice(["relu", "relu_conv", "abs_conv", "layernorm", "gelu"])
    if kind == "layer":
        d = _log_int(rng, 48, 600)
        return {"kind": kind, "d_row": _log_int(rng, 16, 512), "d_col": d, "n": _log_int(rng, 2 * d, 32768), "acts": rng.choice([acts, "correlated"]),
                "prec": rng.choice(sorted(PREC)), "sparsity": round(rng.uniform(0.2, 0.5), 3), "bits": rng.choice([0, 4, 8]),
                "symmetric": rng.random() < 0.5}
    if kind == "hessian":
        d = _log_int(rng, 64, 3072)
        return {"kind": kind, "d_col": d, "n": _log_int(rng, 1024, 65536), "acts": acts, "prec": rng.choice(sorted(PREC))}
    if kind == "refit":
        d = _log_int(rng, 64, 2304)
        return {"kind": kind, "d_row": _log_int(rng, 32, 2304), "d_col": d, "n": _log_int(rng, 2 * d, 16384), "acts": acts,
                "prec": rng.choice(["bf16x3", "fp32"])}
    if kind == "levels":
        return {"kind": kind, "d_row": _log_int(rng, 32, 3072), "d_col": _log_int(rng, 64, 2304), "sparsity": 0.05, "sparsity_step": round(rng.uniform(0.05, 0.1), 3),
                "masks": rng.randint(1, 9)}
    d = _log_int(rng, 64, 4608)
    if kind == "nm":
        m = rng.choice([4, 4, 8])
        d = max(m, d // m * m)
        return {"kind": kind, "d_row": _engine_rows(rng, d), "d_col": d, "n": _log_int(rng, 2 * d, 16384), "acts": acts, "n_keep": m // 2, "m_block": m}
    if kind == "blocks":
        c = rng.choice([4, 4, 4, 8])
        d = max(c, min(d, 3072) // c * c)
        return {"kind": kind, "d_row": _engine_rows(rng, d, 512), "d_col": d, "n": _log_int(rng, 2 * d, 16384), "acts": acts, "block": c,
                "sparsity": round(rng.uniform(0.2, 0.5), 3)}
    case = {"kind": kind, "d_row": _engine_rows(rng, d), "d_col": d, "n": _log_int(rng, 2 * d, 16384), "acts": acts}
    if kind == "prune":
        case.update(trace=d <= 1024 and rng.random() < 0.5, sparsity=round(rng.uniform(0.1, 0.2), 3), sparsity_step=0.1, masks=rng.randint(1, 3))
    if kind == "quant":
        case.update(bits=rng.choice([4, 4, 8]), symmetric=rng.random() < 0.5, outliers=rng.random() < 0.25)
    if kind == "compound":
        case.update(bits=rng.choice([4, 8]), symmetric=rng.random() < 0.5, sparsity=round(rng.uniform(0.2, 0.5), 3))
    return case


# ---- inputs --------------------------------------------------------------------------------------------------------
def _matrix(rows, cols):
    """rows x cols FP32 with a leading dimension that is a multiple of 4 (what the entry points ask for)."""
    return torch.zeros(rows, (cols + 3) // 4 * 4, device="cuda")[:, :cols]


def _activations(acts, d, n, g):
    """A d x n chunk of calibration inputs."""
    X = _matrix(d, n)
    if acts in ("relu_conv", "abs_conv"):          # im2col of a rectified feature map, 3x3 patches
        c = -(-d // 9)
        hw, stride = (56, 2) if acts == "relu_conv" else (14, 1)
        per = ((hw - 1) // stride + 1) ** 2
        done = 0
        while done < n:                            # (a few images at a time)
            imgs = min(-(-(n - done) // per), 32)
            a = torch.randn(imgs, c, hw, hw, device="cuda", generator=g)
            a = a.relu_() if acts == "relu_conv" else a.abs_()
            u = F.unfold(a, 3, padding=1, stride=stride).transpose(0, 1).reshape(9 * c, imgs * per)[:d]
            m = min(imgs * per, n - done)
            X[:, done:done + m] = u[:, :m]
            done += m
        return X
    mix = None
    heavy = None
    if acts == "correlated":                       # covariance A A^T + 0.1 I
        a = torch.randn(d, d, device="cuda", generator=g, dtype=torch.float64)
        mix = torch.linalg.cholesky(a @ a.T + 0.1 * torch.eye(d, device="cuda", dtype=torch.float64)).float()
    elif acts in ("relu", "gelu"):                 # a hidden layer's outputs
        k = max(16, d // 4) if acts == "gelu" else d
        mix = torch.randn(d, k, device="cuda", generator=g) / math.sqrt(k)
    else:                                          # layer norm with a few heavy-tailed channels
        heavy = torch.randperm(d, device="cuda", generator=g)[:max(1, d // 128)]
    for b in range(0, n, 8192):
        e = min(n, b + 8192)
        z = torch.randn(d if mix is None else mix.shape[1], e - b, device="cuda", generator=g)
        if mix is not None:
            z = mix @ z
            z = F.relu(z) if acts == "relu" else F.gelu(z) if acts == "gelu" else z
        else:                                      # Student-t with 3 degrees of freedom
            chi = torch.randn(3, len(heavy), e - b, device="cuda", generator=g).square().sum(0) / 3
            z[heavy] /= chi.sqrt()
            z = (z - z.mean(0)) / (z.var(0, unbiased=False) + 1e-12).sqrt()
        X[:, b:e] = z
    return X


def _weights(rows, d, g):
    W = _matrix(rows, d)
    W.copy_(torch.randn(rows, d, device="cuda", generator=g) * math.sqrt(2.0 / d))
    return W


def _inverse_hessian(case, g):
    d = case["d_col"]
    X = _activations(case["acts"], d, case["n"], g)
    H = torch.zeros(d, d, device="cuda", dtype=torch.float64)
    for b in range(0, case["n"], 8192):
        x = X[:, b:b + 8192].double()
        H.addmm_(x, x.T, alpha=2.0)
    H.diagonal().add_(DAMP * H.diagonal().mean())
    inv = torch.cholesky_inverse(torch.linalg.cholesky(H))
    Hinv = _matrix(d, d)
    Hinv.copy_((inv + inv.T) * 0.5)
    return Hinv


def _workspace(*needs):
    return torch.empty(max(needs), dtype=torch.uint8, device="cuda")


def _levels(case):
    """The numbers of pruned weights of the case's sparsity levels."""
    c = case.get("block", 1)
    s = [case["sparsity"] + i * case.get("sparsity_step", 0.0) for i in range(case.get("masks", 1))]
    return [int(round(min(x, 0.95) * case["d_row"] * case["d_col"])) // c * c for x in s]


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind, d = case["kind"], case["d_col"]
    R = case.get("d_row", 0)
    s = {"case": case}
    if kind == "hessian":
        s["X"] = _activations(case["acts"], d, case["n"], g)
        s["H"] = _matrix(d, d)                     # what earlier chunks have accumulated (every pass adds to it)
        x = s["X"][:, :1024]
        s["H"].copy_(2.0 * x @ x.T)
        s["ws"] = _workspace(obc.obc_workspace_bytes(obc.OP_HESSIAN, 0, d, case["n"]))
        return s
    if kind == "levels":                           # losses that grow along a row, not monotonically
        s["loss"] = torch.rand(R, d, device="cuda", generator=g).square_().mul_(1e-4)
        s["loss"] += torch.linspace(0, 1, d, device="cuda").pow(4) * (0.5 + torch.rand(R, 1, device="cuda", generator=g))
        s["order"] = torch.rand(R, d, device="cuda", generator=g).argsort(1).int()
    if kind in ("layer", "refit"):
        s["X"] = _activations(case["acts"], d, case["n"], g)
        s["H"], s["Hinv"] = _matrix(d, d), _matrix(d, d)
        s["info"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        needs = [obc.obc_workspace_bytes(obc.OP_HESSIAN, 0, d, case["n"]), obc.obc_workspace_bytes(obc.OP_INVERSE, 0, d)]
    elif kind != "levels":
        s["Hinv"] = _inverse_hessian(case, g)
    if kind == "refit":                            # outputs of the dense layer on the dense model's inputs
        W = _weights(R, d, g)
        s["Y"] = _matrix(R, case["n"])
        s["Y"].copy_(W @ s["X"])
        s["Y"] += 0.05 * s["Y"].std() * torch.randn(R, case["n"], device="cuda", generator=g)
        s["G"], s["W_out"] = _matrix(R, d), _matrix(R, d)
        s["ws"] = _workspace(*needs, obc.obc_workspace_bytes(obc.OP_CROSS_GRAM, R, d, case["n"]), obc.obc_workspace_bytes(obc.OP_REFIT, R, d))
        return s
    if kind != "levels":
        s["W"] = _weights(R, d, g)
        s["status"] = torch.zeros(R, dtype=torch.int32, device="cuda")
    pruning = kind in ("layer", "prune", "compound", "blocks")
    if pruning:
        s["order"] = torch.zeros(R, d, dtype=torch.int32, device="cuda")
        s["loss"] = torch.zeros(R, d, device="cuda")
    if pruning or kind == "levels":
        s["ks"] = _levels(case)
        s["counts"] = [torch.zeros(R, dtype=torch.int32, device="cuda") for _ in s["ks"]]
        s["masks"] = [torch.zeros(R, d, dtype=torch.uint8, device="cuda") for _ in s["ks"]]
    if kind in ("layer", "prune", "blocks"):
        s["pruned"] = [_matrix(R, d) for _ in s["ks"]]
    s["trace"] = torch.empty(R, d + 1, d, device="cuda") if kind == "layer" or case.get("trace") else None
    if case.get("bits"):
        s["scale"], s["zero"] = torch.zeros(R, device="cuda"), torch.zeros(R, device="cuda")
        s["W_out"], s["codes"] = _matrix(R, d), torch.zeros(R, d, dtype=torch.int32, device="cuda")
        s["qloss"], s["qorder"] = torch.zeros(R, d, device="cuda"), torch.zeros(R, d, dtype=torch.int32, device="cuda")
    if kind == "nm":
        s["W_out"], s["mask"] = _matrix(R, d), torch.zeros(R, d, dtype=torch.uint8, device="cuda")
        s["order"], s["loss"] = torch.zeros(R, d, dtype=torch.int32, device="cuda"), torch.zeros(R, d, device="cuda")
    if kind == "levels":
        s["ws"] = _workspace(obc.obc_workspace_bytes(obc.OP_SELECT, R, d))
        return s
    engine = obc.OP_PRUNE_BLOCKS if kind == "blocks" else obc.OP_QUANTIZE if kind == "quant" else obc.OP_PRUNE_TRACE
    s["ws"] = _workspace(obc.obc_workspace_bytes(engine, R, d), obc.obc_workspace_bytes(obc.OP_PRUNE_APPLY, R, d),
                         obc.obc_workspace_bytes(obc.OP_QUANTIZE, R, d), obc.obc_workspace_bytes(obc.OP_SELECT, R, d),
                         *(needs if kind == "layer" else []))
    return s


# ---- one pass ------------------------------------------------------------------------------------------------------
def _front(s, case):
    obc.obc_hessian(s["X"], s["H"], prec=PREC[case["prec"]], ws=s["ws"])
    obc.obc_hessian_inverse(s["H"], DAMP, Hinv=s["Hinv"], info=s["info"], ws=s["ws"])


def _masks(s):
    for k, counts, mask in zip(s["ks"], s["counts"], s["masks"]):
        obc.obc_select_global_mask(s["loss"], s["order"], k, counts, mask, ws=s["ws"])


def _final_weights(s, case):
    for counts, out in zip(s["counts"], s["pruned"]):
        obc.obc_prune_apply(s["W"], s["Hinv"], s["order"], counts, out, s["status"], w_trace=s["trace"],
                            trace_steps=case["d_col"] if s["trace"] is not None else 0, ws=s["ws"])


def _obq(s, case):
    obc.obc_minmax_grid(s["W"], case["bits"], case["symmetric"], s["scale"], s["zero"])
    obc.obc_quantize(s["W"], s["Hinv"], s["scale"], s["zero"], case["bits"], case["symmetric"], s["W_out"], s["codes"], s["status"],
                     flags=obc.FLAG_OUTLIERS if case.get("outliers") else 0, loss=s["qloss"], qorder=s["qorder"], ws=s["ws"])


def _outputs(s, *names):
    return {k: s[k] for k in names}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "hessian":
        obc.obc_hessian(s["X"], s["H"], accumulate=True, prec=PREC[case["prec"]], ws=s["ws"])
        return _outputs(s, "H")
    if kind == "levels":
        _masks(s)
        return _outputs(s, "counts", "masks")
    if kind == "refit":
        _front(s, case)
        obc.obc_cross_gram(s["Y"], s["X"], s["G"], prec=PREC[case["prec"]], ws=s["ws"])
        obc.obc_refit(s["G"], s["Hinv"], s["W_out"], prec=PREC[case["prec"]], ws=s["ws"])
        return _outputs(s, "H", "Hinv", "G", "W_out", "info")
    if kind == "nm":
        obc.obc_prune_nm(s["W"], s["Hinv"], case["n_keep"], case["m_block"], s["W_out"], s["status"], order=s["order"], loss=s["loss"],
                         mask=s["mask"], ws=s["ws"])
        return _outputs(s, "W_out", "mask", "order", "loss", "status")
    if kind == "quant":
        _obq(s, case)
        return _outputs(s, "W_out", "codes", "scale", "zero", "qorder", "qloss", "status")
    if kind == "layer":
        _front(s, case)
    if kind == "blocks":
        obc.obc_prune_blocks(s["W"], s["Hinv"], s["order"], s["loss"], s["status"], block=case["block"], ws=s["ws"])
    else:
        obc.obc_prune_trace(s["W"], s["Hinv"], s["order"], s["loss"], s["status"], w_trace=s["trace"], ws=s["ws"])
    _masks(s)
    if kind == "compound":
        obc.obc_quantize(s["W"], s["Hinv"], s["scale"], s["zero"], case["bits"], case["symmetric"], s["W_out"], s["codes"], s["status"],
                         prune_order=s["order"], prune_counts=s["counts"][0], ws=s["ws"])
        return _outputs(s, "W_out", "codes", "scale", "zero", "order", "loss", "masks", "status")
    _final_weights(s, case)
    names = ["pruned", "order", "loss", "masks", "status"]
    if kind == "layer":
        names += ["H", "Hinv", "info"]
        if case["bits"]:
            _obq(s, case)
            names += ["W_out", "codes", "scale", "zero", "qorder", "qloss"]
    return _outputs(s, *names)


# ---- what a pass cannot do without -----------------------------------------------------------------------------------
def _eliminations(d, first, last):
    """Flops of the rank-1 updates of a row's inverse (lower triangle, one multiply and one add per element) while its
    size falls from `first` to `last`."""
    return (first ** 3 - last ** 3) / 3.0


def work(case):
    kind, d, R = case["kind"], case["d_col"], case.get("d_row", 0)
    n, mat, square = case.get("n", 0), 4.0 * R * d, 4.0 * d * d
    if kind == "hessian":
        return {"bytes": 4.0 * d * n + 3 * square, "flops": 1.0 * n * d * (d + 1)}
    if kind == "refit":
        return {"bytes": 4.0 * n * (R + d) + 2 * square + 2 * mat,
                "flops": 1.0 * n * d * (d + 1) + 1.0 * d ** 3 + 2.0 * R * d * n + 2.0 * R * d * d}
    ks = _levels(case) if "sparsity" in case else []
    masks = len(ks) * (4.0 * R + 1.0 * R * d)
    if kind == "levels":
        return {"bytes": 2 * mat + masks, "flops": 1.0 * R * d * len(ks)}
    if kind == "nm":
        return {"bytes": square + 4 * mat + R * d, "flops": R * _eliminations(d, d, d * case["n_keep"] // case["m_block"])}
    if kind == "quant":
        return {"bytes": square + 5 * mat, "flops": R * _eliminations(d, d, 0)}
    # a pruning trace (order, loss) with masks and the final weights of every level
    nbytes, flops = square + 3 * mat + masks + len(ks) * mat, R * _eliminations(d, d, 0)
    if kind == "compound":
        left = d - ks[0] / R
        return {"bytes": nbytes + mat, "flops": flops + R * (_eliminations(d, d, left) + _eliminations(d, left, 0))}
    if kind == "blocks" or (kind == "prune" and not case["trace"]):
        flops += sum(R * _eliminations(d, d, d - k / R) for k in ks)
    if kind == "layer":
        nbytes += 4.0 * d * n + square
        flops += 1.0 * n * d * (d + 1) + 1.0 * d ** 3
        if case["bits"]:
            nbytes, flops = nbytes + 4 * mat, flops + R * _eliminations(d, d, 0)
    if kind == "layer" or case.get("trace"):
        nbytes += 4.0 * R * (d + 1) * d
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "levels":
        return "exact"
    if kind == "hessian":      # sums of FP32 products, of products of split BF16 values, of TF32 values (11 significant bits)
        return {"rel": 1e-3 if case["prec"] == "tf32" else 1e-5}
    if kind == "refit":        # the same sums times an inverse that amplifies their rounding
        return {"rel": 1e-3}
    # The greedy order is a sequence of comparisons: where two candidates tie to FP32 rounding, correct implementations
    # part ways in that row, and its later picks and codes follow other, equally good, paths (measured between settings of
    # the engine that differ in the order of roundings only: up to 0.3 % of the picks of a long layer, 0.6 % in the weights).
    return {"rel": 2e-2, "max": 0.99, "differ": 0.01}
