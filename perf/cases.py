"""The work that is measured for speed: what programs have this library do, through its Python entry points.

Two kinds of program use it.  One prepares a model: it assesses every channel of every weight at 1, 2 and 4 bits, fits
codebooks, encodes, and takes residuals for a low-rank initialiser (`assess`, `fit`, `encode`, `residual`), or turns the
codes back into bf16 weights (`decode`).  The other runs the quantised layers: it trains the low-rank factors (`train`:
forward, input gradient, gradients of the factors) or serves them (`forward`, and `adapters` for several fine-tunes on one
base weight).  Shapes, precision mixes, token counts and ranks are those of the benchmark's workloads and of the tests:
linear layers of 512 to 13824 channels, 1.15 to 2.5 bits per weight (and uniform 4 bits), 1 to 8192 tokens, ranks 16 to 128.
"""
import math

import numpy as np
import torch

import paper_2502_08141_b200 as lw

# precision mixes: share of the output channels at each number of bits
MIXES = {
    "1:50 2:50": {1: 0.50, 2: 0.50},
    "1:30 2:50 4:20": {1: 0.30, 2: 0.50, 4: 0.20},
    "1:60 2:35 4:5": {1: 0.60, 2: 0.35, 4: 0.05},
    "1:85 2:15": {1: 0.85, 2: 0.15},
    "2:75 4:25": {2: 0.75, 4: 0.25},
    "4:100": {4: 1.0},
}

# levels near the quantiles of normalised weights, as a learner starts from (and, moved a little, as it ends)
LEVELS = {
    1: [-0.45, 0.45],
    2: [-0.75, -0.2, 0.25, 0.8],
    4: [-1.0, -0.7, -0.53, -0.4, -0.29, -0.19, -0.09, 0.0, 0.08, 0.16, 0.25, 0.34, 0.44, 0.56, 0.72, 1.0],
}


def listed():
    return [
        # a first call as the quick start makes it: a small layer, one short prompt, nothing kept between calls
        dict(name="serve_tiny", op="forward", N=512, K=512, mix="1:50 2:50", r=16, M=16, deal=False, natural=False),
        # generation for one user: one token at a time through an attention projection
        dict(name="serve_token", op="forward", N=4096, K=4096, mix="1:60 2:35 4:5", r=64, M=1, deal=True, natural=False),
        # a decode batch of several fine-tunes on one base weight: groups of a few tokens each
        dict(name="serve_adapters", op="adapters", N=4096, K=4096, mix="1:30 2:50 4:20", r=64, M=101, groups=6, natural=False),
        # a prompt of ordinary length through a wide layer, in the storage order other tools write
        dict(name="prefill", op="forward", N=11008, K=4096, mix="2:75 4:25", r=64, M=1000, deal=True, natural=True),
        # fine-tuning: the three attention projections of a layer together, half a batch of 4096 tokens
        dict(name="train_qkv", op="train", N=4096, K=4096, mix="1:30 2:50 4:20", r=64, M=2048, count=3, deal=True, reuse=True),
        # fine-tuning: the wide projection of a layer at a full batch - the bulk of a training step's time
        dict(name="train_mlp", op="train", N=11008, K=4096, mix="1:60 2:35 4:5", r=64, M=4096, count=1, deal=True, reuse=True),
        # fine-tuning a layer of odd size on a short, ragged batch, each call on its own
        dict(name="train_ragged", op="train", N=1800, K=2304, mix="1:50 2:50", r=48, M=777, count=1, deal=False, reuse=False),
        # preparing a model: codebooks at the assigned precisions, then the codes, one matrix
        dict(name="fit", op="fit", N=4096, K=4096, mix="1:60 2:35 4:5", iterations=10, natural=False),
        # quantising a layer's seven matrices whose thresholds are known (adapters that share them)
        dict(name="encode_layer", op="encode", N=11008, K=4096, mix="1:60 2:35 4:5", layer=True, natural=False),
        # unpacking a layer's seven matrices to bf16 (to merge, export or evaluate them)
        dict(name="decode_layer", op="decode", N=11008, K=4096, mix="2:75 4:25", layer=True, natural=False),
        # the precision assigner's input: every channel learnt at three precisions, and its error at each
        dict(name="assess", op="assess", N=4096, K=4096, iterations=2),
        # one round of an iterative low-rank initialiser: what quantisation leaves over of a weight
        dict(name="residual", op="residual", N=5120, K=5120, mix="1:85 2:15", natural=False),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _flops(c):
    """Multiply-adds of the products, twice: forward and input gradient, each with its two low-rank products, and the factors'
    gradients (which form both projections again where the calls before have not kept them)."""
    if c["op"] == "train":
        return c.get("count", 1) * (4.0 * c["M"] * c["N"] * c["K"] + (6.0 if c["reuse"] else 8.0) * c["M"] * c["r"] * (c["N"] + c["K"]))
    if c["op"] in ("forward", "adapters"):
        return 2.0 * c["M"] * c["N"] * c["K"] + 2.0 * c["M"] * c["r"] * (c["N"] + c["K"])
    return 0.0


def draw(rng):
    op = rng.choice(["forward", "forward", "adapters", "train", "train", "encode", "decode", "fit", "assess", "residual"])
    top = [c for c in listed() if c["name"] == "train_mlp"][0]
    while True:
        c = dict(op=op, K=128 * int(round(_log(rng, 4, 108))))
        if op in ("forward", "adapters", "train"):
            c.update(N=8 * int(round(_log(rng, 32, 1728))), mix=rng.choice(sorted(MIXES)), r=rng.choice([16, 32, 48, 64, 64, 64, 80, 128]),
                     M=int(round(_log(rng, 1, 8192))))
        else:
            c.update(N=int(round(_log(rng, 256, 13824))))
        if op == "forward":
            c.update(deal=rng.random() < 0.7, natural=rng.random() < 0.3)
        elif op == "adapters":
            c.update(groups=rng.randint(2, 9), natural=rng.random() < 0.3)
            c["M"] = max(c["M"], c["groups"])
        elif op == "train":
            c["deal"] = rng.random() < 0.7
            c["count"] = rng.choice([1, 1, 2, 3]) if c["deal"] else 1
            c["reuse"] = c["deal"] and rng.random() < 0.7
        elif op in ("encode", "decode"):
            c.update(mix=rng.choice(sorted(MIXES)), layer=rng.random() < 0.4, natural=rng.random() < 0.3)
        elif op == "fit":
            c.update(mix=rng.choice(sorted(MIXES)), iterations=rng.choice([2, 10]), natural=rng.random() < 0.3)
        elif op == "assess":
            c.update(iterations=rng.choice([2, 10]))
        else:
            c.update(mix=rng.choice(sorted(MIXES)), natural=rng.random() < 0.3)
        if op in ("forward", "adapters", "train"):
            fits = _flops(c) <= _flops(top)
        else:
            most = {"encode": 2.1e8, "decode": 2.1e8, "residual": 7e7, "fit": 4.6e7, "assess": 4.6e7 if c.get("iterations") == 2 else 1.7e7}
            fits = sum(n * k for n, k in _shapes(c)) <= most[op]
        if fits:
            return c


def _shapes(c):
    """(N, K) of every matrix of the case; a layer has four square projections, two wide ones and one back."""
    if not c.get("layer"):
        return [(c["N"], c["K"])] * c.get("count", 1)
    n, k = c["N"], c["K"]
    return [(n, k), (n, k), (k, n // 128 * 128)] + [(k, k)] * 4    # the largest first, as the group calls advise


# ---------------------------------------------------------------------------------------------- inputs
def _weights(N, K, gen):
    """Rows of different spread, one value in a thousand an outlier of a heavier-tailed kind."""
    sigma = torch.exp(math.log(0.005) + torch.rand((N, 1), device="cuda", generator=gen) * math.log(10.0))
    W = torch.randn((N, K), device="cuda", generator=gen)
    n = max(1, N * K // 1000)
    at = torch.randint(0, N * K, (n,), device="cuda", generator=gen)
    z = torch.randn((5, n), device="cuda", generator=gen)
    t4 = 10.0 * z[0] / torch.sqrt(z[1:].square().sum(0) / 4.0)
    at = torch.unique(at)    # a place drawn twice would take either value
    W.view(-1)[at] = t4[: at.numel()]
    return W.mul_(sigma)


def _precisions(N, mix, rng):
    bits = sorted(MIXES[mix])
    counts = [int(round(MIXES[mix][b] * N)) for b in bits]
    counts[counts.index(max(counts))] += N - sum(counts)
    return rng.permutation(np.repeat(np.array(bits, np.uint8), counts))


def _tables(precs, gen):
    """Per-channel levels around LEVELS and the thresholds halfway between them (fp32 [N, 16] each)."""
    N = precs.size
    p = torch.from_numpy(precs.astype(np.int64)).cuda()
    maps = torch.zeros((N, 16), device="cuda")
    thr = torch.full((N, 16), float("inf"), device="cuda")
    jitter = (torch.rand((N, 16), device="cuda", generator=gen) - 0.5) * 0.06
    for b, levels in LEVELS.items():
        rows = (p == b).nonzero().flatten()
        m = torch.tensor(levels, device="cuda") + jitter[rows, : len(levels)]
        maps[rows, : len(levels)] = m
        thr[rows, : len(levels) - 1] = (0.5 * (m[:, :-1].double() + m[:, 1:].double())).float()
    return maps, thr


def _bf16(shape, scale, gen):
    return (torch.randn(shape, device="cuda", generator=gen) * scale).to(torch.bfloat16)


def _start():
    """The learner's starting tables: host float64 [3, 16] (1, 2, 4 bits)."""
    y0, t0 = np.zeros((3, 16)), np.zeros((3, 16))
    for row, b in enumerate((1, 2, 4)):
        y = np.array(LEVELS[b])
        y0[row, : y.size] = y
        t0[row, : y.size - 1] = 0.5 * (y[:-1] + y[1:])
    return y0, t0


def _weight(N, K, mix, natural, rng, gen, keep=()):
    """One quantised weight as a program holds it, and those of W / thresholds that it still needs."""
    precs = _precisions(N, mix, rng)
    layout = lw.Layout(precs, K, natural=natural)
    maps, thr = _tables(precs, gen)
    W = _weights(N, K, gen)
    w = dict(layout=layout, maps=maps)
    if "codes" in keep:
        w["packed"], w["absmax"] = lw.lowra_encode(layout, W, thr)
    if "W" in keep:
        w["W"], w["thresholds"] = W, thr
    return w


def prepare(case, seed):
    op = case["op"]
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    natural = case.get("natural", False)
    s = dict(op=op, case=case)
    if op == "assess":
        s["W"] = _weights(case["N"], case["K"], gen)
        s["start"] = _start()
        return s
    keep = ("codes",) if op in ("forward", "adapters", "train", "decode") else ("W",)
    s["weights"] = [_weight(n, k, case["mix"], natural, rng, gen, keep) for n, k in _shapes(case)]
    if op == "fit":
        s["start"] = _start()
    if op not in ("forward", "adapters", "train"):
        return s
    N, K, M, r = case["N"], case["K"], case["M"], case["r"]
    n = case.get("groups", 1)
    w = s["weights"][0]
    if case.get("deal", True):
        for x in s["weights"]:
            x["layout"].build_deal()
    s["X"] = _bf16((M, K), 1.0, gen)
    factors = [(_bf16((K, r), 0.01, gen), _bf16((r, N), 0.01, gen)) for _ in range(max(n, len(s["weights"])))]
    if op == "forward":
        s["A"], s["B"] = factors[0]
        if case["deal"]:
            s["ws"] = _workspace(lw.lowra_workspace_bytes(w["layout"], M, r))
    elif op == "adapters":
        cuts = np.sort(rng.choice(np.arange(1, M), n - 1, replace=False)) if M > 1 else []
        s["start"] = np.concatenate([[0], cuts, [M]]).astype(np.int32)
        s["A"], s["B"] = (torch.stack([f[i] for f in factors]) for i in (0, 1))
        s["maps"] = torch.stack([_tables(w["layout"].precs_host, gen)[0] for _ in range(n)])   # each adapter has its own levels
        s["ws"] = _workspace(lw.lowra_batch_workspace_bytes(w["layout"], 4, M, r))
    else:
        s["dY"] = [_bf16((M, N), 1.0, gen) for _ in s["weights"]]
        s["factors"] = factors
        if case["deal"]:    # forward and input gradient keep a workspace each: both projections are needed afterwards
            size = lw.lowra_batch_workspace_bytes(w["layout"], len(s["weights"]), M, r)
            s["ws_f"], s["ws_b"] = _workspace(size), _workspace(size)
    return s


def _workspace(size):
    return lw.lowra_workspace_init(torch.empty(size, dtype=torch.uint8, device="cuda"))


# ---------------------------------------------------------------------------------------------- one pass
SCALE = 2.0


def run(s):
    op, case = s["op"], s["case"]
    if op == "assess":
        maps3, thr3 = lw.lowra_learn_codebooks_all(s["W"], *s["start"], case["iterations"])
        return maps3, thr3, lw.lowra_channel_errors(s["W"], maps3, thr3)
    ws = s["weights"]
    w = ws[0]
    if op == "forward":
        return lw.lowra_lora_forward(w["layout"], w["packed"], w["absmax"], w["maps"], s["X"], s["A"], s["B"], SCALE, workspace=s.get("ws"))
    if op == "adapters":
        return lw.lowra_lora_forward_adapters(w["layout"], w["packed"], w["absmax"], s["maps"], s["X"], s["start"], s["A"], s["B"], SCALE,
                                              workspace=s["ws"])
    if op == "train":
        return _train(s)
    if op == "fit":
        maps, thr = lw.lowra_learn_codebooks(w["layout"], w["W"], *s["start"], case["iterations"])
        return maps, thr, lw.lowra_encode(w["layout"], w["W"], thr)
    if op == "encode":
        if len(ws) == 1:
            return lw.lowra_encode(w["layout"], w["W"], w["thresholds"])
        return lw.lowra_encode_group(ws)
    if op == "decode":
        if len(ws) == 1:
            return lw.lowra_decode(w["layout"], w["packed"], w["absmax"], w["maps"])
        return lw.lowra_decode_group(ws)
    return lw.lowra_quant_error(w["layout"], w["W"], w["maps"], w["thresholds"], want_residual=True)


def _train(s):
    """A training step of one linear module, or of several that read the same input: outputs, input gradients, gradients of
    the low-rank factors."""
    case, ws, X, dY, factors = s["case"], s["weights"], s["X"], s["dY"], s["factors"]
    M, r = case["M"], case["r"]
    ws_f, ws_b = s.get("ws_f"), s.get("ws_b")
    if len(ws) == 1:
        w, (A, B) = ws[0], factors[0]
        Y = [lw.lowra_lora_forward(w["layout"], w["packed"], w["absmax"], w["maps"], X, A, B, SCALE, workspace=ws_f)]
        dX = [lw.lowra_lora_backward_input(w["layout"], w["packed"], w["absmax"], w["maps"], dY[0], A, B, SCALE, workspace=ws_b)]
    else:
        one = lambda i, act, cols: dict(layout=ws[i]["layout"], packed=ws[i]["packed"], absmax=ws[i]["absmax"], maps=ws[i]["maps"],  # noqa: E731
                                        act=act, A=factors[i][0], B=factors[i][1],
                                        out=torch.empty((M, cols), dtype=torch.bfloat16, device="cuda"))
        Y = lw.lowra_lora_forward_batch([one(i, X, case["N"]) for i in range(len(ws))], SCALE, ws_f)
        dX = lw.lowra_lora_backward_input_batch([one(i, dY[i], case["K"]) for i in range(len(ws))], SCALE, ws_b)
    if case["reuse"]:
        grads = [lw.lowra_lora_backward_adapters_reuse(X, dY[i], lw.lowra_workspace_projection(ws_f, M, r, i),
                                                       lw.lowra_workspace_projection(ws_b, M, r, i), r) for i in range(len(ws))]
    else:
        grads = [lw.lowra_lora_backward_adapters(X, dY[i], *factors[i], SCALE) for i in range(len(ws))]
    return dict(Y=Y, dX=dX, grads=grads)


# ---------------------------------------------------------------------------------------------- what it costs at least
def _bits(mix):
    return sum(b * f for b, f in MIXES[mix].items())


def work(case):
    """Inputs read once, outputs written once; products at two operations a multiply-add."""
    op = case["op"]
    total = 0.0
    for n, k in _shapes(case):
        codes = n * k * (_bits(case["mix"]) / 8 + 4 / 64) if "mix" in case else 0.0
        tables = 64.0 * n                                          # 16 fp32 entries a channel
        if op in ("forward", "train", "adapters"):
            a = case.get("groups", 1)
            M, r = case["M"], case["r"]
            total += codes + tables * a + 2.0 * r * (n + k) * a + 2.0 * M * (n + k)
            if op == "train":                                      # dY in, dX and both gradients out
                total += 2.0 * M * (n + k) + 2.0 * r * (n + k)
        elif op == "encode":
            total += 4.0 * n * k + tables + codes
        elif op == "decode":
            total += codes + tables + 2.0 * n * k
        elif op == "fit":
            total += 4.0 * n * k + 2 * tables + codes
        elif op == "assess":
            total += 4.0 * n * k + 6 * tables + 24.0 * n
        else:
            total += 8.0 * n * k + 2 * tables + 8.0 * n
    return {"bytes": total, "flops": _flops(case)}


def tolerance(case):
    op = case["op"]
    if op in ("encode", "decode"):
        return "exact"                     # codes, block maxima and bf16 weights are defined bit for bit
    if op == "residual":
        return {"rel": 1e-6, "max": 2e-6}  # the residual is exact; the error is a sum of squares good to 2^-21
    if op == "assess":
        return {"rel": 1e-5, "max": 1e-3}  # as for fit, and the errors follow the tables
    if op == "fit":
        # fp64 sums rounded to fp32 once: a last-bit step here and there, and a code where a weight sits between two such thresholds
        return {"rel": 1e-6, "max": 1e-4, "differ": 1e-5}
    # fp32 sums in any order, rounded to bf16 (unit 2^-8); the projections between the factors are rounded once more
    return {"rel": 5e-3, "max": 0.02}
