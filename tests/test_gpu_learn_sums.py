"""What the learner's fixed-point sums must not lose, and what they must not cost.

A level next to zero is as good as fp64 sums give it, also in rows whose weights differ widely; and rows of few different values
(ternary, rounded, pruned weights) take about the time of any other row.
"""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_learn_rows import _start

pytestmark = pytest.mark.gpu


def _cancelling_rows(K, heavy):
    """Rows whose middle 4-bit buckets hold pairs of values that nearly cancel; one block is `heavy` times the others."""
    rng = np.random.default_rng(K)
    W = np.empty((12, K), np.float32)
    for r in range(W.shape[0]):
        v = rng.uniform(0.004, 0.035, K // 2)
        x = np.stack([v, -v * (1.0 - 10.0 ** rng.uniform(-7, -4))], 1).reshape(-1)
        x[::64], x[1::64] = 1.0, -1.0                        # every block's absmax
        x *= np.repeat(rng.uniform(0.5, 1.0, K // 64), 64)
        x[64:128] *= heavy
        W[r] = x
    return W


@pytest.mark.parametrize("heavy", [1.0, 1e3, 1e6])
@pytest.mark.parametrize("K", [1024, 4096, 8192, 16512])
def test_levels_next_to_zero(K, heavy):
    import paper_2502_08141_b200 as lw

    W = _cancelling_rows(K, heavy)
    y0, t0 = _start()
    precs = np.full(W.shape[0], 4, np.uint8)
    Wd = torch.from_numpy(W).cuda()
    for T in (1, 3):
        maps, _ = lw.lowra_learn_codebooks(lw.Layout(precs, K), Wd, y0, t0, T)
        maps3, _ = lw.lowra_learn_codebooks_all(Wd, y0, t0, T)
        assert torch.equal(maps, maps3[2])
        ref, _ = oracle.lloyd_max(W, precs, T=T)
        ref = ref.astype(np.float64)
        # both are rounded to fp32 once, this one from means good to 2^-24; the oracle's fp64 sums of K products, which cancel to 1e-7 of the
        # sum of their magnitudes at most, to far less
        assert np.all(np.abs(maps.cpu().numpy() - ref) <= 3 * 2.0 ** -24 * np.abs(ref)), (T, heavy)
        assert (np.abs(ref[:, 7]) < 1e-4).any()


@pytest.mark.parametrize("K", [1024, 8192, 16512])
def test_weights_below_the_grid(K):
    """Buckets whose elements all lie in blocks 2^-60 to 2^-100 as heavy as the row's heaviest still get their mean."""
    import paper_2502_08141_b200 as lw

    rng = np.random.default_rng(K + 1)
    W = np.zeros((6, K), np.float32)
    for r in range(6):
        x = np.sign(rng.standard_normal(K)) * rng.uniform(0.95, 1.0, K)             # the outermost buckets, heavy
        light = np.repeat(rng.random(K // 64) < 0.5, 64)
        x[light] = rng.uniform(-0.85, 0.85, light.sum()) * 2.0 ** -(60.0 + 8.0 * r)
        x[::64] = np.where(light[::64], 2.0 ** -(60.0 + 8.0 * r), 1.0)
        W[r] = x
    y0, t0 = _start()
    for b in (1, 2, 4):
        precs = np.full(6, b, np.uint8)
        maps, _ = lw.lowra_learn_codebooks(lw.Layout(precs, K), torch.from_numpy(W).cuda(), y0, t0, 1)
        maps3, _ = lw.lowra_learn_codebooks_all(torch.from_numpy(W).cuda(), y0, t0, 1)
        assert torch.equal(maps, maps3[{1: 0, 2: 1, 4: 2}[b]])
        ref, _ = oracle.lloyd_max(W, precs, T=1)
        assert np.all(np.abs(maps.cpu().numpy().astype(np.float64) - ref) <= 2.4e-7), b


def _time(f):
    f(); f()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(5):
        torch.cuda.synchronize()
        a.record(); f(); b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def _few_values(bits, T, K, factor):
    import paper_2502_08141_b200 as lw

    N = 2048
    gen = torch.Generator(device="cuda").manual_seed(K)
    W = torch.randn(N, K, device="cuda", generator=gen) * 0.02
    y0, t0 = _start()
    layout = lw.Layout(np.full(N, bits or 1, np.uint8), K)
    run = lambda w: lw.lowra_learn_codebooks(layout, w, y0, t0, T) if bits else lw.lowra_learn_codebooks_all(w, y0, t0, T)
    usual = _time(lambda: run(W))
    ternary = torch.sign(W) * (W.abs() > 0.012).float()
    pruned = W * (torch.rand(N, K, device="cuda", generator=gen) < 0.1)
    rounded = torch.round(W / W.abs().amax(1, keepdim=True) * 7)
    for name, w in (("ternary", ternary), ("pruned", pruned), ("rounded", rounded)):
        assert _time(lambda: run(w)) <= factor * usual, name


@pytest.mark.parametrize("K", [4096, 11008])
@pytest.mark.parametrize("bits,T", [(2, 2), (4, 1)])
def test_rows_of_few_values_looked_through(K, bits, T):
    """Empty buckets are not looked for (the longest took 40 times the usual)."""
    _few_values(bits, T, K, 2.0)


@pytest.mark.parametrize("K,factor", [(4096, 2.5), (8192, 3.2)])
def test_rows_of_few_values_sorted(K, factor):
    """Values that share a cell are placed together, and a threshold in a cell of many is the whole warp's work (the pruned rows took
    3.1 and 4.2 times the usual)."""
    _few_values(0, 2, K, factor)


@pytest.mark.parametrize("K", [256, 1024, 4096, 5120, 8192, 11008, 16384])
def test_crowded_rows_give_the_same_tables(K):
    """Rows of a few values, ordinary ones and rows that are half of either, in the sorted form and (through a layout, one round) in the
    form that looks through the row: one set of tables, the oracle's."""
    import paper_2502_08141_b200 as lw

    rng = np.random.default_rng(K)
    W = rng.standard_normal((12, K)).astype(np.float32) * 0.02
    W[0:3] = np.sign(W[0:3]) * (np.abs(W[0:3]) > 0.012)
    W[3:6] *= rng.random((3, K)) < 0.1
    W[6:8] = np.round(W[6:8] / np.abs(W[6:8]).max() * 7)
    W[8, : K // 2] = 0.02
    W[9, K // 2:] = 0.0
    W[10] = 0.0
    y0, t0 = _start()
    Wd = torch.from_numpy(W).cuda()
    for T in (1, 2, 5):
        maps3, thr3 = lw.lowra_learn_codebooks_all(Wd, y0, t0, T)
        for c, b in enumerate((1, 2, 4)):
            precs = np.full(12, b, np.uint8)
            maps, thr = lw.lowra_learn_codebooks(lw.Layout(precs, K), Wd, y0, t0, T)
            assert torch.equal(maps, maps3[c]) and torch.equal(thr, thr3[c]), (T, b)
            ref, _ = oracle.lloyd_max(W, precs, T=T)
            assert np.all(np.abs(maps.cpu().numpy().astype(np.float64) - ref) <= 2.4e-7), (T, b)
