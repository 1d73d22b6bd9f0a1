"""The learner's time: rows whose blocks differ widely, and one round beside two.

A block 10^6 times heavier than the others leaves nearly every bucket below what the fixed-point sums resolve, so that each is added up again.  In blocks whose values lie
in order a bucket's are found by bisection; a walk through every block for every such bucket took 2.1 to 2.7 times the usual.
"""
import math

import numpy as np
import pytest
import torch

from test_gpu_learn_rows import _start

pytestmark = pytest.mark.gpu


def _us(f, calls=8):
    """GPU time of a call, from a graph of several."""
    f()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(calls):
            f()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = math.inf
    for _ in range(6):
        a.record(); g.replay(); b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return 1e3 * best / calls


def _learner(N, K, bits, W):
    import paper_2502_08141_b200 as lw

    y0, t0 = _start()
    maps, thr = (torch.empty((N, 16) if bits else (3, N, 16), device="cuda") for _ in range(2))
    layout = lw.Layout(np.full(N, bits or 1, np.uint8), K)
    if bits:
        return lambda T, w=W: lw.lowra_learn_codebooks(layout, w, y0, t0, T, maps, thr)
    return lambda T, w=W: lw.lowra_learn_codebooks_all(w, y0, t0, T, maps, thr)


@pytest.mark.parametrize("N,K,bits,T", [(4096, 4096, 0, 2), (4096, 2048, 4, 2), (4096, 4096, 4, 3), (2048, 8192, 4, 2)])
def test_rows_of_unequal_blocks(N, K, bits, T):
    gen = torch.Generator(device="cuda").manual_seed(K)
    W = torch.randn(N, K, device="cuda", generator=gen) * 0.02
    heavy = W.clone()
    heavy[:, 64:128] *= 1e6
    run = _learner(N, K, bits, W)
    usual, unequal = _us(lambda: run(T)), _us(lambda: run(T, heavy))
    assert unequal <= 1.8 * usual, (usual, unequal)


@pytest.mark.parametrize("bits", [4, 0])
@pytest.mark.parametrize("N,K", [(148, 1152), (296, 1152), (296, 1536), (148, 2048)])
def test_one_round_takes_no_longer_than_two(N, K, bits):
    """A few rows go through the order of the whole row from the first round on, not from the second (where blocks' order took 1.1 times as long for one round as that for
    two)."""
    run = _learner(N, K, bits, torch.randn(N, K, device="cuda", generator=torch.Generator(device="cuda").manual_seed(K)) * 0.02)
    one, two = _us(lambda: run(1)), _us(lambda: run(2))
    assert one <= two, (one, two)
