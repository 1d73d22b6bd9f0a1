"""Time of the few-token path where its forms change: a call with less to do takes no longer.

By GPU time, from captured graphs (the forms were chosen by such measurements; a form that is the slower one on one side of its line shows as a step down across it).
"""
import math

import numpy as np
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu


def _forward_us(N, K, mix, r, M, calls=20):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(N + K)
    bf16 = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).to(torch.bfloat16)  # noqa: E731
    layout = lw.Layout(si.precisions(N, mix), K)
    packed = torch.randint(0, 256, (layout.packed_bytes,), dtype=torch.uint8, device="cuda", generator=gen)
    absmax = torch.rand(N * (K // 64), device="cuda", generator=gen)
    maps = torch.linspace(-1, 1, 16, device="cuda").repeat(N, 1)
    X, A, B, Y = bf16(M, K), bf16(K, r), bf16(r, N), bf16(M, N)
    ws = torch.empty(lw.lowra_workspace_bytes(layout, M, r), dtype=torch.uint8, device="cuda")
    call = lambda: lw.lowra_lora_forward(layout, packed, absmax, maps, X, A, B, 1.0, Y=Y, workspace=ws)  # noqa: E731
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(calls):
            call()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = math.inf
    for _ in range(6):
        a.record(); g.replay(); b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return 1e3 * best / calls


@pytest.mark.parametrize("r", [16, 32])
@pytest.mark.parametrize("N,K", [(1024, 1024), (1024, 2048), (1536, 3072)])
def test_sixteen_tokens_take_no_longer_than_seventeen(N, K, r):
    """Three CTAs to an SM, for up to 16 tokens, where two fit in one wave: 1.05 to 1.09 of the time of 17 tokens, which two to an SM take."""
    mix = {1: 0.6, 2: 0.35, 4: 0.05}
    few, more = (_forward_us(N, K, mix, r, M) for M in (16, 17))
    assert few <= more, (few, more)


@pytest.mark.parametrize("mix", [{2: 0.75, 4: 0.25}, {1: 0.3, 2: 0.5, 4: 0.2}])
def test_rank_16_takes_no_longer_than_rank_32(mix):
    """A weight of many channels whose CTAs all formed the projection at rank 16: 1.3 of the time at rank 32, for which it is a launch of its own."""
    low, high = (_forward_us(8192, 384, mix, r, 1) for r in (16, 32))
    assert low <= high, (low, high)


def test_slow_rows_and_many_tokens():
    """Likewise 49 groups of rows, some of 4 bits: 16 tokens took 1.1 of the time of 17."""
    few, more = (_forward_us(3072, 512, {1: 0.6, 2: 0.35, 4: 0.05}, 16, M) for M in (16, 17))
    assert few <= more, (few, more)
