"""Many token groups on one weight, where a CTA takes one group's tokens and all slices of the contraction: every width of a group, rows
that end inside a group of 64, slices of even and uneven length, ranks that reach some slices only - each group bit for bit as a call of its own,
which shares its slices out over a cluster."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu

WIDTHS = (17, 24, 25, 32, 1, 9, 8, 16)


@pytest.mark.parametrize("N,K,r,mix,counts", [
    (4104, 4096, 80, {1: 0.3, 2: 0.5, 4: 0.2}, WIDTHS),          # four slices of two steps to either half
    (4096, 1664, 16, {4: 1.0}, WIDTHS),                          # six and a half steps over four slots; one rank step
    (9000, 256, 128, {1: 0.5, 2: 0.5}, WIDTHS),                  # one step: the first half of the warps has none
    (4096, 4096, 64, {1: 0.6, 2: 0.35, 4: 0.05}, (7,) * 9),      # more groups than one launch takes
])
def test_groups_equal_calls_of_their_own(N, K, r, mix, counts):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(N + K + r)
    precs = si.precisions(N, mix, matrix_id=7)
    layout = lw.Layout(precs, K, natural=N == 9000)
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    packed, absmax = lw.lowra_encode(layout, torch.randn(N, K, device="cuda", generator=gen), thr)
    n, M = len(counts), sum(counts)
    start = [sum(counts[:i]) for i in range(n + 1)]
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    X, A, B = draw(M, K), draw(n, K, r) * 0.05, draw(n, r, N) * 0.05
    tables = (maps.unsqueeze(0) * (1.0 + 0.1 * torch.arange(n, device="cuda").view(n, 1, 1))).contiguous()
    Y = lw.lowra_lora_forward_adapters(layout, packed, absmax, tables, X, start, A, B, 2.0)
    for a in range(n):
        rows = slice(start[a], start[a + 1])
        own = lw.lowra_lora_forward(layout, packed, absmax, tables[a], X[rows], A[a], B[a], 2.0)
        assert torch.equal(Y[rows], own), a
