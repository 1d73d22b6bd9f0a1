"""Several adapters' small token groups where their product changes its form: one CTA for all slices of 64 rows (many groups of up to 16
tokens, slots of one or two steps) or a cluster for them.  Every group's result is bit for bit that of a call of its own, which
takes the other form, and leaves the projection that the gradients read."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,r,counts", [
    (2048, 2048, 64, (1, 2, 8)),                        # slots of one step, rank steps in half of them
    (2048, 2048, 16, (16, 1, 9)),                       # one rank step in all
    (2504, 1152, 128, (3, 5, 2, 8, 1, 4, 7, 2)),        # five steps over four slots: one of two, ranks round twice
    (704, 4096, 48, (8, 8, 8, 8, 8, 8, 8)),             # eight slices
    (4096, 4096, 64, (12, 16)),
    (4096, 4224, 64, (2, 2)),                           # slots of three steps: a cluster after all
    (512, 512, 16, (16, 1, 33)),
    (136, 128, 128, (9, 32)),                           # a contraction of half a step
    (264, 640, 16, (2, 25)),                            # steps that do not come out even
])
def test_groups_equal_calls_of_their_own(N, K, r, counts):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(N + K + r)
    precs = si.precisions(N, {1: 0.3, 2: 0.5, 4: 0.2}, matrix_id=5)
    layout = lw.Layout(precs, K)
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    packed, absmax = lw.lowra_encode(layout, torch.randn(N, K, device="cuda", generator=gen), thr)
    n, M = len(counts), sum(counts)
    start = [sum(counts[:i]) for i in range(n + 1)]
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    X, A, B = draw(M, K), draw(n, K, r) * 0.05, draw(n, r, N) * 0.05
    tables = maps.unsqueeze(0) * (1.0 + 0.1 * torch.arange(n, device="cuda").view(n, 1, 1))
    Y = lw.lowra_lora_forward_adapters(layout, packed, absmax, tables.contiguous(), X, start, A, B, 2.0)
    for a in range(n):
        rows = slice(start[a], start[a + 1])
        own = lw.lowra_lora_forward(layout, packed, absmax, tables[a].contiguous(), X[rows].contiguous(), A[a].contiguous(), B[a].contiguous(), 2.0)
        assert torch.equal(Y[rows], own), a
        T = 2.0 * (X[rows].float() @ A[a].float())      # what the call leaves for the gradients: bf16 of that, ranks padded to 64 with zeros
        ws = torch.zeros(lw.lowra_workspace_bytes(layout, counts[a], r), dtype=torch.uint8, device="cuda")
        lw.lowra_lora_forward(layout, packed, absmax, tables[a].contiguous(), X[rows].contiguous(), A[a].contiguous(), B[a].contiguous(), 2.0, workspace=ws)
        left = lw.lowra_workspace_projection(ws, counts[a], r).float()
        assert bool(((left[:, :r] - T).abs() <= 2.0 ** -8 * T.abs() + 2.0 ** -16 * K ** 0.5).all()) and not bool(left[:, r:].any()), a
