"""Token groups on one weight where a CTA takes a unit and all slices: groups of more than 32 tokens, which are two units, beside smaller ones; eight
slices; a single call of 33 to 64 tokens; with and without a deal.  Each group against fp64 products of its decoded weight, and bit for bit as the
same call on the other layout."""
import numpy as np
import pytest
import torch

import synth_inputs as si
from helpers import FRO_TOL, MAX_TOL, gemm_errors

pytestmark = pytest.mark.gpu

MIX = {1: 0.3, 2: 0.5, 4: 0.2}


@pytest.mark.parametrize("N,K,r,mix,counts", [
    (4096, 4096, 64, MIX, (33, 5, 16, 31, 8, 20)),
    (4104, 4096, 80, MIX, (7, 40, 32, 1, 9, 25)),
    (4096, 1664, 16, {4: 1.0}, (64, 3, 17, 12, 24, 9, 32)),
    (2048, 4096, 128, MIX, (12, 30, 9, 8, 2, 48, 16, 5)),        # eight slices
    (2048, 11008, 64, {1: 0.6, 2: 0.4}, (16,) * 8),              # eight slices of more than five steps each
    (4528, 640, 48, {1: 0.5, 2: 0.5}, (58,)),                    # one call, two units
    (296, 768, 64, {1: 0.5, 2: 0.5}, (33,)),
])
def test_against_fp64(N, K, r, mix, counts):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(N + K + r)
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    precs = si.precisions(N, mix, matrix_id=9)
    layouts = [lw.Layout(precs, K), lw.Layout(precs, K).build_deal()]
    assert lw.lowra_diag_choose(layouts[0], False, counts, r, one_weight=True)["units"] == 1
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    packed, absmax = lw.lowra_encode(layouts[0], torch.randn(N, K, device="cuda", generator=gen), thr)
    n, M = len(counts), sum(counts)
    start = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    X, A, B = draw(M, K), draw(n, K, r) * 0.05, draw(n, r, N) * 0.05
    tables = (maps.unsqueeze(0) * (1.0 + 0.1 * torch.arange(n, device="cuda").view(n, 1, 1))).contiguous()
    results = []
    for layout in layouts:
        ws = lw.lowra_workspace_init(torch.empty(lw.lowra_batch_workspace_bytes(layout, 4, M, r), dtype=torch.uint8, device="cuda"))
        if n == 1:
            results.append(lw.lowra_lora_forward(layout, packed, absmax, tables[0], X, A[0], B[0], 2.0, workspace=ws))
        else:
            results.append(lw.lowra_lora_forward_adapters(layout, packed, absmax, tables, X, start, A, B, 2.0, workspace=ws))
        assert lw.lowra_device_status(ws) == lw.LOWRA_OK
    assert torch.equal(*results)
    for a in range(n):
        W = lw.lowra_decode(layouts[0], packed, absmax, tables[a]).double()
        x = X[start[a]:start[a + 1]].double()
        ref = x @ W.T + 2.0 * (x @ A[a].double()) @ B[a].double()
        emax, efro = gemm_errors(results[0][start[a]:start[a + 1]].float().cpu().numpy(), ref.cpu().numpy())
        assert emax <= MAX_TOL and efro <= FRO_TOL, (a, emax, efro)
