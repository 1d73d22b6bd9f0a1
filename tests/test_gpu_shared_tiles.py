"""Tiles that several clusters share in the tensor-core kernel, each finishing some of it: two to six clusters to a weight tile, T tiles
between two to seven, ranks of one and two widths, row tiles that are almost empty, tokens that leave one CTA of a pair (or the second half of a
tile) without any - both directions, with and without a deal, against fp64 products of the decoded weight, and twice, bit for bit."""
import pytest
import torch

import synth_inputs as si
from helpers import FRO_TOL, MAX_TOL, gemm_errors

pytestmark = pytest.mark.gpu

MIX = {1: 0.4, 2: 0.4, 4: 0.2}


@pytest.mark.parametrize("N,K,r,tokens", [
    (4096, 4096, 64, (65, 129, 256)),       # four clusters a tile, seven for T
    (1032, 4096, 128, (100, 257, 500)),     # a row tile of eight rows
    (2048, 2048, 48, (66, 128, 384, 520)),
    (520, 8192, 96, (70, 300, 1000)),       # six clusters a tile
    (4104, 1536, 16, (130, 400)),           # short contractions forward
])
def test_against_fp64(N, K, r, tokens):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(N + K + r)
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    precs = si.precisions(N, MIX, matrix_id=3)
    layouts = [lw.Layout(precs, K), lw.Layout(precs, K).build_deal()]
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    packed, absmax = lw.lowra_encode(layouts[0], draw(N, K).float(), thr)
    W = lw.lowra_decode(layouts[0], packed, absmax, maps).double()
    A, B = draw(K, r) * 0.05, draw(r, N) * 0.05
    for M in tokens:
        X, dY = draw(M, K), draw(M, N)
        refs = (X.double() @ W.T + 2.0 * (X.double() @ A.double()) @ B.double(), dY.double() @ W + 2.0 * (dY.double() @ B.double().T) @ A.double().T)
        for layout in layouts:
            ws = lw.lowra_workspace_init(torch.empty(lw.lowra_workspace_bytes(layout, M, r), dtype=torch.uint8, device="cuda"))
            for call, act, ref in ((lw.lowra_lora_forward, X, refs[0]), (lw.lowra_lora_backward_input, dY, refs[1])):
                outs = [call(layout, packed, absmax, maps, act, A, B, 2.0, workspace=ws) for _ in range(2)]
                assert lw.lowra_device_status(ws) == lw.LOWRA_OK
                assert torch.equal(*outs), (M, call.__name__)
                emax, efro = gemm_errors(outs[0].float().cpu().numpy(), ref.cpu().numpy())
                assert emax <= MAX_TOL and efro <= FRO_TOL, (M, call.__name__, emax, efro)
