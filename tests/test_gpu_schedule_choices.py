"""Calls whose T tiles have clusters of their own while ranges over all weight tiles go to the others: few channels and many tokens, pieces that
come out a little over a row; one or several clusters to a T tile, 256- and 512-token tiles, ranges of half a tile to two tiles, in both directions.
"""
import numpy as np
import pytest
import torch

import synth_inputs as si
from helpers import FRO_TOL, MAX_TOL, gemm_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M,r,dealt", [
    (1024, 4096, 4096, 64, True),      # two clusters to a T tile, ranges of half a tile
    (1000, 4096, 8100, 128, True),     # one cluster, ranges of a tile and more, ragged
    (1024, 8192, 8192, 16, False),
    (3072, 3072, 2999, 64, True),
    (6144, 2048, 1500, 80, False),
    (2304, 4096, 777, 64, True),       # 256-token tiles
    (3072, 3072, 600, 64, False),
])
def test_ranges_beside_the_t_tiles(N, K, M, r, dealt):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(N + K + M)
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    precs = si.precisions(N, {1: 0.5, 2: 0.4, 4: 0.1}, matrix_id=11)
    layout = lw.Layout(precs, K)
    if dealt:
        layout.build_deal()
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    packed, absmax = lw.lowra_encode(layout, draw(N, K).float(), thr)
    W = lw.lowra_decode(layout, packed, absmax, maps).double()
    A, B = draw(K, r) * 0.05, draw(r, N) * 0.05
    ws = lw.lowra_workspace_init(torch.empty(lw.lowra_workspace_bytes(layout, M, r), dtype=torch.uint8, device="cuda"))
    rows = torch.from_numpy(np.unique(np.concatenate([np.linspace(0, M - 1, 400), [255, 256, 511, 512]]).astype(np.int64))).cuda()
    X, dY = draw(M, K), draw(M, N)
    first = None
    for _ in range(3):
        Y = lw.lowra_lora_forward(layout, packed, absmax, maps, X, A, B, 2.0, workspace=ws)
        dX = lw.lowra_lora_backward_input(layout, packed, absmax, maps, dY, A, B, 2.0, workspace=ws)
        assert lw.lowra_device_status(ws) == lw.LOWRA_OK
        if first is None:
            first = (Y, dX)
            x, d = X[rows].double(), dY[rows].double()
            for got, ref in ((Y, x @ W.T + 2.0 * (x @ A.double()) @ B.double()), (dX, d @ W + 2.0 * (d @ B.double().T) @ A.double().T)):
                emax, efro = gemm_errors(got[rows].float().cpu().numpy(), ref.cpu().numpy())
                assert emax <= MAX_TOL and efro <= FRO_TOL, (emax, efro)
        assert torch.equal(Y.view(torch.int16), first[0].view(torch.int16)) and torch.equal(dX.view(torch.int16), first[1].view(torch.int16))
