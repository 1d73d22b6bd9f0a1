"""Calls cut over all 74 pairs of SMs, where cluster 0 keeps its part of a shared T tile in the place of cluster 1: both directions, one and two halves
of a token tile (the weight tiles finished by their first cluster, and shared), ranks of one and two widths, against fp64 products of the
decoded weight, and twice, bit for bit."""
import pytest
import torch

import synth_inputs as si
from helpers import FRO_TOL, MAX_TOL, gemm_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,r,M,backward", [
    (9184, 6016, 64, 77, True),       # 24 tiles by three clusters, T by two (all of them)
    (9216, 9216, 128, 256, True),
    (6144, 9216, 80, 400, False),     # tiles of 512 tokens, shared
    (9216, 6144, 128, 500, True),
    (4608, 9216, 16, 70, True),       # 36 tiles by two clusters
])
def test_against_fp64(N, K, r, M, backward):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(N + K + r)
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    precs = si.precisions(N, {1: 0.3, 2: 0.5, 4: 0.2}, matrix_id=3)
    layout = lw.Layout(precs, K).build_deal()
    choice = lw.lowra_diag_choose(layout, backward, [M], r)
    assert choice["clusters"] == 74 and choice["w_split"] == (1 if M <= 256 else 3) and choice["t_split"] == 2, choice
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    packed, absmax = lw.lowra_encode(layout, torch.randn(N, K, device="cuda", generator=gen), thr)
    W = lw.lowra_decode(layout, packed, absmax, maps).double()
    A, B, x = draw(K, r) * 0.05, draw(r, N) * 0.05, draw(M, N if backward else K)
    a, b, xd = A.double(), B.double(), x.double()
    ref = xd @ W + 2.0 * (xd @ b.T) @ a.T if backward else xd @ W.T + 2.0 * (xd @ a) @ b
    ws = lw.lowra_workspace_init(torch.empty(lw.lowra_workspace_bytes(layout, M, r), dtype=torch.uint8, device="cuda"))
    call = lw.lowra_lora_backward_input if backward else lw.lowra_lora_forward
    one, two = (call(layout, packed, absmax, maps, x, A, B, 2.0, workspace=ws) for _ in range(2))
    assert lw.lowra_device_status(ws) == lw.LOWRA_OK and torch.equal(one, two)
    emax, efro = gemm_errors(one.float().cpu().numpy(), ref.cpu().numpy())
    assert emax <= MAX_TOL and efro <= FRO_TOL, (emax, efro)
