"""Tiles that several clusters share in launches of several members - the flags of the shared T tiles then lie behind one another, member by member:
batch calls forward and backward, and token groups of several adapters, against fp64 products of the decoded weights, and twice, bit for bit."""
import numpy as np
import pytest
import torch

import synth_inputs as si
from helpers import FRO_TOL, MAX_TOL, gemm_errors

pytestmark = pytest.mark.gpu

MIX = {1: 0.4, 2: 0.4, 4: 0.2}


def close(got, ref):
    emax, efro = gemm_errors(got.float().cpu().numpy(), ref.cpu().numpy())
    assert emax <= MAX_TOL and efro <= FRO_TOL, (emax, efro)


def weight(lw, N, K, gen, matrix_id):
    precs = si.precisions(N, MIX, matrix_id=matrix_id)
    layout = lw.Layout(precs, K).build_deal()
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    packed, absmax = lw.lowra_encode(layout, torch.randn(N, K, device="cuda", generator=gen), thr)
    return dict(layout=layout, packed=packed, absmax=absmax, maps=maps)


def shares(lw, layout, backward, tokens, r, one_weight=False):
    c = lw.lowra_diag_choose(layout, backward, tokens, r, one_weight)
    assert c["w_split"] > 1 and c["t_split"] > 1, c


@pytest.mark.parametrize("N,K,r,M,count,directions", [
    (1024, 4096, 64, 100, 3, (False,)),
    (4096, 1024, 128, 70, 2, (True,)),
    (2048, 4096, 128, 70, 2, (False,)),
    (768, 3072, 16, 256, 4, (False,)),
])
def test_batch_calls(N, K, r, M, count, directions):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(N + K + M)
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    weights = [weight(lw, N, K, gen, i) for i in range(count)]
    factors = [(draw(K, r) * 0.05, draw(r, N) * 0.05) for _ in weights]
    for backward in directions:
        shares(lw, weights[0]["layout"], backward, [M] * count, r)
    ws = lw.lowra_workspace_init(torch.empty(lw.lowra_batch_workspace_bytes(weights[0]["layout"], count, M, r), dtype=torch.uint8, device="cuda"))
    for backward, call in ((False, lw.lowra_lora_forward_batch), (True, lw.lowra_lora_backward_input_batch)):
        acts = [draw(M, N if backward else K) for _ in weights]
        outs = []
        for _ in range(2):
            out = [torch.empty(M, K if backward else N, dtype=torch.bfloat16, device="cuda") for _ in weights]
            outs.append(call([dict(**w, act=act, A=A, B=B, out=o) for w, act, (A, B), o in zip(weights, acts, factors, out)], 2.0, ws))
            assert lw.lowra_device_status(ws) == lw.LOWRA_OK
        for w, act, (A, B), one, two in zip(weights, acts, factors, *outs):
            assert torch.equal(one, two)
            W = lw.lowra_decode(w["layout"], w["packed"], w["absmax"], w["maps"]).double()
            x, a, b = act.double(), A.double(), B.double()
            close(one, x @ W + 2.0 * (x @ b.T) @ a.T if backward else x @ W.T + 2.0 * (x @ a) @ b)


@pytest.mark.parametrize("N,K,r,counts", [(1024, 4096, 64, (100, 130, 70)), (520, 4096, 80, (65, 200, 128, 90))])
def test_groups(N, K, r, counts):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(N + K)
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    w = weight(lw, N, K, gen, 5)
    n, M = len(counts), sum(counts)
    start = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    X, A, B = draw(M, K), draw(n, K, r) * 0.05, draw(n, r, N) * 0.05
    tables = (w["maps"].unsqueeze(0) * (1.0 + 0.1 * torch.arange(n, device="cuda").view(n, 1, 1))).contiguous()
    shares(lw, w["layout"], False, counts, r, one_weight=True)
    ws = lw.lowra_workspace_init(torch.empty(lw.lowra_batch_workspace_bytes(w["layout"], 4, M, r), dtype=torch.uint8, device="cuda"))
    Y, again = (lw.lowra_lora_forward_adapters(w["layout"], w["packed"], w["absmax"], tables, X, start, A, B, 2.0, workspace=ws) for _ in range(2))
    assert lw.lowra_device_status(ws) == lw.LOWRA_OK and torch.equal(Y, again)
    for a in range(n):
        W = lw.lowra_decode(w["layout"], w["packed"], w["absmax"], tables[a]).double()
        x = X[start[a]:start[a + 1]].double()
        close(Y[start[a]:start[a + 1]], x @ W.T + 2.0 * (x @ A[a].double()) @ B[a].double())
