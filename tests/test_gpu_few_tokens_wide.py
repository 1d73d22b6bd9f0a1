"""Forward passes of few tokens on weights of many channels and a short contraction, on either side of the line where they leave
the few-token path for tensor-core tiles (shape and tokens decide; 16 tokens always stay, 65 never do): against the fp64 oracle
within the products' bounds, and a token group like the call for it alone, whichever path its neighbours take."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from helpers import FRO_TOL, MAX_TOL, gemm_errors, make_case

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _bf(bits):
    return _dev(bits.view(np.int16)).view(torch.bfloat16)


@pytest.mark.parametrize("N,K,r,mix,groups", [
    (13824, 256, 80, {1: 0.6, 2: 0.35, 4: 0.05}, (16, 17, 32, 1, 65)),     # the line lies at 17 tokens
    (5632, 384, 16, {2: 0.5, 4: 0.5}, (32, 33, 5, 64, 0, 63)),             # at 33
    (8, 128, 16, {4: 1.0}, (17, 64, 33)),                                  # never
])
def test_either_side_of_the_line(N, K, r, mix, groups):
    import paper_2502_08141_b200 as lw

    s, n = 2.0, len(groups)
    case = make_case(N, K, mix, matrix_id=33, lloyd_iters=1)
    start = np.concatenate([[0], np.cumsum(groups)]).astype(np.int32)
    M = int(start[-1])
    packed, absmax = _dev(case.packed), _dev(case.absmax)
    A_bits = [si.bf16_normal((K, r), 0.05, stream=51 + a) for a in range(n)]
    B_bits = [si.bf16_normal((r, N), 0.05, stream=61 + a) for a in range(n)]
    A, B = torch.stack([_bf(a) for a in A_bits]), torch.stack([_bf(b) for b in B_bits])
    maps, X_bits = torch.stack([_dev(case.maps)] * n), si.activations(M, K, matrix_id=44)
    X = _bf(X_bits)
    for dealt in (False, True):
        layout = lw.Layout(case.precs, K)
        if dealt:
            layout.build_deal()
        ws = lw.lowra_workspace_init(torch.empty(lw.lowra_batch_workspace_bytes(layout, 4, M, r), dtype=torch.uint8, device="cuda"))
        Y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
        lw.lowra_lora_forward_adapters(layout, packed, absmax, maps, X, start, A, B, s, Y=Y, workspace=ws)
        assert lw.lowra_device_status(ws) == lw.LOWRA_OK
        for a in range(n):
            m0, m1 = int(start[a]), int(start[a + 1])
            if m1 == m0:
                continue
            got = Y[m0:m1].view(torch.int16).cpu().numpy().view(np.uint16)
            emax, efro = gemm_errors(si.bf16_bits_to_f32(got), oracle.lora_forward(case.W_hat, X_bits[m0:m1], A_bits[a], B_bits[a], s))
            assert emax <= MAX_TOL and efro <= FRO_TOL, (dealt, a, emax, efro)
            one = lw.lowra_lora_forward(layout, packed, absmax, maps[a], X[m0:m1], A[a], B[a], s)
            assert torch.equal(one.view(torch.int16), Y[m0:m1].view(torch.int16)), (dealt, a)     # (no tile of these is cut)
