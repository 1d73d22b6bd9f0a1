"""Small weights with a low rank: one launch, whose CTAs form the projection themselves.

At the edges of that form (features 128 to 512, ranks 16 and 32, tokens 1 to 16, channels that end inside a group of 64 rows, and the first call past each edge), against
the oracle within the bounds of every product; and bit for bit what the group gets in company, where the projection is a launch of its own.  The projection
left in the workspace: one bf16 rounding, zeros behind the rank.
"""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from helpers import make_case
from test_gpu_few_tokens import FRO_TOL, MAX_TOL, _bf, _bits, _dev, gemm_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,r,mix,natural,tokens", [
    (8, 128, 16, {1: 0.5, 2: 0.5}, False, (1, 8)),
    (200, 256, 32, {1: 0.3, 2: 0.5, 4: 0.2}, True, (3, 16)),
    (264, 384, 32, {4: 1.0}, False, (8, 9)),                        # a step and a half: two slices of twelve
    (512, 512, 16, {1: 0.5, 2: 0.5}, False, (1, 16, 17)),           # the last count takes two launches
    (2560, 512, 32, {2: 1.0}, False, (7, 15)),                      # 40 groups of rows
    (2624, 512, 32, {2: 1.0}, False, (15,)),                        # one more: two launches
    (304, 640, 16, {1: 0.6, 2: 0.35, 4: 0.05}, False, (5,)),        # too long
])
def test_one_launch(N, K, r, mix, natural, tokens):
    import paper_2502_08141_b200 as lw

    s = 1.5
    case = make_case(N, K, mix, matrix_id=(N + K) % 71, lloyd_iters=1)
    layout = lw.Layout(case.precs, K, natural=natural)
    maps, thr = _dev(case.maps), _dev(case.thr)
    packed, absmax = lw.lowra_encode(layout, _dev(case.W), thr)
    A_bits, B_bits = si.bf16_normal((K, r), 0.05, stream=51), si.bf16_normal((r, N), 0.05, stream=52)
    A, B = _bf(A_bits), _bf(B_bits)
    for M in tokens:
        X_bits = si.activations(M, K, matrix_id=M)
        X = _bf(X_bits)
        ws = torch.full((lw.lowra_workspace_bytes(layout, M, r),), 255, dtype=torch.uint8, device="cuda")
        buf = torch.full((M + 2, N), 7.0, dtype=torch.bfloat16, device="cuda")       # a canary row on either side
        lw.lowra_lora_forward(layout, packed, absmax, maps, X, A, B, s, Y=buf[1:M + 1], workspace=ws)
        assert lw.lowra_device_status(ws) == lw.LOWRA_OK
        assert (buf[0] == 7.0).all() and (buf[M + 1] == 7.0).all()
        emax, efro = gemm_errors(si.bf16_bits_to_f32(_bits(buf[1:M + 1])), oracle.lora_forward(case.W_hat, X_bits, A_bits, B_bits, s))
        assert emax <= MAX_TOL and efro <= FRO_TOL, (M, emax, efro)
        T_ref = s * (oracle.bf16_to_f64(X_bits) @ oracle.bf16_to_f64(A_bits))
        T = si.bf16_bits_to_f32(_bits(lw.lowra_workspace_projection(ws, M, r))).astype(np.float64)
        assert np.all(T[:, r:] == 0) and np.abs(T[:, :r] - T_ref).max() <= 2.0 ** -8 * np.abs(T_ref).max()
        company = lw.lowra_lora_forward_adapters(layout, packed, absmax, torch.stack([maps, maps]), torch.cat([X, X[:1]]), np.array([0, M, M + 1], np.int32),
                                                 torch.stack([A, A]), torch.stack([B, B]), s)
        assert torch.equal(company[:M].view(torch.int16), buf[1:M + 1].view(torch.int16)), M
