"""The forward pass's path for few tokens, at the sizes where it can go wrong: token counts around its tiles of 8, 16 and 32
tokens and its upper limit, precision classes that end inside a group of 64 or 16 rows (or are missing), contractions that end
inside a step of 256 indices, every way of splitting the contraction, ranks that leave steps of 16 to some warps only.  Against
the fp64 oracle within the products' bounds (operands equal the oracle's bit for bit; the fp32 sums and the two bf16
roundings are those of every other path)."""
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


def _bits(t):
    return t.view(torch.int16).cpu().numpy().view(np.uint16)


@pytest.mark.parametrize("N,K,r,mix,natural,tokens", [
    (8, 128, 16, {1: 0.5, 2: 0.25, 4: 0.25}, False, (1, 64)),                   # half a step, classes of 2 and 4 rows
    (200, 384, 128, {1: 0.34, 2: 0.33, 4: 0.33}, True, (7, 8, 9)),              # a step and a half, groups that end early
    (136, 640, 80, {2: 1.0}, False, (16, 17)),                                  # one class
    (1096, 1152, 48, {1: 0.02, 2: 0.02, 4: 0.96}, False, (31, 32, 33, 63)),
    (2304, 2176, 96, {1: 0.6, 2: 0.35, 4: 0.05}, True, (1, 48)),                # eight slices of nine steps
    (4096, 4096, 64, {1: 0.3, 2: 0.5, 4: 0.2}, False, (1, 17, 64, 65)),         # the last count takes the other path
])
def test_few_tokens_against_the_oracle(N, K, r, mix, natural, tokens):
    import paper_2502_08141_b200 as lw

    s = 2.0
    case = make_case(N, K, mix, matrix_id=(N + 3 * K) % 79, lloyd_iters=1)
    layouts = [lw.Layout(case.precs, K, natural=natural), lw.Layout(case.precs, K, natural=natural).build_deal()]
    maps, thr = _dev(case.maps), _dev(case.thr)
    packed, absmax = lw.lowra_encode(layouts[0], _dev(case.W), thr)
    A_bits, B_bits = si.bf16_normal((K, r), 0.05, stream=31), si.bf16_normal((r, N), 0.05, stream=32)
    A, B = _bf(A_bits), _bf(B_bits)
    for M in tokens:
        X_bits = si.activations(M, K, matrix_id=M)
        ref = oracle.lora_forward(case.W_hat, X_bits, A_bits, B_bits, s)
        T_ref = s * (oracle.bf16_to_f64(X_bits) @ oracle.bf16_to_f64(A_bits))
        outs = []
        for layout in layouts:
            ws = lw.lowra_workspace_init(torch.empty(lw.lowra_workspace_bytes(layout, M, r), dtype=torch.uint8, device="cuda"))
            buf = torch.full((M + 2, N), 7.0, dtype=torch.bfloat16, device="cuda")     # a canary row on either side
            buf[1:M + 1] = float("nan")
            lw.lowra_lora_forward(layout, packed, absmax, maps, _bf(X_bits), A, B, s, Y=buf[1:M + 1], workspace=ws)
            assert lw.lowra_device_status(ws) == lw.LOWRA_OK
            assert (buf[0] == 7.0).all() and (buf[M + 1] == 7.0).all()
            emax, efro = gemm_errors(si.bf16_bits_to_f32(_bits(buf[1:M + 1])), ref)
            assert emax <= MAX_TOL and efro <= FRO_TOL, (M, emax, efro)
            T = si.bf16_bits_to_f32(_bits(lw.lowra_workspace_projection(ws, M, r))).astype(np.float64)
            assert np.all(T[:, r:] == 0)
            assert np.abs(T[:, :r] - T_ref).max() <= 2.0 ** -8 * np.abs(T_ref).max()    # one bf16 rounding
            outs.append(_bits(buf[1:M + 1]))
        assert np.array_equal(outs[0], outs[1]), M       # with and without a deal: the same


def test_many_small_groups_and_a_large_one():
    """More small groups than one launch takes, an empty one and one that takes the other path: every group as the call for it
    alone, bit for bit."""
    import paper_2502_08141_b200 as lw

    N, K, r, s = 328, 640, 32, 1.5
    groups = [1, 5, 0, 64, 9, 300, 2, 33, 16, 7, 8, 1, 17]
    n = len(groups)
    case = make_case(N, K, {1: 0.3, 2: 0.5, 4: 0.2}, matrix_id=12, lloyd_iters=1)
    start = np.concatenate([[0], np.cumsum(groups)]).astype(np.int32)
    M = int(start[-1])
    maps = _dev(np.stack([si.standin_codebooks(case.precs, matrix_id=70 + a)[0] for a in range(n)]))
    A, B = _bf(si.bf16_normal((n * K, r), 0.05, stream=41)).view(n, K, r), _bf(si.bf16_normal((n * r, N), 0.05, stream=42)).view(n, r, N)
    X = _bf(si.activations(M, K, matrix_id=43))
    packed, absmax = _dev(case.packed), _dev(case.absmax)
    for dealt in (False, True):
        layout = lw.Layout(case.precs, K)
        if dealt:
            layout.build_deal()
        ws = lw.lowra_workspace_init(torch.empty(lw.lowra_batch_workspace_bytes(layout, 4, M, r), dtype=torch.uint8, device="cuda"))
        Y = lw.lowra_lora_forward_adapters(layout, packed, absmax, maps, X, start, A, B, s, workspace=ws)
        assert lw.lowra_device_status(ws) == lw.LOWRA_OK
        for a in range(n):
            m0, m1 = int(start[a]), int(start[a + 1])
            if m1 > m0:
                one = lw.lowra_lora_forward(layout, packed, absmax, maps[a], X[m0:m1], A[a], B[a], s)
                assert torch.equal(one.view(torch.int16), Y[m0:m1].view(torch.int16)), (dealt, a)
