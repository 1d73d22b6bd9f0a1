"""The fused products where their schedule changes: token tiles of 256 and 512 tokens around their edges, weight tiles and
down-projection tiles cut between clusters (two to six ways, ragged last slices), ranges behind whole rows, operand rows that end
inside the first or the second CTA of a pair, two LoRA blocks.  Both directions against the fp64 oracle within the products'
bounds (the fp32 sums of a cut tile are added in another order, nothing else changes), and a repeated call bit for bit the same:
partial tiles are added in a fixed order."""
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


@pytest.mark.parametrize("N,K,r,mix,tokens", [
    (2304, 2048, 64, {1: 0.6, 2: 0.35, 4: 0.05}, (65, 256, 257, 512, 513)),     # both contractions cut, two to three ways
    (136, 4096, 128, {1: 0.5, 2: 0.5}, (300,)),                                # eight rows in the second CTA (forward); a sixth of a tile per cluster
    (4096, 128, 16, {4: 1.0}, (100, 1025)),                                    # one CTA without rows (backward), two contraction blocks (forward)
    (1288, 1664, 80, {2: 0.75, 4: 0.25}, (770, 2600)),                         # the shortest contraction that is cut, two LoRA blocks
    (3848, 3072, 32, {1: 0.85, 2: 0.15}, (1700,)),                             # more than one row of pieces: ranges over the last
])
def test_schedules_against_the_oracle(N, K, r, mix, tokens):
    import paper_2502_08141_b200 as lw

    s = 2.0
    case = make_case(N, K, mix, matrix_id=(N + K) % 73, lloyd_iters=1)
    layout = lw.Layout(case.precs, K).build_deal()
    packed, absmax, maps = _dev(case.packed), _dev(case.absmax), _dev(case.maps)
    A_bits, B_bits = si.bf16_normal((K, r), 0.03, stream=61), si.bf16_normal((r, N), 0.03, stream=62)
    A, B = _bf(A_bits), _bf(B_bits)
    ws = lw.lowra_workspace_init(torch.empty(lw.lowra_workspace_bytes(layout, max(tokens), r), dtype=torch.uint8, device="cuda"))
    for M in tokens:
        X, dY = si.activations(M, K, matrix_id=M), si.out_grads(M, N, matrix_id=M)
        rows = np.unique(np.concatenate([np.linspace(0, M - 1, 48).astype(np.int64), np.arange(max(0, M - 3), M)]))
        for name, call, act, cols, ref in (
                ("forward", lw.lowra_lora_forward, X, N, oracle.lora_forward(case.W_hat, X[rows], A_bits, B_bits, s)),
                ("backward", lw.lowra_lora_backward_input, dY, K, oracle.lora_backward_input(case.W_hat, dY[rows], A_bits, B_bits, s))):
            got = []
            for _ in range(2):
                buf = torch.full((M + 2, cols), 5.0, dtype=torch.bfloat16, device="cuda")     # a canary row on either side
                buf[1:M + 1] = float("nan")
                call(layout, packed, absmax, maps, _bf(act), A, B, s, buf[1:M + 1], ws)
                assert lw.lowra_device_status(ws) == lw.LOWRA_OK, (name, M)
                assert (buf[0] == 5.0).all() and (buf[M + 1] == 5.0).all(), (name, M)
                got.append(_bits(buf[1:M + 1]))
            assert np.array_equal(got[0], got[1]), (name, M)
            assert np.isfinite(si.bf16_bits_to_f32(got[0])).all(), (name, M)
            emax, efro = gemm_errors(si.bf16_bits_to_f32(got[0][rows]), ref)
            assert emax <= MAX_TOL and efro <= FRO_TOL, (name, M, emax, efro)
