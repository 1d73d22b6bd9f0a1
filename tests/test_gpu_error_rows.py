"""Error and residual where the kernel's split of the rows changes: chunks of 512 or 1024 elements, last chunks of 128 to 896,
more chunks to a row than the eight warps that share it, more rows to a CTA than it sums up at a time, and matrices so large that
the reads keep back for the writes.

The residual is one fp32 subtraction per element: bit for bit W - decode(encode(W)).  Errors: four squares in fp32 (2^-23 from
the residual's rounding, three more roundings), sums in fp64 - 2^-21 relative at worst.  The three-precision form forms the same
sums in the same order: equal.
"""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K", [(3, 128), (1, 512), (41, 640), (7, 1024), (29, 1408), (298, 2176), (12, 9216), (5, 9088),
                                 (5000, 256), (8200, 4224)])
def test_split_of_the_rows(N, K):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(N + K)
    W = torch.randn(N, K, device="cuda", generator=gen)
    W[0, 64:128] = 0.0
    precs = si.precisions(N, {1: 0.5, 2: 0.35, 4: 0.15}, matrix_id=K % 61)
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    layout = lw.Layout(precs, K)
    sse, res = lw.lowra_quant_error(layout, W, maps, thr, want_residual=True)
    sse_only, _ = lw.lowra_quant_error(layout, W, maps, thr)
    packed, absmax = lw.lowra_encode(layout, W, thr)
    ref = W - lw.lowra_decode(layout, packed, absmax, maps).float()
    assert torch.equal(res, ref) and torch.equal(sse, sse_only)
    exact = ref.double().square().sum(1)
    assert bool(((sse - exact).abs() <= 2.0 ** -21 * exact).all())
    maps3, thr3 = torch.zeros(3, N, 16, device="cuda"), torch.full((3, N, 16), float("inf"), device="cuda")
    plane = torch.from_numpy(precs).cuda().long() // 2
    rows = torch.arange(N, device="cuda")
    maps3[plane, rows], thr3[plane, rows] = maps, thr
    assert torch.equal(lw.lowra_channel_errors(W, maps3, thr3)[rows, plane], sse)
