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


@pytest.mark.parametrize("N,K", [(3000, 640), (2000, 2176), (1500, 4224), (1000, 9216), (1000, 11008)])
def test_a_rows_error_does_not_depend_on_its_place(N, K):
    """One row over and over, its block maxima spread over six decades, so that fp64 sums show the order of the additions."""
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(K)
    scale = 10.0 ** (-6.0 * torch.rand(K // 64, device="cuda", generator=gen)).repeat_interleave(64)
    W = (torch.randn(K, device="cuda", generator=gen) * scale).expand(N, K).contiguous()
    precs = si.precisions(N, {1: 0.5, 2: 0.35, 4: 0.15}, matrix_id=K % 61)
    plane = torch.from_numpy(precs).cuda().long() // 2
    maps3, thr3 = (torch.empty(3, N, 16, device="cuda") for _ in range(2))
    for c in range(3):
        m, t = si.standin_codebooks(precs[:1] * 0 + (1 << c))
        maps3[c], thr3[c] = torch.from_numpy(m[0]).cuda(), torch.from_numpy(t[0]).cuda()
    sse3 = lw.lowra_channel_errors(W, maps3, thr3)
    assert torch.equal(sse3, sse3[:1].expand(N, 3))
    rows = torch.arange(N, device="cuda")
    sse, _ = lw.lowra_quant_error(lw.Layout(precs, K), W, maps3[plane, rows].contiguous(), thr3[plane, rows].contiguous())
    assert torch.equal(sse, sse3[0, plane])
