"""The quantisation error with thresholds in any order: what is left of the weights is what the codes leave of them.

Thresholds are meant to be sorted, but neither the encoder nor the errors check that.  Both search the same way, so that the residual is W minus the decoded codes, bit for
bit, whatever their order; and the error of every channel at one precision is the one among three.
"""
import numpy as np
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [1, 2, 4])
@pytest.mark.parametrize("K", [128, 640, 4096])
def test_thresholds_in_any_order(K, bits):
    import paper_2502_08141_b200 as lw

    N, L = 40, 1 << bits
    rng = np.random.default_rng(K + bits)
    W = torch.from_numpy(si.weights(N, K, matrix_id=K % 37, kind="llama")).cuda()
    maps, thr = np.zeros((N, 16), np.float32), np.full((N, 16), np.inf, np.float32)
    maps[:, :L], thr[:, : L - 1] = rng.uniform(-1, 1, (N, L)), rng.uniform(-0.7, 0.7, (N, L - 1))
    maps, thr = torch.from_numpy(maps).cuda(), torch.from_numpy(thr).cuda()
    layout = lw.Layout(np.full(N, bits, np.uint8), K)
    packed, absmax = lw.lowra_encode(layout, W, thr)
    left = W - lw.lowra_decode(layout, packed, absmax, maps).float()
    sse, residual = lw.lowra_quant_error(layout, W, maps, thr, want_residual=True)
    assert torch.equal(residual, left)
    alone, _ = lw.lowra_quant_error(layout, W, maps, thr)
    among = lw.lowra_channel_errors(W, torch.stack([maps] * 3), torch.stack([thr] * 3))
    exact = left.double().square().sum(1)
    for e in (sse, alone, among[:, bits >> 1]):
        assert torch.all((e - exact).abs() <= 2.0 ** -21 * exact)
