"""Values exactly on a threshold, after the normalisation's rounding.

Every row's thresholds are normalised values of its own, so that in every block some fl(x * fl(1 / absmax)) equal a threshold where the unrounded product lies
on either side of it.  A kernel that fuses the multiplication with the comparison's subtraction puts about half of them a bucket too low.  Codes are
exact: bit for bit the oracle's; the errors follow the same buckets.
"""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [128, 1152, 4096])
def test_values_on_thresholds(K):
    import paper_2502_08141_b200 as lw

    N = 48
    rng = np.random.default_rng(K)
    W = si.weights(N, K, matrix_id=K % 31, kind="llama").copy()
    W[::5, :] = np.round(W[::5, :] / np.abs(W[::5, :]).max() * 40) * np.float32(0.37)       # many equal values, and zeros of either sign
    W[::10, ::7] = -0.0
    precs = rng.permutation(np.repeat(np.array([1, 2, 4], np.uint8), N // 3))
    absmax = np.abs(W.reshape(N, -1, 64)).max(-1, keepdims=True)
    with np.errstate(divide="ignore"):
        inv = np.where(absmax == 0, np.float32(0), (np.float32(1) / absmax).astype(np.float32))
    n = (W.reshape(N, -1, 64) * inv).astype(np.float32).reshape(N, K)
    thr = np.full((N, 16), np.inf, np.float32)
    maps = np.zeros((N, 16), np.float32)
    for r in range(N):
        L = 1 << int(precs[r])
        thr[r, : L - 1] = np.sort(rng.choice(n[r], L - 1))
        maps[r, :L] = np.sort(rng.uniform(-1, 1, L)).astype(np.float32)
    layout = lw.Layout(precs, K)
    dev = lambda a: torch.from_numpy(a).cuda()
    packed, am = lw.lowra_encode(layout, dev(W), dev(thr))
    packed_ref, am_ref = oracle.encode(W, precs, thr)
    assert np.array_equal(packed.cpu().numpy()[: layout.packed_bytes], packed_ref)
    assert np.array_equal(am.cpu().numpy().view(np.uint32), am_ref.view(np.uint32))
    sse, res = lw.lowra_quant_error(layout, dev(W), dev(maps), dev(thr), want_residual=True)
    sse_ref, res_ref = oracle.quant_error(W, precs, maps, thr)
    assert np.array_equal(res.cpu().numpy().view(np.uint32), res_ref.view(np.uint32))
    alone, _ = lw.lowra_quant_error(layout, dev(W), dev(maps), dev(thr))
    assert np.all(np.abs(sse.cpu().numpy() - sse_ref) <= 2.0 ** -21 * sse_ref) and torch.equal(sse, alone)
