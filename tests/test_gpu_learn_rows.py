"""The codebook learner where it changes over from one kernel to another: by the length of the rows, by the number of rounds
and by precision.

Both kernels add up on one fixed-point grid, so a row's tables do not depend on which of them takes it: a layout (whose 1-bit
rows go through the whole row in every round while its 4-bit rows are sorted) and the three-precision form (always sorted)
have to agree bit for bit.  Against the oracle: 2 ulp of fp32 at 1, as everywhere for the learner - the grid is 2^-46 of the
row's largest weight, far below that.  A third of the rows have absmax values that spread over six decades and zero blocks, so
that many buckets are light or empty.
"""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si

pytestmark = pytest.mark.gpu


def _start():
    y0, t0 = np.zeros((3, 16)), np.zeros((3, 16))
    for c, b in enumerate((1, 2, 4)):
        y, t = oracle.initial_tables(b)
        y0[c, :y.size], t0[c, :t.size] = y, t
    return y0, t0


@pytest.mark.parametrize("K", [128, 1152, 4096, 4224, 5120, 5248, 8192, 8320, 11264, 11392, 16384, 16512])
def test_every_kernel_gives_the_same_tables(K):
    import paper_2502_08141_b200 as lw

    N = 15
    W = si.weights(N, K, matrix_id=K % 59, kind="llama").copy()
    rng = np.random.default_rng(K)
    W[::3] *= np.repeat(10.0 ** rng.uniform(-6, 0, (N // 3, K // 64)), 64, axis=1).astype(np.float32)
    W[6, 64:128] = 0.0
    W[9] = 0.0
    precs = rng.permutation(np.repeat(np.array([1, 2, 4], np.uint8), N // 3))
    layout, Wd, (y0, t0) = lw.Layout(precs, K), torch.from_numpy(W).cuda(), _start()
    plane = {1: 0, 2: 1, 4: 2}
    for T in (1, 2, 12) if K <= 5120 else (1, 2):
        maps, thr = lw.lowra_learn_codebooks(layout, Wd, y0, t0, T)
        maps3, thr3 = lw.lowra_learn_codebooks_all(Wd, y0, t0, T)
        ref, _ = oracle.lloyd_max(W, precs, T=T)
        assert np.all(np.abs(maps.cpu().numpy().astype(np.float64) - ref) <= 2.4e-7), T
        for r, b in enumerate(precs):
            assert torch.equal(maps[r], maps3[plane[int(b)], r]) and torch.equal(thr[r], thr3[plane[int(b)], r]), (T, r)


def test_a_row_without_a_mean():
    """A NaN or an infinity anywhere in a row: NaN levels for that row, in either kernel, and for no other."""
    import paper_2502_08141_b200 as lw

    W = si.weights(6, 256, matrix_id=3, kind="llama").copy()
    W[1, 77] = np.nan
    W[4, 200] = np.inf
    y0, t0 = _start()
    for T in (2, 12):
        maps3, _ = lw.lowra_learn_codebooks_all(torch.from_numpy(W).cuda(), y0, t0, T)
        maps1, _ = lw.lowra_learn_codebooks(lw.Layout(np.ones(6, np.uint8), 256), torch.from_numpy(W).cuda(), y0, t0, T)
        for m in (maps3[0], maps1):
            assert torch.isnan(m[:, :2]).all(1).tolist() == [False, True, False, False, True, False], T
