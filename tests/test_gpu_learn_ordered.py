"""The learner's kernel for blocks in order at the edges of its sizes: the last row length for a number of warps (or a part of a block per lane) and the first
for the next, whose last warp is nearly empty.

The tables have to be the three-precision form's bit for bit (one fixed-point grid, whatever the order of the additions) and the
oracle's to 2 ulp of fp32 at 1, as everywhere for the learner.  Some rows hold equal values, zero blocks, both zeros and weights of six decades.
"""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from test_gpu_learn_rows import _start

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [256, 512, 640, 1024, 1152, 2048, 2176, 6144, 6272, 8192, 8320, 10240, 10368, 12288, 12416, 14336, 14464, 16384])
def test_blocks_in_order(K):
    import paper_2502_08141_b200 as lw

    N = 12
    W = si.weights(N, K, matrix_id=K % 47, kind="llama").copy()
    rng = np.random.default_rng(K)
    W[::4] *= np.repeat(10.0 ** rng.uniform(-6, 0, (N // 4, K // 64)), 64, axis=1).astype(np.float32)
    W[1] = np.round(W[1] / np.abs(W[1]).max() * 3) * 0.25
    W[1, :64] = np.where(rng.random(64) < 0.5, -0.0, 0.0)
    W[2, K - 64:] = 0.0
    W[3, 64:] = 0.0
    y0, t0 = _start()
    Wd = torch.from_numpy(W).cuda()
    for T in (1, 4):
        maps3, thr3 = lw.lowra_learn_codebooks_all(Wd, y0, t0, T)
        for c, b in enumerate((1, 2, 4)):
            precs = np.full(N, b, np.uint8)
            maps, thr = lw.lowra_learn_codebooks(lw.Layout(precs, K), Wd, y0, t0, T)
            assert torch.equal(maps, maps3[c]) and torch.equal(thr, thr3[c]), (T, b)
            ref, _ = oracle.lloyd_max(W, precs, T=T)
            assert np.all(np.abs(maps.cpu().numpy().astype(np.float64) - ref) <= 2.4e-7), (T, b)
