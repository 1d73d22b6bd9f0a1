"""The learner with many rows: blocks in order for several rounds, three kernels in one call, and what each kernel's slow ways must not lose or cost.

Which kernel takes a row depends on the number of rows.  With 1200 of them (nine to an SM)
  all precisions and 4 bits   go by the blocks' order in the first round; in later ones where the tables in kernel_for say so (2048, 4096, 6144 values: to the second or third at least)
  2 bits                      from the second round on; 1 bit: 1152 to 2048 values from the third, 4096 from the fourth
while a call of 148 of them takes 4-bit rows of 1152 to 6144 values through the whole row's order (above 3072 values from the second round on) and most of the others through the row in
every round.  One fixed-point grid: the same
tables bit for bit.
"""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from test_gpu_learn_rows import _start
from test_gpu_learn_sums import _few_values

pytestmark = pytest.mark.gpu

N, PART = 1200, 148


def _rows(K):
    W = si.weights(N, K, matrix_id=K % 43, kind="llama").copy()
    rng = np.random.default_rng(K)
    W[::7] *= np.repeat(10.0 ** rng.uniform(-6, 0, (W[::7].shape[0], K // 64)), 64, axis=1).astype(np.float32)
    W[3::11, 64:128] *= np.float32(1e6)                     # nearly every bucket is added up again
    W[5::13] = np.round(W[5::13] / np.abs(W[5::13]).max(1, keepdims=True) * 3) * np.float32(0.25)
    W[11, K - 64:] = 0.0
    W[17, 64:] = 0.0
    W[19] = 0.0
    return W


@pytest.mark.parametrize("K", [1152, 2048, 3072, 4096, 4608, 6144])
def test_many_rows_as_few(K):
    import paper_2502_08141_b200 as lw

    W = _rows(K)
    Wd, (y0, t0) = torch.from_numpy(W).cuda(), _start()
    some = np.unique(np.concatenate([np.arange(0, 24), np.arange(140, N, 97)]))
    parts = [slice(i, min(i + PART, N)) for i in range(0, N, PART)]
    for T in (1, 2, 3, 4):
        maps3, thr3 = lw.lowra_learn_codebooks_all(Wd, y0, t0, T)
        few = [lw.lowra_learn_codebooks_all(Wd[p], y0, t0, T) for p in parts]
        assert torch.equal(maps3, torch.cat([m for m, _ in few], 1)) and torch.equal(thr3, torch.cat([t for _, t in few], 1)), T
        for c, b in enumerate((1, 2, 4)):
            maps, thr = lw.lowra_learn_codebooks(lw.Layout(np.full(N, b, np.uint8), K), Wd, y0, t0, T)
            few = [lw.lowra_learn_codebooks(lw.Layout(np.full(p.stop - p.start, b, np.uint8), K), Wd[p], y0, t0, T) for p in parts]
            assert torch.equal(maps, torch.cat([m for m, _ in few])) and torch.equal(thr, torch.cat([t for _, t in few])), (T, b)
            assert torch.equal(maps, maps3[c]) and torch.equal(thr, thr3[c]), (T, b)
            if T in (2, 3):
                ref, _ = oracle.lloyd_max(W[some], np.full(some.size, b, np.uint8), T=T)
                assert np.all(np.abs(maps[torch.from_numpy(some).cuda()].cpu().numpy().astype(np.float64) - ref) <= 2.4e-7), (T, b)


def test_three_kernels_in_one_call():
    """Rows of 3072 values and three rounds: 1-bit rows through the row, 2-bit rows by their blocks' order, 4-bit rows by the whole row's, in three launches that do not wait for
    one another to begin.  What follows on the stream finds all tables in place."""
    import paper_2502_08141_b200 as lw

    K, T = 3072, 3
    W = _rows(K)
    rng = np.random.default_rng(1)
    precs = rng.permutation(np.repeat(np.array([1, 2, 4], np.uint8), [600, 360, 240]))
    Wd, (y0, t0) = torch.from_numpy(W).cuda(), _start()
    layout = lw.Layout(precs, K)
    maps3, thr3 = lw.lowra_learn_codebooks_all(Wd, y0, t0, T)
    plane = torch.from_numpy(precs.astype(np.int64) >> 1).cuda()
    rows = torch.arange(N, device="cuda")
    want_maps, want_thr = maps3[plane, rows], thr3[plane, rows]
    want = lw.lowra_encode(layout, Wd, want_thr)
    for _ in range(5):
        maps, thr = (torch.full((N, 16), 7.0, device="cuda") for _ in range(2))
        lw.lowra_learn_codebooks(layout, Wd, y0, t0, T, maps, thr)
        packed, absmax = lw.lowra_encode(layout, Wd, thr)
        assert torch.equal(maps, want_maps) and torch.equal(thr, want_thr)
        assert torch.equal(packed[: layout.packed_bytes], want[0][: layout.packed_bytes]) and torch.equal(absmax, want[1])


@pytest.mark.parametrize("K", [1024, 4096, 8192, 11008])
def test_weights_below_the_grid_in_the_whole_rows_order(K):
    """Buckets whose elements all lie in blocks 2^-60 to 2^-100 as heavy as the row's heaviest, for ten rounds: both forms bring the whole row into order, and both agree with the oracle."""
    import paper_2502_08141_b200 as lw

    rng = np.random.default_rng(K + 2)
    W = np.zeros((6, K), np.float32)
    for r in range(6):
        x = np.sign(rng.standard_normal(K)) * rng.uniform(0.95, 1.0, K)
        light = np.repeat(rng.random(K // 64) < 0.5, 64)
        x[light] = rng.uniform(-0.85, 0.85, light.sum()) * 2.0 ** -(60.0 + 8.0 * r)
        x[::64] = np.where(light[::64], 2.0 ** -(60.0 + 8.0 * r), 1.0)
        W[r] = x
    y0, t0 = _start()
    Wd, precs = torch.from_numpy(W).cuda(), np.full(6, 4, np.uint8)
    maps, thr = lw.lowra_learn_codebooks(lw.Layout(precs, K), Wd, y0, t0, 10)
    maps3, thr3 = lw.lowra_learn_codebooks_all(Wd, y0, t0, 10)
    assert torch.equal(maps, maps3[2]) and torch.equal(thr, thr3[2])
    ref, _ = oracle.lloyd_max(W, precs, T=10)
    assert np.all(np.abs(maps.cpu().numpy().astype(np.float64) - ref) <= 2.4e-7)


@pytest.mark.parametrize("bits,T,K,factor", [(0, 4, 4096, 2.2), (0, 4, 8192, 3.0),             # the whole row's order: pruned rows are crowded in one cell
                                             (1, 2, 4096, 1.5), (2, 1, 11008, 1.5)])          # through the row: empty buckets are not looked for
def test_rows_of_few_values(bits, T, K, factor):
    _few_values(bits, T, K, factor)
