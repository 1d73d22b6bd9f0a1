"""lowra_diag_choose: what a call would run, asked without a GPU - its refusals, and that every choice fits the GPU and the scratch."""
import random

import numpy as np
import pytest

import paper_2502_08141_b200 as lw
import synth_inputs as si


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2502_08141_b200 import build
    build.build()


def layout_of(N, K, mix):
    return lw.Layout(si.precisions(N, mix, matrix_id=1), K, device="cpu")


def test_every_choice_fits():
    rng = random.Random(3)
    seen = set()
    for _ in range(400):
        N, K, r = 8 * rng.randint(32, 1728), 128 * rng.randint(4, 108), rng.choice([16, 48, 64, 80, 128])
        mix = rng.choice([{1: 0.5, 2: 0.5}, {4: 1.0}, {1: 0.6, 2: 0.35, 4: 0.05}])
        count = rng.choice([1, 1, 1, 2, 4])
        tokens = [int(round(2 ** rng.uniform(0, 13))) for _ in range(count)]
        layout = layout_of(N, K, mix)
        for backward in (False, True):
            c = lw.lowra_diag_choose(layout, backward, tokens, r)
            if c["few_tokens"]:
                assert not backward and max(tokens) <= 64 and c["tile_tokens"] == 0
                continue
            assert backward or max(tokens) > 16
            tiles = [-(-m // c["tile_tokens"]) for m in tokens]
            rows, blocks = -(-(K if backward else N) // 256), -(-(N if backward else K) // 64) + -(-r // 64)
            assert c["tile_tokens"] in (256, 512) and 1 <= c["clusters"] <= 74
            if c["w_split"] > 1:
                assert c["clusters"] == sum(tiles) * (rows * c["w_split"] + c["t_split"]) and blocks // c["w_split"] >= 12
            if c["t_split"] > 1:
                assert sum(tiles) * c["t_split"] < 74 and c["t_split"] <= 7
            seen.add((c["tile_tokens"], c["w_split"] > 1, c["t_split"] > 1))
    assert len(seen) >= 6, seen


def test_groups_of_few_tokens():
    layout = layout_of(4096, 4096, {1: 0.3, 2: 0.5, 4: 0.2})
    assert lw.lowra_diag_choose(layout, False, [1], 64)["units"] == 0
    assert lw.lowra_diag_choose(layout, False, [17, 17, 17, 17, 17, 16], 64, one_weight=True)["units"] == 1
    assert lw.lowra_diag_choose(layout, False, [8] * 8, 64)["units"] == 0          # weights of their own


@pytest.mark.parametrize("N,K,r,mix,tokens,units", [
    (264, 512, 16, {2: 0.75, 4: 0.25}, [44], 0),                  # wide units of 4-bit rows: slower than the slices (9.1 us, 7.9)
    (1720, 512, 48, {4: 1.0}, [34], 0),
    (4528, 640, 64, {1: 0.5, 2: 0.5}, [58], 1),                   # faster without 4-bit rows (8.6 us, 10.2)
    (4632, 512, 64, {1: 0.85, 2: 0.15}, [1] * 8, 1),
    (5800, 640, 64, {1: 0.3, 2: 0.5, 4: 0.2}, [8] * 7, 1),        # and with them in narrow units
])
def test_units_where_they_are_faster(N, K, r, mix, tokens, units):
    assert lw.lowra_diag_choose(layout_of(N, K, mix), False, tokens, r, one_weight=True) == dict(few_tokens=1, units=units, tile_tokens=0, clusters=0,
                                                                                                 w_split=1, t_split=1)


@pytest.mark.parametrize("N,K,M,r,mix,backward,choice", [
    # 512-token tiles shared by three clusters took 34.7 and 36.1 us, their estimates counted the T tile's second 64 ranks as nothing
    (2672, 1152, 1437, 128, {1: 0.85, 2: 0.15}, True, dict(tile_tokens=256, w_split=1)),         # 28.4
    (5016, 2944, 404, 128, {1: 0.5, 2: 0.5}, False, dict(tile_tokens=256, w_split=1)),           # 30.8
    (9184, 6016, 77, 64, {1: 0.3, 2: 0.5, 4: 0.2}, True, dict(clusters=74, t_split=2)),          # 45 - 47; two clusters a tile, on 55, 54.5
    # on all SMs, tiles of 256 tokens: the first cluster of a tile finishes it
    (5888, 4352, 168, 64, {1: 0.85, 2: 0.15}, False, dict(clusters=74, w_split=1, t_split=5)),   # 27.8; shared 32.0
    (3224, 8832, 209, 128, {1: 0.85, 2: 0.15}, True, dict(clusters=74, w_split=1, t_split=4)),   # 28.3; shared 32.9
    (4096, 4096, 128, 64, {1: 0.6, 2: 0.4}, False, dict(tile_tokens=256, w_split=4, t_split=7)),
    (7016, 4608, 36, 64, {2: 0.75, 4: 0.25}, False, dict(few_tokens=0)),                          # 33; few-token path 43
    (2048, 2048, 64, 64, {1: 0.6, 2: 0.4}, False, dict(few_tokens=1)),                            # 12; tiles 21
])
def test_measured_choices(N, K, M, r, mix, backward, choice):
    got = lw.lowra_diag_choose(layout_of(N, K, mix), backward, [M], r)
    assert {k: got[k] for k in choice} == choice


@pytest.mark.parametrize("tokens,r,code", [([0], 64, "SHAPE"), ([1] * 9, 64, "SHAPE"), ([100] * 5, 64, "SHAPE"), ([1], 24, "SHAPE")])
def test_refusals(tokens, r, code):
    with pytest.raises(lw.LowraError) as e:
        lw.lowra_diag_choose(layout_of(512, 512, {2: 1.0}), False, np.array(tokens), r)
    assert e.value.code == getattr(lw, "LOWRA_ERR_" + code)
