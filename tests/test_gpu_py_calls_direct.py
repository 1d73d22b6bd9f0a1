"""The extension module's own answers: an output for the ordinary call, a status where the library refuses, None for whatever the interpreted way
is to look at - so that a native way which never answers does not pass for one that does."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu

N, K, M, r = 264, 384, 5, 16


@pytest.mark.parametrize("dealt", [False, True])
@pytest.mark.parametrize("backward", [False, True])
def test_answers(dealt, backward):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(1)
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    precs = si.precisions(N, {1: 0.3, 2: 0.5, 4: 0.2}, matrix_id=5)
    layout = lw.Layout(precs, K)
    if dealt:
        layout.build_deal()
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    packed, absmax = lw.lowra_encode(layout, draw(N, K).float(), thr)
    cols, act = (K, draw(M, N)) if backward else (N, draw(M, K))
    names = ("address", "device", "packed", "absmax", "maps", "act", "A", "B", "s", "out", "workspace")
    ordinary = dict(zip(names, (layout.address, layout.device_index, packed, absmax, maps, act, draw(K, r), draw(r, N), 2.0, None, None)))
    ask = lambda **change: (lw._py_calls.backward_input if backward else lw._py_calls.forward)(*{**ordinary, **change}.values())
    want = ask()
    assert type(want) is torch.Tensor and want.shape == (M, cols) and not want.requires_grad
    ws = lw.lowra_workspace_init(torch.empty(lw.lowra_workspace_bytes(layout, M, r), dtype=torch.uint8, device="cuda"))
    out = torch.empty(M, cols, dtype=torch.bfloat16, device="cuda")
    assert ask(out=out, workspace=ws) is out and torch.equal(out, want)
    for good in (dict(s=2), dict(act=torch.nn.Parameter(act)), dict(A=torch.nn.Parameter(ordinary["A"])), dict(packed=packed.view(torch.int8))):
        assert torch.equal(ask(**good), want), good.keys()
    assert ask(workspace=ws[:256]) == lw.LOWRA_ERR_WORKSPACE
    assert ask(A=draw(K, 24), B=draw(24, N), workspace=ws) == lw.LOWRA_ERR_SHAPE

    class Sub(torch.Tensor):
        pass

    for left in (dict(device=layout.device_index + 1), dict(act=act.float()), dict(act=act.cpu()), dict(act=act[:, :-64].contiguous()), dict(act=act.as_subclass(Sub)),
                 dict(A=ordinary["A"].t().contiguous().t()), dict(B=draw(r + 16, N)), dict(maps=maps.double()), dict(maps=maps[:-1]), dict(absmax=absmax[:-1]),
                 dict(packed=packed[:-1]), dict(packed=None), dict(out=out[:-1]), dict(out=out.float()), dict(workspace=ws.cpu()), dict(s="2"), dict(s=None),
                 dict(A=draw(K, 24), B=draw(24, N))):
        assert ask(**left) is None, left.keys()
