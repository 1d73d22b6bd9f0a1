"""The extension module's batches, gradients of the factors and views of a workspace: what the interpreted way gives (a call that names its stream takes that), a status
where the library refuses, None for whatever the interpreted way is to look at."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu

N, K, M, r = 264, 384, 70, 48


def _weights(lw, gen, n):
    precs = si.precisions(N, {1: 0.3, 2: 0.5, 4: 0.2}, matrix_id=5)
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    out = []
    for _ in range(n):
        layout = lw.Layout(precs, K).build_deal()
        packed, absmax = lw.lowra_encode(layout, torch.randn(N, K, device="cuda", generator=gen), thr)
        out.append(dict(layout=layout, packed=packed, absmax=absmax, maps=maps))
    return out


@pytest.mark.parametrize("backward", [False, True])
def test_batches(backward):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(1)
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    members = [dict(w, act=draw(M, N if backward else K), A=draw(K, r), B=draw(r, N), out=torch.empty(M, K if backward else N, dtype=torch.bfloat16, device="cuda"))
               for w in _weights(lw, gen, 3)]
    ws = lw.lowra_workspace_init(torch.empty(lw.lowra_batch_workspace_bytes(members[0]["layout"], 3, M, r), dtype=torch.uint8, device="cuda"))
    call = lw.lowra_lora_backward_input_batch if backward else lw.lowra_lora_forward_batch
    want = [o.clone() for o in call(members, 2.0, ws, torch.cuda.current_stream())]
    for m in members:
        m["out"].fill_(float("nan"))
    got = lw._py_calls.batch(backward, members, 2, ws)
    assert type(got) is list and all(o is m["out"] and torch.equal(o, w) for o, m, w in zip(got, members, want)) and len(got) == 3
    assert lw._py_calls.batch(backward, members, 2.0, ws[:256]) == lw.LOWRA_ERR_WORKSPACE
    with pytest.raises(lw.LowraError):
        call(members, 2.0, ws[:256])
    last = members[2]
    for left in (dict(act=last["act"].float()), dict(act=last["act"][:-1]), dict(out=last["out"].t().contiguous().t()), dict(A=draw(K, 32)), dict(maps=None),
                 dict(packed=last["packed"][:-1]), dict(layout=None), dict(B=last["B"].cpu())):
        assert lw._py_calls.batch(backward, members[:2] + [{**last, **left}], 2.0, ws) is None, left.keys()
    for args in ((backward, tuple(members), 2.0, ws), (backward, [], 2.0, ws), (backward, members + members, 2.0, ws), (backward, members, "2", ws),
                 (backward, members, 2.0, ws.cpu()), (backward, [{k: v for k, v in last.items() if k != "out"}], 2.0, ws)):
        assert lw._py_calls.batch(*args) is None
    with pytest.raises(ValueError):
        call(members[:2] + [dict(last, act=last["act"][:-1])], 2.0, ws)


@pytest.mark.parametrize("reuse", [False, True])
def test_gradients(reuse):
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(2)
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    X, dY, rp = draw(M, K), draw(M, N), 64
    if reuse:
        names, values = ("X", "dY", "T", "U", "r", "dA", "dB", "workspace"), (X, dY, draw(M, rp), draw(M, rp), r, None, None, None)
        native, call = lw._py_calls.gradients_reuse, lw.lowra_lora_backward_adapters_reuse
    else:
        names, values = ("X", "dY", "A", "B", "s", "dA", "dB", "workspace"), (X, dY, draw(K, r), draw(r, N), 2.0, None, None, None)
        native, call = lw._py_calls.gradients, lw.lowra_lora_backward_adapters
    ordinary = dict(zip(names, values))
    ask = lambda **change: native(*{**ordinary, **change}.values())
    want = call(*values, stream=torch.cuda.current_stream())
    same = lambda got: type(got) is tuple and all(torch.equal(a, b) and a.shape == b.shape and not a.requires_grad for a, b in zip(got, want))
    assert same(ask()) and same(call(*values)) and same(ask(X=torch.nn.Parameter(X)))
    dA, dB = torch.empty_like(want[0]), torch.empty_like(want[1])
    ws = torch.empty(lw.lowra_adapter_workspace_bytes(M, r), dtype=torch.uint8, device="cuda")
    got = ask(dA=dA, dB=dB, workspace=ws)
    assert got[0] is dA and got[1] is dB and same(got)
    assert ask(workspace=ws[:16]) == lw.LOWRA_ERR_WORKSPACE
    third = names[2]
    for left in (dict(X=X.float()), dict(X=X.t().contiguous().t()), dict(dY=dY[:-1]), dict(dY=dY.cpu()), {third: ordinary[third][:-1]}, {third: None}, dict(dA=dA[:-1]),
                 dict(dB=dB.float()), dict(workspace=ws.cpu()), {names[4]: "2"}, {names[4]: None}):
        assert ask(**left) is None, left.keys()


def test_projections():
    import paper_2502_08141_b200 as lw

    layout = lw.Layout(si.precisions(N, {1: 0.5, 2: 0.5}, matrix_id=5), K)
    ws = torch.empty(lw.lowra_batch_workspace_bytes(layout, 3, M, r), dtype=torch.uint8, device="cuda")
    for member in range(3):
        native, p = lw._py_calls.projection(ws, M, r, member), lw.lib().lowra_workspace_projection(ws.data_ptr(), member, M, r)
        assert native.shape == (M, 64) and native.dtype == torch.bfloat16 and native.data_ptr() == p and native.untyped_storage().data_ptr() == ws.untyped_storage().data_ptr()
        assert lw.lowra_workspace_projection(ws, M, r, member).data_ptr() == p
    for args in ((ws.cpu(), M, r, 0), (ws[:256], M, r, 0), (ws, M, 24, 0), (ws, M, r, -1), (ws, str(M), r, 0), (ws.view(torch.int8), M, r, 0), (None, M, r, 0)):
        assert lw._py_calls.projection(*args) is None
