"""Arrays that the kernels would read or write out of range, or misread, are refused on the host, by either way through the binding; what is longer
than needed, of another shape, or page-locked host memory is taken as ever."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu

N, K, M, r = 264, 384, 5, 16


@pytest.fixture(scope="module")
def problem():
    import paper_2502_08141_b200 as lw

    gen = torch.Generator(device="cuda").manual_seed(1)
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    precs = si.precisions(N, {1: 0.3, 2: 0.5, 4: 0.2}, matrix_id=5)
    layout = lw.Layout(precs, K)
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    packed, absmax = lw.lowra_encode(layout, draw(N, K).float(), thr)
    return dict(lw=lw, layout=layout, packed=packed, absmax=absmax, maps=maps, A=draw(K, r), B=draw(r, N), X=draw(M, K), dY=draw(M, N))


def product(p, backward, native, **change):
    lw, q = p["lw"], {**p, **change}
    call, act = (lw.lowra_lora_backward_input, q["dY"]) if backward else (lw.lowra_lora_forward, q["X"])
    stream = None if native else torch.cuda.current_stream()
    return call(q["layout"], q["packed"], q["absmax"], q["maps"], act, q["A"], q["B"], 2.0, q.get("out"), q.get("workspace"), stream)


@pytest.mark.parametrize("native", [False, True])
@pytest.mark.parametrize("backward", [False, True])
def test_products(problem, backward, native):
    p, cols = problem, K if backward else N
    run = lambda **change: product(p, backward, native, **change)
    new = lambda *shape, dtype=torch.bfloat16: torch.empty(*shape, dtype=dtype, device="cuda")
    want = run()
    for change, says in ((dict(out=new(M - 1, cols)), "elements"), (dict(out=new(M, cols, dtype=torch.float32)), "bfloat16"),
                         (dict(out=new(M, 2 * cols)[:, ::2]), "contiguous"), (dict(out=torch.empty(M, cols).bfloat16()), "CUDA"),
                         (dict(maps=p["maps"].double()), "float32"), (dict(maps=p["maps"].bfloat16()), "float32"), (dict(maps=p["maps"][:-1]), "elements"),
                         (dict(maps=p["maps"].cpu()), "CUDA"), (dict(absmax=p["absmax"][:, :-1].contiguous()), "elements"),
                         (dict(absmax=p["absmax"].double()), "float32"), (dict(packed=p["packed"][:-1]), "bytes"), (dict(packed=p["packed"].cpu()), "CUDA"),
                         (dict(workspace=torch.empty(1 << 20, dtype=torch.uint8)), "CUDA"), (dict(workspace=new(1 << 20, dtype=torch.uint8)[::2]), "contiguous")):
        with pytest.raises(ValueError, match=says):
            run(**change)
    longer = new(M + 3, cols)
    longer[M:] = 7.0
    assert run(out=longer) is longer and torch.equal(longer[:M], want) and bool((longer[M:] == 7.0).all())
    for change in (dict(out=new(M * cols)), dict(maps=p["maps"].view(-1)), dict(packed=p["packed"].view(torch.int8)), dict(maps=p["maps"].cpu().pin_memory()),
                   dict(absmax=torch.cat([p["absmax"], p["absmax"]]))):
        assert torch.equal(run(**change).view(-1), want.view(-1)), change.keys()


def refused(call, changes):
    call()
    for change, says in changes:
        with pytest.raises(ValueError, match=says):
            call(**change)


@pytest.mark.parametrize("native", [False, True])
def test_codec_learner_and_errors(problem, native, monkeypatch):
    p, lw, layout = problem, problem["lw"], problem["layout"]
    if not native:      # as for an interpreter without an extension module of its own
        monkeypatch.setattr(lw, "_fits", lw._no_verdict)
    new = lambda *shape, dtype=torch.float32: torch.empty(*shape, dtype=dtype, device="cuda")
    W, thr = torch.randn(N, K, device="cuda"), p["maps"].sort().values
    short_packed, short_absmax = p["packed"][:-1], new(N, K // 64 - 1)
    outs = ((dict(packed=short_packed), "packed"), (dict(absmax=short_absmax), "absmax"))
    refused(lambda **k: lw.lowra_encode(layout, W, thr, **k), outs)
    refused(lambda **k: lw.lowra_encode_group([dict(layout=layout, W=W, thresholds=thr, **k)]), outs)
    one = dict(layout=layout, packed=p["packed"], absmax=p["absmax"], maps=p["maps"])
    outs += ((dict(maps=p["maps"][:-1]), "maps"), (dict(out=new(N - 1, K, dtype=torch.bfloat16)), "out"))
    refused(lambda **k: lw.lowra_decode(**{**one, **k}), outs)
    refused(lambda **k: lw.lowra_decode_group([{**one, **k}]), outs)
    offsets = torch.from_numpy(lw.lowra_natural_offsets(layout.precs_host, K).view("int64")).cuda()
    refused(lambda **k: lw.lowra_reorder_rows(**{**dict(layout=layout, to_natural=True, offsets=offsets, packed=p["packed"], absmax=p["absmax"]), **k}),
            ((dict(packed=short_packed), "packed"), (dict(absmax=short_absmax), "absmax"), (dict(packed_out=short_packed), "packed_out"),
             (dict(absmax_out=short_absmax), "absmax_out"), (dict(absmax_out=new(N, K // 64, dtype=torch.float64)), "absmax_out"), (dict(offsets=offsets.cpu()), "offsets")))
    levels = [[-0.5, 0.5] + [0.0] * 14, [-0.7, -0.2, 0.2, 0.7] + [0.0] * 12, [-1.0 + i / 8 for i in range(16)]]
    tables = ((dict(maps=new(N - 1, 16)), "maps"), (dict(thresholds=new(N - 1, 16)), "thresholds"))
    refused(lambda **k: lw.lowra_learn_codebooks(**{**dict(layout=layout, W=W, init_levels=levels, init_thresholds=levels, iterations=1), **k}),
            tables + ((dict(W=W[:-1]), "W"),))
    refused(lambda **k: lw.lowra_quant_error(layout, W, p["maps"], thr, **k), ((dict(sse=new(N - 1, dtype=torch.float64)), "sse"), (dict(sse=new(N)), "sse"),
                                                                               (dict(residual=new(N - 1, K)), "residual")))
    three = p["maps"].expand(3, N, 16).contiguous()
    refused(lambda **k: lw.lowra_channel_errors(W, three, three, **k), ((dict(sse3=new(N, 2, dtype=torch.float64)), "sse3"),))


@pytest.mark.parametrize("native", [False, True])
def test_other_products(problem, native, monkeypatch):
    p, lw = problem, problem["lw"]
    if not native:
        monkeypatch.setattr(lw, "_fits", lw._no_verdict)
    layout = lw.Layout(p["layout"].precs_host, K).build_deal()
    new = lambda *shape, dtype=torch.bfloat16: torch.empty(*shape, dtype=dtype, device="cuda")
    ws = lambda size: lw.lowra_workspace_init(torch.empty(size, dtype=torch.uint8, device="cuda"))
    weight = ((dict(packed=p["packed"][:-1]), "packed"), (dict(absmax=p["absmax"][:-1]), "absmax"), (dict(packed=p["packed"].cpu()), "packed"))
    host_ws = (dict(workspace=torch.empty(1 << 20, dtype=torch.uint8)), "workspace")
    size = lw.lowra_batch_workspace_bytes(layout, 4, M, r)
    for call, act, cols in ((lw.lowra_lora_forward_batch, "X", N), (lw.lowra_lora_backward_input_batch, "dY", K)):
        one = dict(layout=layout, packed=p["packed"], absmax=p["absmax"], maps=p["maps"], act=p[act], A=p["A"], B=p["B"], out=new(M, cols))
        refused(lambda workspace=ws(size), **k: call([{**one, **k}], 2.0, workspace), weight + ((dict(maps=p["maps"][:-1]), "maps"), (dict(maps=p["maps"].double()), "maps"), host_ws))
    one = dict(layout=layout, packed=p["packed"], absmax=p["absmax"], maps=p["maps"], X=p["X"], A=p["A"], B=p["B"], s=2.0)
    short_y = (dict(Y=new(M - 1, N)), "Y")
    refused(lambda **k: lw.lowra_lora_forward_static(**{**one, **k}), weight + ((dict(maps=p["maps"][:-1]), "maps"), short_y,
                                                                              (dict(status_out=new(2, dtype=torch.uint8)), "status_out")))
    many = {**one, **{k: one[k].unsqueeze(0).contiguous() for k in ("maps", "A", "B")}, "group_start": [0, M]}
    refused(lambda **k: lw.lowra_lora_forward_adapters(**{**many, **k}), weight + (short_y, host_ws))
    outs = ((dict(dA=new(K - 1, r)), "dA"), (dict(dB=new(r, N, dtype=torch.float32)), "dB"), host_ws)
    refused(lambda **k: lw.lowra_lora_backward_adapters(p["X"], p["dY"], p["A"], p["B"], 2.0, **k), outs)
    T = new(M, 64).zero_()
    refused(lambda **k: lw.lowra_lora_backward_adapters_reuse(p["X"], p["dY"], T, T, r, **k), outs)
    P = new(M, 128).zero_()
    refused(lambda **k: lw.lowra_dense_nt(**{**dict(P=P, Q=new(64, 128).zero_()), **k}), ((dict(Q=new(64, 64)), "Q"), (dict(C=new(M, 63)), "C"), host_ws))
