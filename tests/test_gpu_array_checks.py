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
