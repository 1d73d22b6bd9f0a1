"""The products' native way through the binding against the interpreted one (which a stream argument takes): the same results, memory handed
in or not, with and without a deal, and the same refusals."""
import pytest
import torch

import synth_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 70])
@pytest.mark.parametrize("dealt", [False, True])
def test_same_as_the_interpreted_way(M, dealt):
    import paper_2502_08141_b200 as lw

    N, K, r = 264, 384, 16
    gen = torch.Generator(device="cuda").manual_seed(M)
    draw = lambda *shape: torch.randn(*shape, device="cuda", generator=gen).bfloat16()
    precs = si.precisions(N, {1: 0.3, 2: 0.5, 4: 0.2}, matrix_id=5)
    layout = lw.Layout(precs, K)
    if dealt:
        layout.build_deal()
    maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
    packed, absmax = lw.lowra_encode(layout, draw(N, K).float(), thr)
    A, B = draw(K, r), draw(r, N)
    assert lw._py_calls is not None
    for call, act, cols in ((lw.lowra_lora_forward, draw(M, K), N), (lw.lowra_lora_backward_input, draw(M, N), K)):
        args = (layout, packed, absmax, maps, act, A, B)
        long_way = call(*args, 2.0, stream=torch.cuda.current_stream())
        assert torch.equal(call(*args, 2.0), long_way)
        assert torch.equal(call(*args, 2), long_way)
        assert torch.equal(call(layout, packed, absmax, maps, torch.nn.Parameter(act), A, B, 2.0), long_way)
        ws = lw.lowra_workspace_init(torch.empty(lw.lowra_workspace_bytes(layout, M, r), dtype=torch.uint8, device="cuda"))
        out = torch.empty(M, cols, dtype=torch.bfloat16, device="cuda")
        assert call(*args, 2.0, out, ws) is out and torch.equal(out, long_way)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            other = call(*args, 2.0)
        side.synchronize()
        assert torch.equal(other, long_way)
        with pytest.raises(ValueError, match="shape"):
            call(layout, packed, absmax, maps, act[:, :-64].contiguous(), A, B, 2.0)
        with pytest.raises(ValueError, match="contiguous"):
            call(layout, packed, absmax, maps, act, A.t().contiguous().t(), B, 2.0)
        with pytest.raises(ValueError, match="bfloat16"):
            call(layout, packed, absmax, maps, act.float(), A, B, 2.0)
        with pytest.raises(lw.LowraError) as refused:
            call(layout, packed, absmax, maps, act, draw(K, 24), draw(24, N), 2.0)
        assert refused.value.code == lw.LOWRA_ERR_SHAPE
        with pytest.raises(lw.LowraError) as refused:
            call(*args, 2.0, out, ws[:256])
        assert refused.value.code == lw.LOWRA_ERR_WORKSPACE
