"""What a workspace carries from call to call: the flags of the fused calls, which are "up" when they hold the number of the call,
must never lie where another call leaves its down-projected tokens (whose bits can be any number); and calls of so many tokens
that their flags do not fit beside the others.
"""
import numpy as np
import pytest
import torch

import synth_inputs as si
from helpers import FRO_TOL, MAX_TOL, gemm_errors

pytestmark = pytest.mark.gpu


class _Problem:
    def __init__(self, N, K, r, dealt=True, adapters=1):
        import paper_2502_08141_b200 as lw

        self.lw, self.N, self.K, self.r = lw, N, K, r
        self.gen = torch.Generator(device="cuda").manual_seed(N + K + r)
        precs = si.precisions(N, {1: 0.3, 2: 0.5, 4: 0.2}, matrix_id=7)
        self.layout = lw.Layout(precs, K)
        if dealt:
            self.layout.build_deal()
        maps, thr = (torch.from_numpy(t).cuda() for t in si.standin_codebooks(precs))
        self.maps = maps
        self.packed, self.absmax = lw.lowra_encode(self.layout, self.draw(N, K).float(), thr)
        self.A, self.B = self.draw(K, r) * 0.05, self.draw(r, N) * 0.05

    def draw(self, *shape):
        return torch.randn(*shape, device="cuda", generator=self.gen).bfloat16()

    def call(self, backward, act, ws):
        f = self.lw.lowra_lora_backward_input if backward else self.lw.lowra_lora_forward
        return f(self.layout, self.packed, self.absmax, self.maps, act, self.A, self.B, 2.0, workspace=ws)

    def right(self, backward, act, out, rows):
        W = self.lw.lowra_decode(self.layout, self.packed, self.absmax, self.maps).double()
        a, A, B = act[rows].double(), self.A.double(), self.B.double()
        ref = a @ W + 2.0 * (a @ B.T) @ A.T if backward else a @ W.T + 2.0 * (a @ A) @ B
        emax, efro = gemm_errors(out[rows].float().cpu().numpy(), ref.cpu().numpy())
        return emax <= MAX_TOL and efro <= FRO_TOL


@pytest.mark.parametrize("backward", [False, True])
@pytest.mark.parametrize("M", [70, 300, 1000])
def test_no_flag_is_read_from_old_projections(backward, M):
    """A call whose "T ready" flags are withheld has to run out of time, also where an earlier call of more tokens has left
    T values with the bits of this call's number."""
    p = _Problem(512, 640, 64)
    lw = p.lw
    ws = lw.lowra_workspace_init(torch.empty(lw.lowra_workspace_bytes(p.layout, 2000, p.r), dtype=torch.uint8, device="cuda"))
    act = p.draw(M, p.N if backward else p.K)
    lw.lowra_workspace_projection(ws, 2000, p.r).view(torch.int32).fill_(1)     # the first call's number
    lw.lowra_set_wait_limit(2_000_000)
    try:
        lw.lowra_diag_drop_t_flags(1)
        p.call(backward, act, ws)
        assert lw.lowra_device_status(ws) == lw.LOWRA_ERR_TIMEOUT
    finally:
        lw.lowra_diag_drop_t_flags(0)
        lw.lowra_set_wait_limit(0)
    lw.lowra_workspace_init(ws)
    assert p.right(backward, act, p.call(backward, act, ws), slice(None))
    assert lw.lowra_device_status(ws) == lw.LOWRA_OK


def test_groups_of_few_and_of_many_tokens_keep_apart():
    """Several adapters, one of them with a few tokens: its projection (at its tokens' rows) is written before the larger
    group's launch raises its flags."""
    p = _Problem(512, 640, 64)
    lw, M = p.lw, 316
    X = p.draw(M, p.K)
    two = lambda t: torch.stack([t, t])
    ws = lw.lowra_workspace_init(torch.empty(lw.lowra_batch_workspace_bytes(p.layout, 4, M, p.r), dtype=torch.uint8, device="cuda"))
    Y = lw.lowra_lora_forward_adapters(p.layout, p.packed, p.absmax, two(p.maps), X, [0, 300, M], two(p.A), two(p.B), 2.0, workspace=ws)
    left = lw.lowra_workspace_projection(ws, M, p.r)[300:].clone()
    assert lw.lowra_device_status(ws) == lw.LOWRA_OK and p.right(False, X, Y, slice(None))
    own = lw.lowra_workspace_init(torch.empty_like(ws))
    p.call(False, X[300:].contiguous(), own)
    assert torch.equal(left.view(torch.int16), lw.lowra_workspace_projection(own, M - 300, p.r).view(torch.int16))


def test_every_group_is_served_while_flags_are_withheld():
    """The diagnostic keeps the few-token groups on the tensor-core tiles; the first group's launch uses it up, and the
    second group must not fall between the two paths."""
    p = _Problem(512, 640, 64, dealt=False)
    lw, M = p.lw, 308
    X = p.draw(M, p.K)
    two = lambda t: torch.stack([t, t])
    ws = torch.empty(lw.lowra_workspace_bytes(p.layout, M, p.r), dtype=torch.uint8, device="cuda")
    Y = torch.full((M, p.N), float("nan"), dtype=torch.bfloat16, device="cuda")
    lw.lowra_set_wait_limit(2_000_000)
    try:
        lw.lowra_diag_drop_t_flags(1)
        lw.lowra_lora_forward_adapters(p.layout, p.packed, p.absmax, two(p.maps), X, [0, 300, M], two(p.A), two(p.B), 2.0, Y=Y, workspace=ws)
        assert p.right(False, X, Y, slice(300, M))
    finally:
        torch.cuda.synchronize()
        lw.lowra_diag_drop_t_flags(0)
        lw.lowra_set_wait_limit(0)


def test_initialising_touches_the_header_only():
    """A call that brings no workspace pays for one each time: what is cleared does not grow with the workspace, and what is not cleared
    is not relied on."""
    p = _Problem(512, 640, 64)
    lw = p.lw
    ws = torch.empty(lw.lowra_workspace_bytes(p.layout, 600, p.r), dtype=torch.uint8, device="cuda").fill_(0xA5)
    lw.lowra_workspace_init(ws)
    assert not bool(ws[:4096].any()) and bool((ws[4096:] == 0xA5).all())
    for M in (600, 300, 10, 600):
        for backward in (False, True):
            act = p.draw(M, p.N if backward else p.K)
            assert p.right(backward, act, p.call(backward, act, ws), slice(None))
    assert lw.lowra_device_status(ws) == lw.LOWRA_OK


def test_scratch_of_a_call_belongs_to_its_stream(monkeypatch):
    """A call on a stream of its own, with no workspace passed: cleared on that stream and taken from its memory, not the current one's."""
    p = _Problem(512, 640, 64)
    lw = p.lw
    side = torch.cuda.Stream()
    X, dY = p.draw(300, p.K), p.draw(300, p.N)
    torch.cuda.synchronize()
    seen = []
    init, empty = lw.lowra_workspace_init, torch.empty
    monkeypatch.setattr(lw, "lowra_workspace_init", lambda ws, stream=None: (seen.append(stream), init(ws, stream))[1])

    def record(*size, **kw):
        if kw.get("dtype") is torch.uint8:
            seen.append(torch.cuda.current_stream())
        return empty(*size, **kw)
    monkeypatch.setattr(lw.torch, "empty", record)
    Y = lw.lowra_lora_forward(p.layout, p.packed, p.absmax, p.maps, X, p.A, p.B, 2.0, stream=side)
    dX = lw.lowra_lora_backward_input(p.layout, p.packed, p.absmax, p.maps, dY, p.A, p.B, 2.0, stream=side)
    lw.lowra_lora_backward_adapters(X, dY, p.A, p.B, 2.0, stream=side)
    monkeypatch.undo()
    side.synchronize()
    assert len(seen) == 5 and all(s == side for s in seen)
    assert p.right(False, X, Y, slice(None)) and p.right(True, dY, dX, slice(None))


OPTIONAL = 73 * 256 * 1024     # LOWRA_WORKSPACE_OPTIONAL


@pytest.mark.parametrize("dealt", [False, True])
@pytest.mark.parametrize("N,K,M", [(512, 640, 300), (1800, 2304, 777), (2304, 1792, 2500), (1800, 2304, 7500)])
def test_a_workspace_of_half_the_partial_tiles(N, K, M, dealt):
    """As large as it had to be while partial tiles held 256 tokens: still accepted, and nothing behind its end is written."""
    p = _Problem(N, K, 80, dealt)
    lw = p.lw
    least = lw.lowra_workspace_bytes(p.layout, M, p.r) - OPTIONAL
    # what was asked for then: status, T, one flag per 256 tokens and CTA, about 32 bytes a channel for the deal, 74 slots of 256 KB
    entries = 2 * (4 * ((N + 127) // 128) + 40)
    up = lambda x: (x + 255) // 256 * 256
    assert least <= 256 + up(M * 128 * 2) + up(((M + 255) // 256 + 2 + 148) * 4) + up(entries * 512) + up(entries * 4) + 74 * 262144
    whole = torch.empty(least + OPTIONAL, dtype=torch.uint8, device="cuda").fill_(0xA5)
    ws = whole[:least]
    if dealt:
        lw.lowra_workspace_init(ws)
    rows = torch.from_numpy(np.unique(np.linspace(0, M - 1, 500).astype(np.int64))).cuda()
    for backward in (False, True):
        act = p.draw(M, p.N if backward else p.K)
        for _ in range(2):
            out = p.call(backward, act, ws)
            assert lw.lowra_device_status(ws) == lw.LOWRA_OK and p.right(backward, act, out, rows)
        with pytest.raises(lw.LowraError) as e:
            p.call(backward, act, whole[:least - 1])
        assert e.value.code == lw.LOWRA_ERR_WORKSPACE
    assert bool((whole[least:] == 0xA5).all())


@pytest.mark.parametrize("dealt", [False, True])
def test_more_tokens_than_the_flags_have_room_for(dealt):
    """From about 104 000 tokens on the "T ready" flags lie behind T and are cleared by every call."""
    p = _Problem(136, 128, 16, dealt)
    lw = p.lw
    counts = [103_900, 300, 120_001, 120_001, 104_100]
    ws = torch.empty(lw.lowra_workspace_bytes(p.layout, max(counts), p.r), dtype=torch.uint8, device="cuda").fill_(0xA5)
    if dealt:
        lw.lowra_workspace_init(ws)
    acts = [p.draw(max(counts), p.K), p.draw(max(counts), p.N)]
    for M in counts:
        rows = torch.from_numpy(np.unique(np.linspace(0, M - 1, 4000).astype(np.int64))).cuda()
        for backward in (False, True):
            act = acts[backward][:M]
            out = p.call(backward, act, ws)
            assert lw.lowra_device_status(ws) == lw.LOWRA_OK
            assert p.right(backward, act, out, rows), (M, backward)
