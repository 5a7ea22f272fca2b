"""DecodeGraph.step on a token's own tensors (the graph's node is pointed at them), on ones that have to be copied first,
and replay() on what the buffers hold: the same outputs, states and caches as the eager fused call, bit for bit."""
import pytest
import torch

import paper_2402_18668_b200 as based
from paper_2402_18668_b200.generation import DecodeGraph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("B,H,d_v,window,sym", [(1, 3, 64, 16, False), (2, 16, 128, 64, True), (5, 7, 112, 100, False),
                                                (40, 16, 128, 64, True)])
def test_step_equals_the_eager_call(dtype, B, H, d_v, window, sym):
    g = torch.Generator(device="cuda").manual_seed(B + d_v)
    rnd = lambda *s, dt=dtype: torch.randn(*s, generator=g, device="cuda").to(dt)
    kv, z = based.new_state(B, H, d_v, sym=sym)
    kv.copy_(rnd(*kv.shape)); z.copy_(rnd(*z.shape).abs() + 5.0)
    kc, vc = rnd(B, H, window, 64), rnd(B, H, window, 64)
    eager = [t.clone() for t in (kv, z, kc, vc)]
    pos = torch.tensor([window - 2, 0], dtype=torch.int32, device="cuda")
    graph = DecodeGraph(kv, z, kc, vc, pos=window - 2, dtype=dtype, sym=sym)
    token = None
    for kind in ("own", "own", "strided", "replay", "own", "other dtype", "buffers", "swapped buffers", "replay"):
        if kind == "replay":
            got = [t.clone() for t in (graph.replay(), graph.out_lin, graph.out_swa)[1:]]
        else:
            token = [rnd(B, H, 16), rnd(B, H, 16), rnd(B, H, d_v), rnd(B, H, 64), rnd(B, H, 64), rnd(B, H, 64)]
            given = token
            if kind == "strided":
                given = [torch.stack([t, t], dim=-1)[..., 0] for t in token]
            elif kind == "other dtype":                    # bf16 values in the other type: the conversion is exact
                token = [t.bfloat16().to(dtype) for t in token]
                given = [t.to(torch.float32 if dtype == torch.bfloat16 else torch.bfloat16) for t in token]
            elif kind == "buffers":
                given = [graph.q, graph.k, graph.v, graph.qw, graph.kw, graph.vw]
                token = [t.clone() for t in given]
            elif kind == "swapped buffers":                # copied one after the other: q from k's buffer, then k from q's new one
                given = [graph.k, graph.q, graph.v, graph.qw, graph.kw, graph.vw]
                token = [graph.k.clone(), graph.k.clone()] + [t.clone() for t in given[2:]]
            got = [t.clone() for t in graph.step(*given)]
        want = based.based_generation_step(*token[:3], *eager[:2], *token[3:], *eager[2:], pos,
                                           flags=based.BASED_STATE_SYM if sym else 0)
        for a, b in zip(got + [kv, z, kc, vc, graph.q, graph.k, graph.v, graph.qw, graph.kw, graph.vw],
                        list(want) + eager + token):
            assert torch.equal(a, b), kind
        assert int(graph.pos) == int(pos[0]) and based.based_poll_error() == based.BASED_OK


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("place,source", [("v", "out_swa"), ("v", "out_lin"), ("qw", "out_swa"), ("vw", "out_swa"), ("kw", "kc"),
                                          ("qw", "kv")])
def test_step_on_what_the_step_writes(dtype, place, source):
    """Inputs that lie in an output of the step before (B 40: many CTAs, so that some write while others still read), a cache
    or the state are copied first: the outputs, and what the buffers and a replay() hold, are those of the values."""
    B, H = 40, 16
    window = 1 if source == "kc" else 64
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    kv, z = based.new_state(B, H, 64)
    kv.copy_(rnd(*kv.shape)); z.copy_(rnd(*z.shape).abs() + 50.0)
    kc, vc = rnd(B, H, window, 64).to(dtype), rnd(B, H, window, 64).to(dtype)
    eager = [t.clone() for t in (kv, z, kc, vc)]
    pos = torch.tensor([70, 0], dtype=torch.int32, device="cuda")
    graph = DecodeGraph(kv, z, kc, vc, pos=70, dtype=dtype)
    names = ("q", "k", "v", "qw", "kw", "vw")
    for turn in range(3):
        token = {n: rnd(B, H, 16 if n in "qk" else 64).to(dtype) for n in names}
        if turn > 0:                            # (the first step gives the outputs their values)
            token[place] = {"out_swa": graph.out_swa, "out_lin": graph.out_lin, "kc": kc[:, :, 0],
                            "kv": kv.view(dtype).view(-1)[:B * H * 64].view(B, H, 64)}[source]
        values = [token[n].clone() for n in names]
        for replay in (False, True):
            got = [t.clone() for t in (graph.step(*(token[n] for n in names)) if not replay else
                                       (graph.replay(), graph.out_lin, graph.out_swa)[1:])]
            want = based.based_generation_step(*values[:3], *eager[:2], *values[3:], *eager[2:], pos)
            for a, b in zip(got + [kv, z, kc, vc] + [getattr(graph, n) for n in names], list(want) + eager + values):
                assert torch.equal(torch.nan_to_num(a.float()), torch.nan_to_num(b.float())), (turn, replay)
    assert based.based_poll_error() == based.BASED_OK


@pytest.mark.skipif(not torch.cuda.is_available() or torch.cuda.device_count() < 2, reason="needs a second device")
def test_step_on_a_device_that_is_not_current():
    """A graph on cuda:1 while cuda:0 is current: every step runs on cuda:1's current stream, ordered with the copies there."""
    with torch.cuda.device(1):
        g = torch.Generator(device="cuda").manual_seed(9)
        rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
        kv, z = based.new_state(2, 4, 64)
        kv.copy_(rnd(*kv.shape)); z.copy_(rnd(*z.shape).abs() + 50.0)
        kc, vc = rnd(2, 4, 64, 64).bfloat16(), rnd(2, 4, 64, 64).bfloat16()
        eager = [t.clone() for t in (kv, z, kc, vc)]
        pos = torch.tensor([70, 0], dtype=torch.int32, device="cuda")
        token = [rnd(2, 4, w).bfloat16() for w in (16, 16, 64, 64, 64, 64)]
    assert torch.cuda.current_device() == 0
    graph = DecodeGraph(kv, z, kc, vc, pos=70)
    for kind in ("own", "copied", "replay"):
        given = [t.float() for t in token] if kind == "copied" else token
        got = [t.clone() for t in ((graph.replay(), graph.out_lin, graph.out_swa)[1:] if kind == "replay" else graph.step(*given))]
        with torch.cuda.device(1):
            want = based.based_generation_step(*token[:3], *eager[:2], *token[3:], *eager[2:], pos)
        for a, b in zip(got + [kv, z, kc, vc], list(want) + eager):
            assert torch.equal(a, b), kind


@pytest.mark.parametrize("B,sym", [(2, False), (40, True)])
def test_steps_on_streams_in_turn(B, sym):
    """Steps of one graph on three streams in turn, without a wait between them: each runs behind the one before it."""
    H, d_v = 16, 128
    g = torch.Generator(device="cuda").manual_seed(B)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    kv, z = based.new_state(B, H, d_v, sym=sym)
    kv.copy_(rnd(*kv.shape)); z.copy_(rnd(*z.shape).abs() + 50.0)
    kc, vc = rnd(B, H, 64, 64).bfloat16(), rnd(B, H, 64, 64).bfloat16()
    eager = [t.clone() for t in (kv, z, kc, vc)]
    pos = torch.tensor([60, 0], dtype=torch.int32, device="cuda")
    tokens = [[rnd(B, H, w).bfloat16() for w in (16, 16, d_v, 64, 64, 64)] for _ in range(12)]
    graph = DecodeGraph(kv, z, kc, vc, pos=60, sym=sym)
    streams = [torch.cuda.current_stream(), torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    for i, t in enumerate(tokens):
        with torch.cuda.stream(streams[(i * i + i // 3) % 3]):
            graph.step(*t)
    torch.cuda.synchronize()
    for t in tokens:
        want = based.based_generation_step(*t[:3], *eager[:2], *t[3:], *eager[2:], pos, flags=based.BASED_STATE_SYM if sym else 0)
    for a, b in zip([graph.out_lin, graph.out_swa, kv, z, kc, vc], list(want) + eager):
        assert torch.equal(a, b)
    assert int(graph.pos) == 72 and based.based_poll_error() == based.BASED_OK


def test_step_under_capture_is_refused():
    kv, z = based.new_state(1, 2, 64)
    kc = torch.zeros(1, 2, 16, 64, dtype=torch.bfloat16, device="cuda")
    graph = DecodeGraph(kv, z, kc, torch.zeros_like(kc), pos=3)
    token = [torch.ones(1, 2, w, dtype=torch.bfloat16, device="cuda") for w in (16, 16, 64, 64, 64, 64)]
    with pytest.raises(Exception):
        with torch.cuda.graph(torch.cuda.CUDAGraph()):
            graph.step(*token)
    graph.step(*token)
    assert int(graph.pos) == 4
