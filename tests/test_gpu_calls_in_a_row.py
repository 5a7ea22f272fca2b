"""Times of calls that follow one another, each as a dependent launch where that pays: a call does not slow the next one down, and fewer
heads do not take longer than more."""
import pytest
import torch

import paper_2402_18668_b200 as based

pytestmark = pytest.mark.gpu


def microseconds(*steps):
    """Each step's time, repeated in a graph; the least of ten turns, the steps in turn."""
    graphs = []
    for step in steps:
        step()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for _ in range(20):
                step()
        graphs.append(graph)
    best = [float("inf")] * len(steps)
    for _ in range(10):
        for i, graph in enumerate(graphs):
            start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            start.record()
            graph.replay()
            end.record()
            end.synchronize()
            best[i] = min(best[i], start.elapsed_time(end) * 50)
    return best


def inputs(BH, L, d, d_v):
    g = torch.Generator(device="cuda").manual_seed(BH + L)
    q, k = (torch.randn(1, BH, L, d, generator=g, device="cuda").mul(0.25).bfloat16() for _ in range(2))
    return q, k, torch.randn(1, BH, L, d_v, generator=g, device="cuda").bfloat16()


def prefill(BH, L, d, d_v, state=False):
    q, k, v = inputs(BH, L, d, d_v)
    out = torch.empty_like(v)
    kw = dict(zip(("kv_state", "z_state"), based.new_state(1, BH, d_v, d_feat=d))) if state else {}
    return lambda: based.based_prefill(q, k, v, out=out, **kw)


@pytest.mark.parametrize("d,d_v,BH,L,state", [(24, 64, 20, 4096, False), (8, 64, 40, 2048, False), (24, 64, 10, 4096, False),
                                              (32, 112, 10, 4096, True), (32, 112, 16, 2048, True)])
def test_behind_itself(d, d_v, BH, L, state):
    """Behind itself a call takes no longer than behind a small kernel, that one's time included (1.04 to 1.16 times as long where its
    long CTAs share the SMs that the call before leaves first)."""
    call, small = prefill(BH, L, d, d_v, state), torch.empty(256, device="cuda")

    def both():
        small.zero_()
        call()

    alone, behind = microseconds(call, both)
    assert alone <= 1.02 * behind


def backward(BH, L, d_v):
    q, k, v = inputs(BH, L, 16, d_v)
    out = based.based_prefill(q, k, v)
    dout = torch.randn_like(v)
    return lambda: based.based_prefill_backward(q, k, v, dout, out=out)


def test_backward_of_fewer_heads():
    """Two heads' block-wise backward is well below twelve heads' (0.95 of it while the scan of the block states was a dependent launch)."""
    two, twelve = microseconds(backward(2, 3000, 128), backward(12, 3000, 128))
    assert two <= 0.9 * twelve


def test_backward_with_a_tile_for_every_sm():
    """128 tiles take little longer than 64, each an SM of its own (1.11 times where they share the SMs that are left first)."""
    half, whole = microseconds(backward(8, 1024, 128), backward(16, 1024, 128))
    assert whole <= 1.075 * half


def test_heads_after_a_wave():
    """49 heads after a wave of 148 take no longer than 74 (1.04 of it in segments, with five chunks)."""
    fewer, more = microseconds(prefill(197, 640, 16, 64), prefill(222, 640, 16, 64))
    assert fewer <= 1.02 * more
