"""The gated convolution over a sequence at the edges of its blocks: 2, 4 and 8 tokens per thread with a remainder, part of a block
of 512 channels, every width, and more blocks of tokens than a grid has rows."""
import pytest
import torch

import paper_2402_18668_b200 as based

pytestmark = pytest.mark.gpu


def _want(a, g, h, b2):
    a, g, h, b2 = (t.double() for t in (a, g, h, b2))
    x = b2 + h[0] * g
    for j in range(1, h.shape[0]):
        x[:, j:] += h[j] * g[:, :-j]
    return a * x * torch.sigmoid(x)


@pytest.mark.parametrize("width", [1, 2, 3, 4])
@pytest.mark.parametrize("dtype,B,N,C", [
    (torch.bfloat16, 1, 1, 8), (torch.bfloat16, 2, 3, 520), (torch.float32, 2, 3, 520), (torch.bfloat16, 3, 1023, 1544),
    (torch.float32, 3, 1023, 1544), (torch.bfloat16, 8, 6147, 1000), (torch.float32, 1, 4099, 2056), (torch.bfloat16, 1, 131075, 8)])
def test_blocks_of_tokens(dtype, B, N, C, width):
    gen = torch.Generator(device="cuda").manual_seed(N + width)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    a, g, h, b2 = rnd(B, N, C).to(dtype), rnd(B, N, C).to(dtype), rnd(width, C) * 0.5, rnd(C)
    out = based.baseconv_gate_forward(a, g, h, b2)
    want = _want(a, g, h, b2)
    # bf16: one rounding of the result (2^-9); fp32: a few of 2^-24 in the sum and in the sigmoid
    rtol = 2.0 ** -8 if dtype == torch.bfloat16 else 2.0 ** -20
    assert torch.allclose(out.double(), want, rtol=rtol, atol=2.0 ** -20)
    assert torch.equal(based.baseconv_gate_forward(a, g, h, b2, out=a), out)          # in place of a
    assert based.based_poll_error() == based.BASED_OK


def test_values_that_are_not_finite():
    """Each element by itself: NaN where the filter meets an infinity of both signs or the gate is -inf, else as the formula says."""
    N, C = 40, 512
    gen = torch.Generator(device="cuda").manual_seed(3)
    a, g = (torch.randn(1, N, C, generator=gen, device="cuda").bfloat16() for _ in range(2))
    h, b2 = torch.randn(3, C, generator=gen, device="cuda"), torch.zeros(C, device="cuda")
    g[0, 5, ::7] = float("inf"); g[0, 20, ::5] = float("-inf"); a[0, 30, ::3] = float("nan"); g[0, 35, ::11] = 1e37
    out, want = based.baseconv_gate_forward(a, g, h, b2), _want(a, g, h, b2)
    finite = torch.isfinite(want) & (want.abs() < 1e38)
    assert torch.isfinite(out[finite]).all() and torch.allclose(out[finite].double(), want[finite], rtol=2.0 ** -7, atol=2.0 ** -20)
    assert (torch.isnan(out) == torch.isnan(want)).all()


def test_behind_a_kernel_that_leaves_the_sm_to_shared_memory():
    """The loads in flight need L1, which the kernel asks for: behind the sliding window, whose CTAs take an SM's shared memory, the
    convolution takes its own time, not the 1.5 to 1.7 times that it takes on what such a kernel leaves."""
    gen = torch.Generator(device="cuda").manual_seed(9)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    a, g, h, b2 = rnd(8, 1024, 8192).bfloat16(), rnd(8, 1024, 8192).bfloat16(), rnd(3, 8192), rnd(8192)
    qw, kw, vw = (rnd(4, 16, 2048, 64).bfloat16() for _ in range(3))
    out, out_w = torch.empty_like(a), torch.empty_like(vw)

    def conv():
        based.baseconv_gate_forward(a, g, h, b2, out=out)

    def window():
        based.swa_forward(qw, kw, vw, out=out_w, window=64)

    def both():
        window()
        conv()

    def replays(step):
        step()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for _ in range(20):
                step()
        return graph

    graphs = {f: replays(f) for f in (conv, window, both)}
    best = dict.fromkeys(graphs, float("inf"))
    for _ in range(10):
        for f, graph in graphs.items():
            start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            start.record()
            graph.replay()
            end.record()
            end.synchronize()
            best[f] = min(best[f], start.elapsed_time(end))
    assert best[both] - best[window] <= 1.25 * best[conv], best
