"""fp32 forward and backward on the tensor cores (operands in three bf16 parts): lengths at the edges of the own tiles (128)
and looped tiles (64), loops shared by one to eight CTAs, longest loops first and not, every value width, both forms."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
import paper_2402_18668_b200.autograd
from paper_2402_18668_b200 import workloads as wl
from parity import TOL_F32, row_err

pytestmark = pytest.mark.gpu

# Sums of up to a few hundred products, each good to 2^-24 of its size: 2^-24 sqrt(300) = 1e-6 of a head's largest entry, a few
# times that at the worst entry of thousands (fp32 multiply-adds pair by pair: 1 to 4e-6 on these)
TOL = 1e-5

# Relative to 64 bits in the 2-norm.  An operand's parts keep 24 bits and the products left out are below 2^-25 of it; with the
# sums' own rounding 1 to 3e-7 is measured, whatever the inputs' magnitude.  Two parts in place of three would show 4e-6.
TOL_NORM = 1e-6


def norm_err(got, want):
    return np.linalg.norm(wl.to_f64(got) - want) / np.linalg.norm(want)


def inputs(BH, L, d_v, seed):
    w = wl.Workload("parts", 1, BH, L, 16, d_v, "f32", 1.0)
    gen = wl.generator(seed)
    return (*wl.prefill_inputs(w, gen), torch.randn(1, BH, L, d_v, generator=gen))


def forward(q, k, v, flags=0, out=None):
    """based_prefill_f32_parts."""
    B, H, L, d_v = v.shape
    lib, p = based.binding.lib(), lambda t: ctypes.c_void_p(t.data_ptr())
    lib.based_f32_parts_bytes.restype = lib.based_prefill_workspace_bytes.restype
    n = lib.based_f32_parts_bytes(B, H, L, 16, d_v, 0)
    out, ws = torch.empty_like(v) if out is None else out, torch.empty(n, dtype=torch.uint8, device="cuda")
    lib.based_prefill_f32_parts.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_int] * 6 + [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p]
    st = lib.based_prefill_f32_parts(p(q), p(k), p(v), p(out), B, H, L, 16, d_v, flags, p(ws), n,
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == based.BASED_OK
    return out


@pytest.mark.parametrize("d_v", [64, 112, 128])
@pytest.mark.parametrize("BH,L", [(2, 33), (1, 64), (3, 65), (2, 127), (150, 128), (2, 129), (1, 193), (80, 200), (1, 513), (40, 500)])
@pytest.mark.parametrize("flags", [0, based.BASED_NUMERATOR_ONLY])
def test_f32_parts(BH, L, d_v, flags):
    q, k, v, g = inputs(BH, L, d_v, BH * 1000 + L + d_v)
    lib, heads = based.binding.lib(), sorted({0, BH // 2, BH - 1})
    x = [t.cuda() for t in (q, k, v, g)]
    s = [wl.to_f64(t[:, heads]) for t in (q, k, v, g)]
    before = based.launch_count()
    y = forward(*x[:3], flags)
    assert based.launch_count() - before == 2                    # parts, outputs
    assert torch.equal(based.autograd.linear_attention(*x[:3], numerator_only=bool(flags)), y)
    want, _, _ = oracle.linattn_quadratic(*s[:3])
    if flags:
        c = s[0] @ s[1].swapaxes(-1, -2)
        want = want * np.tril(1 + c / 4 + c * c / 32).sum(-1, keepdims=True)
    assert row_err(wl.to_f64(y[:, heads]), want) <= TOL_F32
    assert norm_err(y[:, heads], want) <= TOL_NORM
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    if d_v == 64:
        got = based.based_prefill_backward(*x, flags=flags)
        for a, b in zip(got, oracle.linattn_backward(*s, numerator_only=bool(flags))):
            assert norm_err(a[:, heads], b) <= TOL_NORM
        assert all(torch.equal(a, b) for a, b in zip(got, based.based_prefill_backward(*x, flags=flags)))
        # with the scratch of the call without parts
        n = lib.based_prefill_backward_workspace_bytes(1, BH, L, 64, 0)
        ws, old = torch.empty(n, dtype=torch.uint8, device="cuda"), [torch.empty_like(t) for t in x[:3]]
        assert lib.based_prefill_backward(*(p(t) for t in x), *(p(t) for t in old), 1, BH, L, 16, 64, 0, flags, p(ws), n, stream) == 0
        for a, b in zip(got, old):
            assert (a - b).abs().max() <= 2 * TOL * b.abs().max()
    assert based.based_poll_error() == based.BASED_OK


@pytest.mark.parametrize("d_v", [64, 128])
def test_f32_parts_outputs_on_sixteen_bytes(d_v):
    """Arrays that start on a 16-byte boundary only."""
    q, k, v, g = (t.cuda() for t in inputs(2, 150, d_v, 5))
    off = [torch.empty(t.numel() + 4, device="cuda")[4:].view(t.shape).copy_(t) for t in (q, k, v, g)]
    out = torch.empty(v.numel() + 4, device="cuda")[4:].view(v.shape)
    assert torch.equal(forward(*off[:3], out=out), forward(q, k, v))


@pytest.mark.parametrize("big", [1e30, 3.4e38])
@pytest.mark.parametrize("BH,L", [(2, 200), (150, 100)])
def test_f32_parts_of_large_values(BH, L, big):
    """Values whose first part is next to the largest bf16, or rounds past it, and their rows' neighbours."""
    q, k, v, g = (t.cuda() for t in inputs(BH, L, 64, 7))
    at = L // 2
    vb = v.clone()
    vb[:, :, at, 3] = big
    want = forward(q, k, v)
    out = forward(q, k, vb)
    assert torch.allclose(out[:, :, :at], want[:, :, :at], rtol=0, atol=1e-4)
    cols = [c for c in range(64) if c != 3]
    assert torch.allclose(out[..., cols], want[..., cols], rtol=0, atol=1e-4)
    # column 3 from the value on: one term is all of it; infinite only where the sum over D would overflow in fp32
    x = [wl.to_f64(t[:, :1]) for t in (q, k, vb)]
    c = x[0] @ x[1].swapaxes(-1, -2)
    weights = np.tril(1 + c / 4 + c * c / 32)
    num = (weights @ x[2])[0, 0, at:, 3]
    ref, got = num / weights.sum(-1)[0, 0, at:], wl.to_f64(out[:, :1])[0, 0, at:, 3]
    fits = np.abs(num) < 0.999 * np.finfo(np.float32).max
    assert fits.any() and (big > 1e38 or fits.all()) and (np.abs(got - ref)[fits] <= TOL * np.abs(ref)[fits]).all()


def test_f32_parts_slabs_of_heads():
    """More heads than the parts' scratch holds at a time, the output gradient as it lies and not: heads of both slabs and
    their seam against the same heads alone."""
    B, H, L = 2, 150, 1000
    assert 2 * L * (2 * 96 + 2 * 384) * B * H // 2 > 256 << 20
    g = torch.Generator(device="cuda").manual_seed(3)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    q, k, v, dout = r(B, H, L, 16), r(B, H, L, 16), r(B, H, L, 64), r(B, L, H, 64)
    x = [t.requires_grad_(True) for t in (q, k, v)]
    y = based.autograd.linear_attention(*x)
    got = torch.autograd.grad(y, x, dout.transpose(1, 2), retain_graph=True)
    again = torch.autograd.grad(y, x, dout.transpose(1, 2).contiguous())
    assert all(torch.equal(a, b) for a, b in zip(got, again))
    y = y.detach().view(1, B * H, L, 64)
    flat = [t.detach().reshape(1, B * H, L, -1) for t in (q, k, v, dout.transpose(1, 2))]
    for h in (0, 149, 278, 279, 280, 299):
        one = [t[:, h:h + 1].contiguous() for t in flat]
        want = forward(*one[:3])
        assert norm_err(y[:, h:h + 1], wl.to_f64(want)) <= 2 * TOL_NORM
        for a, b in zip(got, based.based_prefill_backward(*one)):
            assert norm_err(a.reshape(1, B * H, L, -1)[:, h:h + 1], wl.to_f64(b)) <= 2 * TOL_NORM
    assert based.based_poll_error() == based.BASED_OK


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("which", [0, 1, 2])
@pytest.mark.parametrize("BH,L,d_v", [(2, 200, 64), (150, 40, 112), (2, 70, 128)])
def test_f32_parts_non_finite_tokens_stay_behind(BH, L, d_v, which, bad):
    """A non-finite q, k or v of one token leaves the rows before it as they are, and the others are non-finite where based_prefill's
    are."""
    x = [t.cuda() for t in inputs(BH, L, d_v, L)[:3]]
    want = forward(*x)
    for at in sorted({L // 2, L - 1, 5}):
        y = [t.clone() for t in x]
        y[which][:, :, at, 1] = bad
        out, ref = forward(*y), based.based_prefill(*y)
        assert torch.allclose(out[:, :, :at], want[:, :, :at], rtol=0, atol=TOL_F32 * 0.1)
        assert torch.equal(torch.isfinite(out), torch.isfinite(ref))
        ok = torch.isfinite(ref)
        assert torch.allclose(out[ok], ref[ok], rtol=1e-5, atol=1e-4)


@pytest.mark.parametrize("scale", [1e-30, 1e-36])
@pytest.mark.parametrize("small", ["v", "dout", "q", "k"])
@pytest.mark.parametrize("BH,L", [(2, 64), (3, 300), (150, 129)])
def test_f32_parts_of_small_values(BH, L, small, scale):
    """Parts of such values would be bf16 subnormals, or nothing, if the values were split as they are."""
    x = dict(zip(("q", "k", "v", "dout"), inputs(BH, L, 64, L)))
    x[small] *= scale
    heads = sorted({0, BH // 2, BH - 1})
    s = [wl.to_f64(t[:, heads]) for t in x.values()]
    d = [t.cuda() for t in x.values()]
    assert norm_err(forward(*d[:3])[:, heads], oracle.linattn_quadratic(*s[:3])[0]) <= TOL_NORM
    for flags in (0, based.BASED_NUMERATOR_ONLY):
        for a, b in zip(based.based_prefill_backward(*d, flags=flags), oracle.linattn_backward(*s, numerator_only=bool(flags))):
            assert norm_err(a[:, heads], b) <= TOL_NORM
    assert based.based_poll_error() == based.BASED_OK


def test_a_workspace_of_the_documented_size_is_used():
    """Nothing but the gradients is allocated beside it; the route follows its size."""
    x = [t.cuda() for t in inputs(4, 300, 64, 11)]
    q, v = x[0], x[2]
    small, large = (torch.empty(n, dtype=torch.uint8, device="cuda") for n in
                    (based.based_prefill_backward_workspace_bytes(1, 4, 300, 64, 0), based.based_f32_parts_bytes(1, 4, 300, 16, 64, True)))
    assert small.nbytes < large.nbytes

    def call(workspace):
        torch.cuda.synchronize()
        torch.cuda.reset_peak_memory_stats()
        before, launched = torch.cuda.memory_allocated(), based.launch_count()
        g = based.based_prefill_backward(*x, workspace=workspace)
        return g, torch.cuda.max_memory_allocated() - before - 2 * q.nbytes - v.nbytes, based.launch_count() - launched
    (g_small, extra, launched), (g_large, extra_l, launched_l) = call(small), call(large)
    assert extra <= 3 * 512 and launched == 2 and extra_l <= 3 * 512 and launched_l == 3
    g_none, extra, _ = call(None)
    assert extra >= large.nbytes and all(torch.equal(a, b) for a, b in zip(g_none, g_large))
    for a, b in zip(g_small, g_large):
        assert norm_err(a, wl.to_f64(b)) <= 2 * TOL_NORM


def test_f32_parts_without_room_for_the_scratch():
    """A device with room for the results but not for the scratch: the routes that need none, as where the scratch is refused."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()                                      # (no large block that what follows would be cut from)
    x = [t.cuda() for t in inputs(100, 2000, 64, 13)]
    q, k, v, g = x
    lies = g.transpose(1, 2).contiguous().transpose(1, 2)         # the heads of a token side by side
    documented = torch.empty(based.based_prefill_backward_workspace_bytes(1, 100, 2000, 64, 0), dtype=torch.uint8, device="cuda")
    want_y = based.based_prefill(q, k, v)
    want = based.based_prefill_backward(*x, workspace=documented)
    leaves = [t.requires_grad_(True) for t in (q, k, v)]
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    # the results take 51 MB (forward) and 77 MB (backward, with a copy of dout 128 MB); the scratch 115 and 192 MB
    for room, call in [(96 << 20, lambda: [based.autograd.linear_attention(q, k, v).detach()]),
                       (176 << 20, lambda: based.based_prefill_backward(*(t.detach() for t in x)))]:
        torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + room) / total)
        try:
            got = call()
        finally:
            torch.cuda.set_per_process_memory_fraction(1.0)
        assert all(torch.equal(a, b) for a, b in zip(got, [want_y] if len(got) == 1 else want))
        del got
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
    y = based.autograd.linear_attention(*leaves)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (176 << 20)) / total)
    try:
        got = torch.autograd.grad(y, leaves, lies)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("which", range(4))
@pytest.mark.parametrize("BH,L", [(1, 64), (3, 300), (1, 1000), (150, 70)])
@pytest.mark.parametrize("flags", [0, based.BASED_NUMERATOR_ONLY])
def test_f32_parts_gradients_of_non_finite_tokens(BH, L, which, bad, flags):
    """A non-finite q, k, v or dout of one token: the gradients that it does not enter are those without it, whichever way dout lies."""
    assert based.based_f32_parts_bytes(1, BH, L, 16, 64, True) > 0
    x = [t.cuda() for t in inputs(BH, L, 64, L)]
    want = based.based_prefill_backward(*x, flags=flags)
    at = torch.arange(L, device="cuda")
    for t in sorted({L // 2, L - 1, 5}):
        before, behind, others, none = at < t, at > t, at != t, at < 0
        # rows of dq, dk, dv.  A query's statistics carry a bad k or v to every key at or before it, unless there are none (numerator)
        clean = [(others, behind, behind),
                 (before, others, others) if flags else (before, none, none),
                 (before, others, at >= 0) if flags else (before, none, at >= 0),
                 (others, behind, behind)][which]
        y = [u.clone() for u in x]
        y[which][:, :, t, 1] = bad
        leaves = [u.clone().requires_grad_(True) for u in y[:3]]
        lies = y[3].transpose(1, 2).contiguous().transpose(1, 2)
        for got in (based.based_prefill_backward(*y, flags=flags),
                    torch.autograd.grad(based.autograd.linear_attention(*leaves, numerator_only=bool(flags)), leaves, lies)):
            for a, b, rows in zip(got, want, clean):
                if rows.any():
                    assert norm_err(a[:, :, rows], wl.to_f64(b[:, :, rows])) <= 2 * TOL_NORM
    assert based.based_poll_error() == based.BASED_OK
