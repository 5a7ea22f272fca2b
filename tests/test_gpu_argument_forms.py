"""Forms in which the one-token steps and the convolution take their arguments besides the plain one: the same result."""
import pytest
import torch

import paper_2402_18668_b200 as based

pytestmark = pytest.mark.gpu


def _rnd(seed, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda").to(dtype)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("view", [lambda t: t[:, :, None], lambda t: t.view(-1, t.shape[-1]), lambda t: t.view(-1)])
def test_views_of_a_window_step(dtype, view):
    q, k, v = (_rnd(i, 2, 3, 64, dtype=dtype) for i in range(3))
    caches = [_rnd(3 + i, 2, 3, 16, 64, dtype=dtype) for i in range(2)]
    plain = [c.clone() for c in caches]
    want = based.swa_decode_step(q, k, v, *plain, 5)
    out = torch.empty_like(view(q))
    based.swa_decode_step(q, view(k), view(v), *caches, 5, out=out)
    assert torch.equal(out.view(want.shape), want)
    for a, b in zip(caches, plain):
        assert torch.equal(a, b)
    with pytest.raises(ValueError):
        based.swa_decode_step(q, k[:1], v, *caches, 5)
    with pytest.raises(ValueError):
        based.swa_decode_step(q, k, v, *caches, 5, out=out[:1])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("step", [True, False])
def test_views_of_a_convolution(dtype, step):
    shape = (3, 64) if step else (3, 9, 64)
    a, g, h, b2 = _rnd(0, *shape, dtype=dtype), _rnd(1, *shape, dtype=dtype), _rnd(2, 3, 64), _rnd(3, 64)
    state = _rnd(4, 3, 2, 64, dtype=dtype)

    def call(g, h, b2, out=None):
        s = state.clone()
        r = based.baseconv_gate_step(a, g, h, b2, s, out=out) if step else based.baseconv_gate_forward(a, g, h, b2, out=out)
        return r.view(shape), s
    want = call(g, h, b2)
    forms = [dict(out=torch.empty(a.numel(), dtype=dtype, device="cuda")), dict(h=h[:, :, None])]
    if step:
        forms += [dict(g=g[:, None]), dict(b2=b2[None]), dict(h=h[:, None])]
    for form in forms:
        for x, y in zip(call(**{"g": g, "h": h, "b2": b2, **form}), want):
            assert torch.equal(x, y)
    for bad in (dict(g=g[:2]), dict(h=h[:, :32].contiguous()), dict(b2=b2[:32]), dict(out=torch.empty(a.numel() - 1, dtype=dtype, device="cuda"))):
        with pytest.raises(ValueError):
            call(**{"g": g, "h": h, "b2": b2, **bad})


def test_numbers_of_other_types():
    """Windows, positions, scales and flags that int() and float() take."""
    q = _rnd(0, 1, 2, 70, 64)
    want = based.swa_forward(q, q, q, window=16, softmax_scale=0.5)
    for window, scale in ((16.0, "0.5"), ("16", torch.tensor(0.5))):
        assert torch.equal(based.swa_forward(q, q, q, window=window, softmax_scale=scale), want)
    q1, k, v = _rnd(1, 1, 2, 64), _rnd(2, 1, 2, 16, 64), _rnd(3, 1, 2, 16, 64)
    pos = torch.tensor([5], dtype=torch.int32, device="cuda")
    for f, p in ((based.swa_decode_step, 5.0), (based.swa_decode_step_ragged, pos)):
        assert torch.equal(f(q1, q1, q1, k.clone(), v.clone(), p, softmax_scale="0.5"),
                           f(q1, q1, q1, k.clone(), v.clone(), 5 if f is based.swa_decode_step else pos, softmax_scale=0.5))
    x, y = _rnd(4, 1, 2, 30, 16), _rnd(5, 1, 2, 30, 64)
    for a, b in zip(based.based_prefill_backward(x, x, y, y, flags=4.0), based.based_prefill_backward(x, x, y, y, flags=4)):
        assert torch.equal(a, b)
    x1, y1 = x[:, :, 0].contiguous(), y[:, :, 0].contiguous()
    states = [tuple(t + 1.0 for t in based.new_state(1, 2, 64)) for _ in range(2)]
    assert torch.equal(based.based_decode_step_flags(x1, x1, y1, *states[0], flags=4.0),
                       based.based_decode_step_flags(x1, x1, y1, *states[1], flags=4))
