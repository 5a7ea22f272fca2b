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
