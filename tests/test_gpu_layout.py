"""based_tokens_to_heads (bytes copied, so exact), the gradients that reach the library through it, and the convolution
step at batch sizes on both sides of its rows-per-thread rule."""
import ctypes

import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import binding as b
from paper_2402_18668_b200 import workloads as wl
from paper_2402_18668_b200.autograd import linear_attention
from parity import row_err, tol_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,H,row", [(1, 1, 1, 8), (2, 37, 3, 56), (3, 130, 5, 64), (2, 1000, 16, 128), (1, 4097, 2, 24)])
def test_tokens_to_heads(B, L, H, row):
    x = torch.randn(B, L, H, row, device="cuda").bfloat16()
    y = torch.full((B, H, L, row), float("nan"), dtype=x.dtype, device="cuda")
    st = b.lib().based_tokens_to_heads(ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr()), B, H, L, 2 * row, b._stream())
    assert st == 0 and torch.equal(y, x.transpose(1, 2))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("B,H,L,d_v", [(2, 3, 70, 112), (1, 2, 300, 64)])
def test_gradients_do_not_depend_on_the_layout_of_dout(dtype, B, H, L, d_v):
    g = torch.Generator(device="cuda").manual_seed(L)
    q, k = ((torch.randn(B, H, L, 16, generator=g, device="cuda") * 0.5).to(dtype).requires_grad_(True) for _ in range(2))
    v = torch.randn(B, H, L, d_v, generator=g, device="cuda").to(dtype).requires_grad_(True)
    dout = torch.randn(B, L, H, d_v, generator=g, device="cuda").to(dtype).transpose(1, 2)
    want = torch.autograd.grad(linear_attention(q, k, v), (q, k, v), dout.contiguous())
    got = torch.autograd.grad(linear_attention(q, k, v), (q, k, v), dout)
    assert all(torch.equal(a, c) for a, c in zip(got, want))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("width", [1, 2, 3, 4])
@pytest.mark.parametrize("B,C", [(1, 64), (5, 1032), (73, 8192), (74, 8192), (77, 8200)])
def test_convolution_step_rows_per_thread(dtype, width, B, C):
    gen = wl.generator(B + C + width)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    a, g = (torch.randn(B, C, generator=gen).to(dt) for _ in range(2))
    h, b2 = torch.randn(width, C, generator=gen), torch.randn(C, generator=gen)
    st = torch.randn(B, width - 1, C, generator=gen).to(dt)
    state = st.cuda()
    out = based.baseconv_gate_step(a.cuda(), g.cuda(), h.cuda(), b2.cuda(), state if width > 1 else None)
    f = lambda t: t.double()
    x = f(h[0]) * f(g) + f(b2) + sum(f(h[j]) * f(st[:, j - 1]) for j in range(1, width))
    want = f(a) * x / (1 + torch.exp(-x))
    assert row_err(wl.to_f64(out), want.numpy()) <= tol_for(dtype)
    assert torch.equal(state.cpu(), torch.cat([g[:, None], st], dim=1)[:, :width - 1])


@pytest.mark.parametrize("B,H,L,d_v", [(4, 16, 800, 64), (2, 8, 1100, 64), (4, 16, 1100, 128), (1, 8, 4200, 128), (2, 3, 129, 128),
                                       (3, 50, 200, 64), (2, 16, 1300, 112), (4, 16, 1100, 112), (2, 3, 129, 112), (2, 1, 64, 64)])
def test_gradients_of_dout_as_it_lies(B, H, L, d_v):
    """bf16, block by block (a CTA per head, sums of every block with few heads, blocks of 512) and by tiles."""
    g = torch.Generator(device="cuda").manual_seed(L)
    q, k = ((torch.randn(B, H, L, 16, generator=g, device="cuda") * 0.5).bfloat16().requires_grad_(True) for _ in range(2))
    v = torch.randn(B, H, L, d_v, generator=g, device="cuda").bfloat16().requires_grad_(True)
    dout = torch.randn(B, L, H, d_v, generator=g, device="cuda").bfloat16().transpose(1, 2)
    y = linear_attention(q, k, v)
    want = torch.autograd.grad(y, (q, k, v), dout.contiguous(), retain_graph=True)
    got = torch.autograd.grad(y, (q, k, v), dout)
    assert all(torch.equal(a, c) for a, c in zip(got, want))
    assert based.based_poll_error() == based.BASED_OK
