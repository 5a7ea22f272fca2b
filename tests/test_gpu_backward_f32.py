"""fp32 backward on 64 x 64 tiles: lengths at the tile edges, own tiles shared by one to eight CTAs of a cluster (few
heads) and not shared (many), every value width, both forms."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import workloads as wl
from parity import TOL_F32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_v,BH,L", [(64, 1, 63), (64, 2, 65), (64, 2, 128), (112, 3, 129), (128, 2, 257), (64, 1, 700),
                                      (64, 150, 130), (128, 80, 200), (64, 32, 513), (128, 74, 256),
                                      (64, 75, 256)])
@pytest.mark.parametrize("flags", [0, based.BASED_NUMERATOR_ONLY])
def test_backward_f32_tiles(d_v, BH, L, flags):
    w = wl.Workload("bwd32", 1, BH, L, 16, d_v, "f32", 1.0)
    gen = wl.generator(BH * 1000 + L + d_v)
    q, k, v = wl.prefill_inputs(w, gen)
    g = torch.randn(1, BH, L, d_v, generator=gen)
    heads = sorted({0, BH // 2, BH - 1})
    want = oracle.linattn_backward(*(wl.to_f64(t[:, heads]) for t in (q, k, v, g)), numerator_only=bool(flags))
    got = based.based_prefill_backward(q.cuda(), k.cuda(), v.cuda(), g.cuda(), flags=flags)
    assert based.based_poll_error() == based.BASED_OK
    for a, b in zip(got, want):
        a = wl.to_f64(a[:, heads])
        assert np.isfinite(a).all()
        assert (np.abs(a - b).max(axis=(0, 2, 3)) <= TOL_F32 * np.abs(b).max(axis=(0, 2, 3))).all()
    again = based.based_prefill_backward(q.cuda(), k.cuda(), v.cuda(), g.cuda(), flags=flags)
    assert all(torch.equal(a, b) for a, b in zip(got, again))


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("L,at", [(200, 100), (64, 62), (300, 129)])
def test_backward_non_finite_values_stay_where_they_belong(L, at, bad):
    """A non-finite v leaves dq of the rows before it as it is (fp32), a non-finite output gradient dk of the keys behind it
    (both types)."""
    w = wl.Workload("bad", 1, 3, L, 16, 64, "f32", 0.5)
    gen = wl.generator(L)
    q, k, v = (t.cuda() for t in wl.prefill_inputs(w, gen))
    g = torch.randn(1, 3, L, 64, generator=gen).cuda()
    want = based.based_prefill_backward(q, k, v, g)
    vb, gb = v.clone(), g.clone()
    vb[:, :, at], gb[:, :, at] = bad, bad
    assert torch.equal(based.based_prefill_backward(q, k, vb, g)[0][:, :, :at], want[0][:, :, :at])
    got = based.based_prefill_backward(q, k, v, gb)
    assert torch.equal(got[1][:, :, at + 1:], want[1][:, :, at + 1:]) and not torch.isfinite(got[1][:, :, 0]).all()
    q, k, v, g, gb = (t.bfloat16() for t in (q, k, v, g, gb))
    for out in (None, based.based_prefill(q, k, v)):
        want = based.based_prefill_backward(q, k, v, g, out=out)
        got = based.based_prefill_backward(q, k, v, gb, out=out)
        assert torch.equal(got[1][:, :, at + 1:], want[1][:, :, at + 1:])


@pytest.mark.parametrize("B,H,L,d_v", [(2, 3, 65, 128), (1, 5, 257, 112), (3, 30, 40, 64), (2, 4, 200, 64), (1, 2, 1, 112), (5, 9, 130, 128)])
@pytest.mark.parametrize("flags", [0, based.BASED_NUMERATOR_ONLY])
def test_backward_f32_reads_dout_as_a_projection_leaves_it(B, H, L, d_v, flags):
    """[B,L,H,d_v], on fp32 multiply-adds: the gradients of the copy [B,H,L,d_v], bit for bit."""
    g = torch.Generator(device="cuda").manual_seed(L)
    q, k, v, dout = (torch.randn(B, H, L, d, generator=g, device="cuda") for d in (16, 16, d_v, d_v))
    n = based.based_prefill_backward_workspace_bytes(B, H, L, d_v, based.BASED_F32)
    ws, got = torch.empty(n, dtype=torch.uint8, device="cuda"), [torch.empty_like(t) for t in (q, k, v)]
    as_it_lies = dout.transpose(1, 2).contiguous()
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    st = based.lib().based_prefill_backward_tokens_first(p(q), p(k), p(v), p(as_it_lies), *map(p, got), B, H, L, 16, d_v, based.BASED_F32,
                                                         flags, p(ws), n, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == based.BASED_OK
    assert all(torch.equal(a, b) for a, b in zip(got, based.based_prefill_backward(q, k, v, dout, flags=flags, workspace=ws)))
