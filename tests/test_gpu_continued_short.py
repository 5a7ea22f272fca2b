"""Continued bf16 calls that read the caller's state themselves (one piece per head, and the recompute mode's pieces): all
ten feature blocks in both formats, lengths around a chunk, widths with idle lanes, outputs and states against the oracle."""
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import workloads as wl
from parity import TOL_BF16, assert_state_close, row_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("d_v", [64, 112, 128])
@pytest.mark.parametrize("BH,L", [(1, 1), (3, 128), (2, 129), (32, 777), (150, 200), (5, 700)])
def test_continued_from_the_callers_state(BH, L, d_v, sym):
    L0 = 50
    w = wl.Workload("cont", 1, BH, L0 + L, 16, d_v, "bf16", 0.7)
    q, k, v = wl.prefill_inputs(w, wl.generator(BH * 7 + L + d_v))
    heads = sorted({0, BH // 2, BH - 1})
    f64 = lambda t: wl.to_f64(t[:, heads])
    _, S0, z0 = oracle.linattn_recurrent(*(wl.to_f64(t[:, :, :L0]) for t in (q, k, v)))
    y, S, z_ref = oracle.linattn_recurrent(f64(q), f64(k), f64(v))
    kv, z = torch.from_numpy(S0).float().cuda(), torch.from_numpy(z0).float().cuda()
    if sym:
        kv, z = based.based_state_to_sym(kv, z)
    out = based.based_prefill(*(t[:, :, L0:].contiguous().cuda() for t in (q, k, v)), kv_state=kv, z_state=z,
                              flags=based.BASED_STATE_CONTINUE | (based.BASED_STATE_SYM if sym else 0))
    assert based.based_poll_error() == based.BASED_OK
    if sym:
        kv, z = based.based_state_from_sym(kv, z)
    assert row_err(wl.to_f64(out[:, heads]), y[:, :, L0:]) <= TOL_BF16
    assert_state_close(wl.to_f64(kv[:, heads]), S, wl.to_f64(z[:, heads]), z_ref, "bf16")


def _call(q, k, v, kv, z, flags, workspace):
    """based_prefill through the C ABI, on a workspace of the caller's (or none)."""
    out = torch.empty_like(v)
    p = lambda t: None if t is None else t.data_ptr()
    st = based.lib().based_prefill(p(q), p(k), p(v), p(out), p(kv), p(z), *q.shape[:3], 16, v.shape[-1], based.BASED_BF16, flags,
                                   p(workspace), 0 if workspace is None else workspace.nbytes, torch.cuda.current_stream().cuda_stream)
    assert st == based.BASED_OK
    return out


@pytest.mark.parametrize("B,H,L,d_v", [(3, 16, 777, 112), (1, 18, 1000, 64), (1, 2, 900, 128)])
def test_pieces_read_the_state_before_it_is_overwritten(B, H, L, d_v):
    """Many continued calls one after the other while another stream keeps taking SMs, on a workspace that holds anything, and
    replayed as a graph: bit for bit the call on its own.  Without a workspace: the same up to rounding."""
    w = wl.Workload("cont", B, H, L, 16, d_v, "bf16", 0.5)
    q, k, v = (t.cuda() for t in wl.prefill_inputs(w, wl.generator(L)))
    g = torch.Generator().manual_seed(1)
    kv0, z0 = torch.randn(B, H, 273, d_v, generator=g).cuda(), torch.rand(B, H, 273, generator=g).cuda()
    z0[:, :, 0] += 100.0
    kv, z = kv0.clone(), z0.clone()
    want = (_call(q, k, v, kv, z, 1, torch.zeros(2048, dtype=torch.uint8, device="cuda")), kv.clone(), z.clone())
    other = torch.cuda.Stream()
    dq, dv = torch.randn(1, 300, 16, device="cuda").bfloat16(), torch.randn(1, 300, 128, device="cuda").bfloat16()
    state = based.new_state(1, 300, 128)
    ws = torch.randint(0, 256, (2048,), dtype=torch.uint8, device="cuda")
    bad = torch.zeros((), dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    for _ in range(100):
        with torch.cuda.stream(other):
            for _ in range(3):
                based.based_decode_step(dq, dq, dv, *state)
        kv.copy_(kv0); z.copy_(z0)
        out = _call(q, k, v, kv, z, 1, ws)
        for a, b in zip((out, kv, z), want):
            bad += (a != b).sum()
    assert int(bad) == 0
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = _call(q, k, v, kv, z, 1, ws)
    for _ in range(20):
        kv.copy_(kv0); z.copy_(z0)
        graph.replay()
        for a, b in zip((out, kv, z), want):
            bad += (a != b).sum()
    assert int(bad) == 0
    kv.copy_(kv0); z.copy_(z0)
    out = _call(q, k, v, kv, z, 1, None)
    assert row_err(wl.to_f64(out), wl.to_f64(want[0])) <= TOL_BF16
    assert_state_close(wl.to_f64(kv), wl.to_f64(want[1]), wl.to_f64(z), wl.to_f64(want[2]), "bf16")
    assert based.based_poll_error() == based.BASED_OK
