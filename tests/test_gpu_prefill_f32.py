"""fp32 prefill cut into cluster segments: lengths at the edges of its tiles (16, 32, 64 tokens) and segment counts from
one to sixteen per head, every value width, both state formats, from the empty state and continued."""
import numpy as np
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import workloads as wl
from parity import TOL_F32, assert_state_close, row_err

pytestmark = pytest.mark.gpu


# heads x length -> segments per head: 2 x 1..17 -> 1, 2 x 33..260 -> 2 to 16, 2 x 700 -> 16, 60 x 130 -> 1 or 2, 150 heads -> 1
@pytest.mark.parametrize("d_v", [64, 112, 128])
@pytest.mark.parametrize("BH,L", [(2, 1), (2, 16), (2, 17), (2, 33), (2, 64), (2, 65), (2, 127), (2, 260), (2, 700), (60, 130), (150, 70)])
def test_prefill_f32_segments(BH, L, d_v):
    w = wl.Workload("seg", 1, BH, 2 * L, 16, d_v, "f32", 1.0)
    q, k, v = wl.prefill_inputs(w, wl.generator(BH * 1000 + L + d_v))
    y_ref, S_ref, z_ref = oracle.linattn_recurrent(*(wl.to_f64(t) for t in (q, k, v)))
    _, S1, z1 = oracle.linattn_recurrent(*(wl.to_f64(t[:, :, :L]) for t in (q, k, v)))
    first, second = ([t[:, :, s].contiguous().cuda() for t in (q, k, v)] for s in (slice(0, L), slice(L, 2 * L)))
    full, sym = based.new_state(1, BH, d_v), based.new_state(1, BH, d_v, sym=True)
    for st, flag in ((full, 0), (sym, based.BASED_STATE_SYM)):
        for t in st:
            t.fill_(float("nan"))                       # the empty state must not read the buffers
        y1 = based.based_prefill(*first, kv_state=st[0], z_state=st[1], flags=flag)
        a = st if flag == 0 else based.based_state_from_sym(*st)
        assert_state_close(wl.to_f64(a[0]), S1, wl.to_f64(a[1]), z1, "f32")
        y2 = based.based_prefill(*second, kv_state=st[0], z_state=st[1], flags=flag | based.BASED_STATE_CONTINUE)
        a = st if flag == 0 else based.based_state_from_sym(*st)
        assert_state_close(wl.to_f64(a[0]), S_ref, wl.to_f64(a[1]), z_ref, "f32")
        assert row_err(wl.to_f64(torch.cat([y1, y2], dim=2)), y_ref) <= TOL_F32
    assert row_err(wl.to_f64(based.based_prefill(*first)), y_ref[:, :, :L]) <= TOL_F32      # no state asked for


# the definition form at the edges of its tiles (16 or 32 rows, groups of 32 keys, eight groups a CTA) and of its rule, and the
# chunked kernel on the other side of it: 2 x 2049, 16 x 900 (and continued 8 x 640, 60 x 128), 64 x 300
@pytest.mark.parametrize("BH,L,d_v", [(1, 2048, 64), (2, 257, 112), (3, 31, 64), (3, 32, 128), (5, 513, 64), (64, 33, 64), (64, 97, 64),
                                      (100, 16, 112), (2, 2049, 64), (16, 900, 64), (8, 640, 64), (60, 128, 64), (64, 300, 64)])
def test_prefill_f32_either_form(BH, L, d_v):
    test_prefill_f32_segments(BH, L, d_v)


def test_prefill_f32_keeps_an_uneven_full_state_apart():
    """Rows (m, n) and (n, m) of a caller's state that differ: outputs use their sum, and each keeps its own value plus
    the tokens' share."""
    B, H, L, d_v = 1, 2, 100, 64
    w = wl.Workload("uneven", B, H, L, 16, d_v, "f32", 1.0)
    q, k, v = wl.prefill_inputs(w, wl.generator(4))
    g = torch.Generator().manual_seed(5)
    kv0, z0 = torch.randn(B, H, 273, d_v, generator=g), torch.rand(B, H, 273, generator=g)
    z0[:, :, 0] += 50.0
    kv, z = kv0.cuda(), z0.cuda()
    based.based_prefill(q.cuda(), k.cuda(), v.cuda(), kv_state=kv, z_state=z, flags=based.BASED_STATE_CONTINUE)
    _, S, zz = oracle.linattn_recurrent(*(wl.to_f64(t) for t in (q, k, v)))
    # one rounding of a sum of magnitude |kv0| + |S| per element, and the sums' own: 1e-5 of the largest entry
    assert np.abs(wl.to_f64(kv) - (wl.to_f64(kv0) + S)).max() <= 1e-5 * np.abs(S).max()
    assert np.abs(wl.to_f64(z) - (wl.to_f64(z0) + zz)).max() <= 1e-5 * np.abs(zz).max()


@pytest.mark.parametrize("d_v,L", [(64, 1), (64, 200), (112, 3), (128, 70)])
def test_prefill_f32_adds_to_a_full_state(d_v, L):
    """A continued call adds to a full state: nothing added leaves it bit for bit (infinities too), and many short pieces
    leave no drift."""
    H = 2
    w = wl.Workload("add", 1, H, L, 16, d_v, "f32", 0.1)
    q, k, v = (t.cuda() for t in wl.prefill_inputs(w, wl.generator(d_v + L)))
    g = torch.Generator().manual_seed(5)
    kv, z = (torch.randn(1, H, *s, generator=g).cuda() for s in ((273, d_v), (273,)))
    z[:, :, 0] += 500.0
    kv[0, 1, 1 + 16 + 3 * 16 + 5, 7] = kv[0, 1, 1 + 16 + 5 * 16 + 3, 7] = float("inf")
    before = [t[:, :, 1:].clone() for t in (kv, z)]       # zero keys: only the constant's row grows
    based.based_prefill(q, torch.zeros_like(k), v, kv_state=kv, z_state=z, flags=based.BASED_STATE_CONTINUE)
    assert torch.equal(kv[:, :, 1:], before[0]) and torch.equal(z[:, :, 1:], before[1])
    kv = torch.randn(1, H, 273, d_v, generator=g).mul(1e3).cuda()
    z = torch.rand(1, H, 273, generator=g).cuda() * 1e3 + 1e4
    S = wl.to_f64(kv)
    _, dS, _ = oracle.linattn_recurrent(*(wl.to_f64(t) for t in (q, k, v)))
    n = 200
    for _ in range(n):
        based.based_prefill(q, k, v, kv_state=kv, z_state=z, flags=based.BASED_STATE_CONTINUE)
    # a few roundings of 2^-24 a call and entry, up or down by the entry: their median over thousands of entries stays within
    # a tenth of n 2^-24 (3.4e-8 lost on every call would be a half of it)
    pairs = [1 + 16 + 16 * m + c for m in range(16) for c in range(16) if c != m]
    err = ((wl.to_f64(kv) - (S + n * dS)) / np.abs(S + n * dS))[:, :, pairs]
    assert abs(np.median(err)) <= 0.1 * n * 2.0 ** -24


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("which", [0, 1, 2])
@pytest.mark.parametrize("BH,L,d_v", [(2, 200, 64), (150, 40, 112), (2, 13, 128)])
def test_prefill_f32_non_finite_tokens_stay_behind(BH, L, d_v, which, bad):
    """A non-finite q, k or v of one token (padding behind a prompt, for instance) leaves the rows before it as they are."""
    w = wl.Workload("bad", 1, BH, L, 16, d_v, "f32", 0.5)
    x = [t.cuda() for t in wl.prefill_inputs(w, wl.generator(L))]
    want = based.based_prefill(*x)
    for at in sorted({L // 2, L - 1, 5}):
        y = [t.clone() for t in x]
        y[which][:, :, at] = bad
        out = based.based_prefill(*y)
        # the same sums where no value is taken for infinite, in another grouping where one is
        assert torch.allclose(out[:, :, :at], want[:, :, :at], rtol=0, atol=TOL_F32 * 0.1)
        assert not torch.isfinite(out[:, :, at]).all()
        if which == 0:
            assert torch.isfinite(out[:, :, at + 1:]).all()
