"""Feature dimensions other than 16, bf16: outputs and state come from two kernels that run side by side.  What follows in
the stream has to see both complete, call after call; rows (m, n) and (n, m) of the state are stored from one sum."""
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import workloads as wl
from parity import TOL_BF16, assert_state_close, row_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_feat,d_v", [(8, 64), (24, 64), (24, 112), (32, 128), (32, 64), (8, 128)])
@pytest.mark.parametrize("BH,L", [(1, 1), (3, 64), (2, 129), (5, 300), (200, 193), (64, 1500)])
def test_outputs_and_state_side_by_side(d_feat, d_v, BH, L):
    w = wl.Workload("beside", 1, BH, L, d_feat, d_v, "bf16", 0.5, decode_steps=1)
    gen = wl.generator(BH * 100 + L + d_feat)
    q, k, v = (t.cuda() for t in wl.prefill_inputs(w, gen))
    qs, ks, vs = (t[0].cuda() for t in wl.decode_inputs(w, gen))
    heads = sorted({0, BH - 1})
    y, S, z_ref = oracle.linattn_quadratic(*(wl.to_f64(t[:, heads]) for t in (q, k, v)))
    first = None
    for rep in range(20):
        kv, z = based.new_state(1, BH, d_v, d_feat=d_feat)
        kv.fill_(float("nan")); z.fill_(float("nan"))
        out = based.based_prefill(q, k, v, kv_state=kv, z_state=z)
        before = kv.clone(), z.clone()                      # next in the stream
        token = based.based_decode_step(qs, ks, vs, kv, z)
        got = [out, *before, token, kv, z]
        if first is None:
            first = got
            assert row_err(wl.to_f64(out[:, heads]), y) <= TOL_BF16
            assert_state_close(wl.to_f64(before[0][:, heads]), S, wl.to_f64(before[1][:, heads]), z_ref, "bf16")
            pairs = before[0][:, :, 1 + d_feat:].view(1, BH, d_feat, d_feat, d_v)
            assert torch.equal(pairs, pairs.transpose(2, 3))
        assert all(torch.equal(a, b) for a, b in zip(got, first)), rep
    assert torch.equal(based.based_prefill(q, k, v), first[0])
    assert based.based_poll_error() == based.BASED_OK
