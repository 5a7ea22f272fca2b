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
