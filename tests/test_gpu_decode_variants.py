"""The decode step's variants: numbers of heads on both sides of each rule (clusters of four and two CTAs per head, two and
four CTAs per SM, evict-first beyond L2), every value width and state format, against the oracle on sampled heads."""
import numpy as np
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import workloads as wl
from parity import assert_state_close, row_err, tol_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("dtype,d_v", [("f32", 64), ("bf16", 112), ("bf16", 128), ("f32", 128)])
@pytest.mark.parametrize("BH", [1, 37, 38, 74, 75, 296, 297, 592, 593, 1500])
def test_decode_variants(BH, dtype, d_v, sym):
    w = wl.Workload("dec", 1, BH, 20, 16, d_v, dtype, 0.5, decode_steps=2)
    gen = wl.generator(BH + d_v)
    q, k, v = wl.prefill_inputs(w, gen)
    qs, ks, vs = wl.decode_inputs(w, gen)
    heads = sorted({0, BH // 2, BH - 1})
    _, S, zz = oracle.linattn_recurrent(*(wl.to_f64(t) for t in (q, k, v)))
    kv, z = torch.from_numpy(S).float().cuda(), torch.from_numpy(zz).float().cuda()
    if sym:
        kv, z = based.based_state_to_sym(kv, z)
    step = based.based_decode_step_sym if sym else based.based_decode_step
    S, zz = S[:, heads], zz[:, heads]
    for t in range(2):
        out = step(qs[t].cuda(), ks[t].cuda(), vs[t].cuda(), kv, z)
        y, S, zz = oracle.decode_step(*(wl.to_f64(x[t][:, heads]) for x in (qs, ks, vs)), S, zz)
        assert row_err(wl.to_f64(out[:, heads]), y) <= tol_for(dtype)
    if sym:
        kv, z = based.based_state_from_sym(kv, z)
    # the fp32 state read back once folded and unfolded: 1e-6 of a row's largest entry per rounding, far below 1e-4
    assert_state_close(wl.to_f64(kv[:, heads]), S, wl.to_f64(z[:, heads]), zz, "f32" if dtype == "f32" else "bf16")
    assert np.isfinite(wl.to_f64(kv)).all()
