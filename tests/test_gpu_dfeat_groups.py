"""Definition-form forward of d' 8, 24 and 32 with two row groups per CTA: lengths at the edges of the query tiles (128) and
key tiles (64), fewer key tiles than sets of scores, loops that wrap them, every value width, both forms, with the state and
without."""
import numpy as np
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import workloads as wl
from parity import TOL_BF16, assert_state_close, row_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,d_v", [(8, 64), (24, 64), (32, 112), (24, 128)])
@pytest.mark.parametrize("BH,L", [(2, 1), (1, 64), (2, 65), (2, 129), (1, 192), (3, 257), (1, 700), (150, 130), (40, 300)])
@pytest.mark.parametrize("flags", [0, based.BASED_NUMERATOR_ONLY])
def test_forward_groups(d, d_v, BH, L, flags):
    w = wl.Workload("groups", 1, BH, L, d, d_v, "bf16", 0.5)
    q, k, v = wl.prefill_inputs(w, wl.generator(BH * 1000 + L + d))
    heads = sorted({0, BH // 2, BH - 1})
    s = [wl.to_f64(t[:, heads]) for t in (q, k, v)]
    y_ref, S_ref, z_ref = oracle.linattn_quadratic(*s)
    if flags:
        c = s[0] @ s[1].swapaxes(-1, -2)
        y_ref = y_ref * np.tril(1 + c / d ** 0.5 + c * c / (2 * d)).sum(-1, keepdims=True)
    x = [t.cuda() for t in (q, k, v)]
    y = based.based_prefill(*x, flags=flags)
    assert row_err(wl.to_f64(y[:, heads]), y_ref) <= TOL_BF16
    kv, z = based.new_state(1, BH, d_v, d_feat=d)
    assert torch.equal(based.based_prefill(*x, kv_state=kv, z_state=z, flags=flags), y)
    assert_state_close(wl.to_f64(kv[:, heads]), S_ref, wl.to_f64(z[:, heads]), z_ref, "bf16")
    assert based.based_poll_error() == based.BASED_OK
