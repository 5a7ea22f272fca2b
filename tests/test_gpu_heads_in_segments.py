"""bf16 prefill with a few heads more than whole waves of one CTA per SM: those run in a launch of their own, cut into segments.
Every head's outputs and state, on both sides of the cut and of the rule's lines, in both state formats, and what follows a slot
left as it was."""
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import workloads as wl
from parity import TOL_BF16, assert_state_close, row_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_v,BH,L", [(64, 149, 129), (64, 222, 300), (64, 223, 300), (128, 150, 512), (112, 160, 513), (64, 197, 1000),
                                      (64, 198, 1000), (112, 149, 2047), (64, 296, 2048), (64, 298, 1921), (128, 157, 128)])
@pytest.mark.parametrize("state", ["none", "full", "sym"])
def test_heads_after_whole_waves(d_v, BH, L, state):
    w = wl.Workload("waves", 1, BH, L, 16, d_v, "bf16", 0.5)
    q, k, v = wl.prefill_inputs(w, wl.generator(BH + L + d_v))
    x = [t.cuda() for t in (q, k, v)]
    flags = based.BASED_STATE_SYM if state == "sym" else 0
    if state == "none":
        y = based.based_prefill(*x)
    else:
        kv, z = based.new_state(1, BH, d_v, sym=state == "sym")
        kv.fill_(float("nan")); z.fill_(float("nan"))
        y = based.based_prefill(*x, kv_state=kv, z_state=z, flags=flags)
        assert torch.isfinite(kv).all() and torch.isfinite(z).all()
    heads = sorted({0, 147, 148, BH - BH % 148 - 1, min(BH - BH % 148, BH - 1), BH - 1})
    y_ref, S, z_ref = oracle.linattn_quadratic(*(wl.to_f64(t[:, heads]) for t in (q, k, v)))
    assert row_err(wl.to_f64(y[:, heads]), y_ref) <= TOL_BF16
    if state == "full":
        assert_state_close(wl.to_f64(kv[:, heads]), S, wl.to_f64(z[:, heads]), z_ref, "bf16")
    if state == "sym":
        kv2, z2 = based.new_state(1, BH, d_v)
        assert torch.equal(based.based_prefill(*x, kv_state=kv2, z_state=z2), y)
        assert_state_close(wl.to_f64(kv2[:, heads]), S, wl.to_f64(z2[:, heads]), z_ref, "bf16")
        kf, zf = based.based_state_from_sym(kv, z)
        assert_state_close(wl.to_f64(kf[:, heads]), S, wl.to_f64(zf[:, heads]), z_ref, "bf16")
    # the rest of the heads against calls of fewer heads, which take another plan
    for s in (slice(0, 100), slice(100, BH)):
        part = based.based_prefill(*(t[:, s].contiguous() for t in x))
        assert row_err(wl.to_f64(y[:, s]), wl.to_f64(part)) <= TOL_BF16
    assert based.based_poll_error() == based.BASED_OK
