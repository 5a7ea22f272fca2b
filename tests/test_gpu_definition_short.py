"""bf16 calls of one chunk without a state take the definition form's kernels at d' 16 as well: lengths at the edges of the key
tiles (64) and of the chunk (128; 129 is the chunked kernel's), with heads that fill the chip once and more, both forms; and the
lines between those kernels at other d', where the number of tiles and the length decide."""
import numpy as np
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import workloads as wl
from parity import TOL_BF16, assert_state_close, row_err

pytestmark = pytest.mark.gpu


def case(d, d_v, BH, L):
    w = wl.Workload("short", 1, BH, L, d, d_v, "bf16", 0.5)
    q, k, v = wl.prefill_inputs(w, wl.generator(BH * 1000 + L + d))
    heads = sorted({0, BH // 2, BH - 1})
    return [t.cuda() for t in (q, k, v)], heads, [wl.to_f64(t[:, heads]) for t in (q, k, v)]


@pytest.mark.parametrize("d_v", [64, 112, 128])
@pytest.mark.parametrize("BH,L", [(1, 1), (2, 17), (3, 64), (2, 65), (149, 127), (5, 128), (297, 128), (600, 33), (2, 129)])
@pytest.mark.parametrize("flags", [0, based.BASED_NUMERATOR_ONLY])
def test_one_chunk(d_v, BH, L, flags):
    x, heads, s = case(16, d_v, BH, L)
    y_ref, _, _ = oracle.linattn_quadratic(*s)
    if flags:
        c = s[0] @ s[1].swapaxes(-1, -2)
        y_ref = y_ref * np.tril(1 + c / 4 + c * c / 32).sum(-1, keepdims=True)
    y = based.based_prefill(*x, flags=flags)
    assert row_err(wl.to_f64(y[:, heads]), y_ref) <= TOL_BF16
    assert based.based_poll_error() == based.BASED_OK


@pytest.mark.parametrize("d_v", [64, 112, 128])
@pytest.mark.parametrize("BH", [1, 16, 296, 297, 700])
@pytest.mark.parametrize("flags", [0, based.BASED_NUMERATOR_ONLY])
def test_one_chunk_same_bits_beside_a_state(d_v, BH, flags):
    """The outputs do not depend on whether the state is asked for (up to L 128 another kernel gives them then)."""
    for L in (1, 17, 32, 33, 64, 65, 97, 100, 127, 128, 129):
        gen = torch.Generator(device="cuda").manual_seed(BH * 1000 + L)
        q, k = (torch.randn(1, BH, L, 16, generator=gen, device="cuda").mul(0.5).bfloat16() for _ in range(2))
        v = torch.randn(1, BH, L, d_v, generator=gen, device="cuda").bfloat16()
        kv, z = based.new_state(1, BH, d_v)
        assert torch.equal(based.based_prefill(q, k, v, flags=flags), based.based_prefill(q, k, v, kv_state=kv, z_state=z, flags=flags)), L
    assert based.based_poll_error() == based.BASED_OK


@pytest.mark.parametrize("BH,L", [(64, 64), (64, 65), (296, 100), (297, 100), (37, 1024), (38, 1024), (49, 1408), (49, 1409), (50, 1409),
                                  (5, 4096)])
def test_lines_between_the_kernels(BH, L):
    x, heads, s = case(24, 64, BH, L)
    y_ref, S_ref, z_ref = oracle.linattn_quadratic(*s)
    y = based.based_prefill(*x)
    kv, z = based.new_state(1, BH, 64, d_feat=24)
    y_beside = based.based_prefill(*x, kv_state=kv, z_state=z)
    assert row_err(wl.to_f64(y[:, heads]), y_ref) <= TOL_BF16
    assert torch.equal(y, y_beside)
    assert_state_close(wl.to_f64(kv[:, heads]), S_ref, wl.to_f64(z[:, heads]), z_ref, "bf16")
    assert based.based_poll_error() == based.BASED_OK
