"""Order of the tile passes' grid (longest loops of all heads first, or head by head) and the lines of the block-wise
backward: one wave of tiles and a little more, ragged ends, both sides of the lines, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import workloads as wl
from parity import TOL_BF16, row_err

pytestmark = pytest.mark.gpu


def _inputs(BH, L, d_feat, d_v):
    w = wl.Workload("order", 1, BH, L, d_feat, d_v, "bf16", 0.5)
    gen = wl.generator(BH * 1000 + L + d_v)
    return (*wl.prefill_inputs(w, gen), torch.randn(1, BH, L, d_v, generator=gen).bfloat16())


def _check(q, k, v, g, with_out):
    BH = q.shape[1]
    heads = sorted({0, BH // 2, BH - 1})
    want = oracle.linattn_backward(*(wl.to_f64(t[:, heads]) for t in (q, k, v, g)))
    qd, kd, vd, gd = (t.cuda() for t in (q, k, v, g))
    out = based.based_prefill(qd, kd, vd)
    got = based.based_prefill_backward(qd, kd, vd, gd, out=out if with_out else None)
    assert based.based_poll_error() == based.BASED_OK
    for a, b in zip(got, want):
        a = wl.to_f64(a[:, heads])
        assert (np.abs(a - b).max(axis=(0, 2, 3)) <= TOL_BF16 * np.abs(b).max(axis=(0, 2, 3))).all()
    return out, heads


# tiles of 128 rows: 148 of them is one per SM
@pytest.mark.parametrize("d_feat", [16, 24])
@pytest.mark.parametrize("d_v,BH,L", [(64, 37, 512), (64, 30, 513), (128, 75, 190), (112, 74, 255), (64, 149, 64)])
@pytest.mark.parametrize("with_out", [True, False])
def test_tile_passes_in_either_order(d_feat, d_v, BH, L, with_out):
    q, k, v, g = _inputs(BH, L, d_feat, d_v)
    out, heads = _check(q, k, v, g, with_out)
    want = oracle.linattn_quadratic(*(wl.to_f64(t[:, heads]) for t in (q, k, v)))[0]
    assert row_err(wl.to_f64(out[:, heads]), want) <= TOL_BF16


@pytest.mark.parametrize("d_v,BH,L,tokens", [(64, 19, 2047, 0), (64, 19, 2048, 256), (64, 18, 2000, 256), (128, 63, 2047, 0),
                                             (112, 24, 2049, 256), (128, 16, 4096, 512), (128, 15, 4100, 256),
                                             (64, 74, 800, 256), (64, 75, 1281, 256), (112, 74, 1100, 256), (128, 75, 1024, 256)])
def test_lines_of_the_blockwise_path(d_v, BH, L, tokens):
    assert based.lib().based_prefill_backward_block_tokens(1, BH, L, 16, d_v, 1, 0, 1) == tokens
    _check(*_inputs(BH, L, 16, d_v), True)


@pytest.mark.parametrize("what", ["backward f32", "backward bf16", "state"])
def test_scratch_of_a_call_belongs_to_its_stream(what):
    """Scratch of a call on another stream than the current one is not handed out on the current one, where nothing waits for that
    call; and the results are those of the current stream."""
    B, H, L, d_v = {"backward f32": (2, 16, 1024, 64), "backward bf16": (4, 16, 2048, 64), "state": (1, 148, 2048, 128)}[what]
    g = torch.Generator(device="cuda").manual_seed(1)
    dt = torch.float32 if what == "backward f32" else torch.bfloat16
    q, v, dout = (torch.randn(B, H, L, d, generator=g, device="cuda").to(dt) for d in (16, d_v, d_v))

    def call(stream=None):
        if what == "state":
            return based.based_prefill_state(q, v, stream=stream)
        return based.based_prefill_backward(q, q, v, dout, stream=stream)
    want = call()
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    got = call(other)
    torch.cuda.synchronize()
    reserved = torch.cuda.memory_reserved()
    after = torch.empty((11 if what == "state" else 25) << 20, dtype=torch.uint8, device="cuda")     # (the scratch: 12 and 28 to 30 MB)
    assert torch.cuda.memory_reserved() > reserved
    del after
    assert all(torch.equal(a, b) for a, b in zip(got, want))
