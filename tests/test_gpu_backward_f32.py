"""fp32 backward on 64 x 64 tiles: lengths at the tile edges, own tiles shared by one to eight CTAs of a cluster (few
heads) and not shared (many), every value width, both forms."""
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
