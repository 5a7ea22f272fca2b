"""Block-wise bf16 backward: the tiles of the first block (queries) and of the last (keys) need no block state and run beside the
states' kernel, ahead of all other tiles.  Last blocks of one token to a whole block, two blocks, blocks of 256 and 512 tokens, with the
running states and the scanned ones; calls back to back into the same buffers give the same bits."""
import numpy as np
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import workloads as wl
from parity import TOL_BF16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_v,BH,L", [(64, 64, 769), (64, 80, 1024), (64, 150, 897), (112, 70, 1025), (128, 64, 1281), (64, 3, 1026),
                                      (64, 1, 1100), (128, 2, 2048), (112, 16, 4097)])
@pytest.mark.parametrize("flags", [0, based.BASED_NUMERATOR_ONLY])
def test_tiles_beside_the_states(d_v, BH, L, flags):
    assert based.binding.lib().based_prefill_backward_block_tokens(1, BH, L, 16, d_v, based.BASED_BF16, flags, 1) in (256, 512)
    w = wl.Workload("beside", 1, BH, L, 16, d_v, "bf16", 0.5)
    gen = wl.generator(BH * 1000 + L + d_v)
    q, k, v = wl.prefill_inputs(w, gen)
    g = torch.randn(1, BH, L, d_v, generator=gen).bfloat16()
    heads = sorted({0, BH - 1})
    want = oracle.linattn_backward(*(wl.to_f64(t[:, heads]) for t in (q, k, v, g)), numerator_only=bool(flags))
    x = [t.cuda() for t in (q, k, v, g)]
    out = based.based_prefill(*x[:3], flags=flags)
    runs = [based.based_prefill_backward(*x, out=out, flags=flags) for _ in range(8)]
    for a, b in zip(runs[0], want):
        a = wl.to_f64(a[:, heads])
        assert (np.abs(a - b).max(axis=(0, 2, 3)) <= TOL_BF16 * np.abs(b).max(axis=(0, 2, 3))).all()
    assert all(torch.equal(a, b) for r in runs[1:] for a, b in zip(r, runs[0]))
    assert based.based_poll_error() == based.BASED_OK


@pytest.mark.parametrize("BH,L,block", [(64, 768, 0), (64, 769, 256), (16, 1024, 0), (16, 1025, 256), (3, 767, 0), (3, 768, 256), (33, 896, 0),
                                        (33, 897, 256)])
def test_lines_between_the_paths(BH, L, block):
    assert based.binding.lib().based_prefill_backward_block_tokens(1, BH, L, 16, 64, based.BASED_BF16, 0, 1) == block
    gen = wl.generator(BH * 1000 + L)
    w = wl.Workload("lines", 1, BH, L, 16, 64, "bf16", 0.5)
    q, k, v = wl.prefill_inputs(w, gen)
    g = torch.randn(1, BH, L, 64, generator=gen).bfloat16()
    heads = sorted({0, BH - 1})
    want = oracle.linattn_backward(*(wl.to_f64(t[:, heads]) for t in (q, k, v, g)))
    x = [t.cuda() for t in (q, k, v, g)]
    for a, b in zip(based.based_prefill_backward(*x, out=based.based_prefill(*x[:3])), want):
        a = wl.to_f64(a[:, heads])
        assert (np.abs(a - b).max(axis=(0, 2, 3)) <= TOL_BF16 * np.abs(b).max(axis=(0, 2, 3))).all()
