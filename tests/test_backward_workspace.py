"""Scratch of the bf16 backward: the size asked for holds what the call lays out in it, with the forward output and without (the two
take the block-wise path from different lengths on), and a call writes nothing behind it."""
import itertools

import numpy as np
import pytest
import torch

import oracle
import paper_2402_18668_b200 as based
from paper_2402_18668_b200 import workloads as wl
from parity import TOL_BF16


def _aligned(n):
    return (n + 255) // 256 * 256


def _laid_out(lib, BH, L, d_v, W):
    """Bytes of the rows' statistics, the blocks' row sums (twice), with fewer than 64 heads their own fp32 sums, their states, the
    recomputed forward output and that pass's scratch."""
    blocks = BH * -(-L // W)
    parts = [BH * L * 8, blocks * 160 * 4, blocks * 160 * 4, blocks * 160 * d_v * 4 if BH < 64 else 0, blocks * 160 * d_v * 2, BH * L * d_v * 2,
             lib.based_prefill_workspace_bytes(1, BH, L, 16, d_v, based.BASED_BF16)]
    return sum(_aligned(n) for n in parts)


def test_size_holds_the_block_wise_layout():
    lib = based.binding.lib()
    lengths = sorted({*range(700, 1100), *range(1270, 1290), *range(1530, 1540), *range(2040, 2056), 512, 3000, 4096, 8192, 16384})
    bad = []
    for d_v, BH, L in itertools.product((64, 112, 128), (*range(1, 80), 128, 148, 200, 296), lengths):
        size = lib.based_prefill_backward_workspace_bytes(1, BH, L, d_v, based.BASED_BF16)
        for with_out, flags in ((0, 0), (1, 0), (0, based.BASED_NUMERATOR_ONLY)):
            W = lib.based_prefill_backward_block_tokens(1, BH, L, 16, d_v, based.BASED_BF16, flags, with_out)
            if size < (_laid_out(lib, BH, L, d_v, W) if W else BH * L * 8):
                bad.append((d_v, BH, L, with_out, flags))
    assert not bad, bad


@pytest.mark.gpu
@pytest.mark.parametrize("d_v,BH,L", [(64, 5, 1024), (64, 16, 1024), (64, 31, 1024), (64, 16, 1023), (64, 16, 1025), (64, 3, 768), (64, 33, 897),
                                      (64, 64, 769), (64, 64, 1280), (128, 16, 1536), (112, 64, 1024)])
@pytest.mark.parametrize("with_out", [False, True])
def test_nothing_behind_the_scratch(d_v, BH, L, with_out):
    gen = wl.generator(BH * 1000 + L + d_v)
    w = wl.Workload("scratch", 1, BH, L, 16, d_v, "bf16", 0.5)
    q, k, v = wl.prefill_inputs(w, gen)
    g = torch.randn(1, BH, L, d_v, generator=gen).bfloat16()
    heads = sorted({0, BH - 1})
    want = oracle.linattn_backward(*(wl.to_f64(t[:, heads]) for t in (q, k, v, g)))
    x = [t.cuda() for t in (q, k, v, g)]
    n = based.based_prefill_backward_workspace_bytes(1, BH, L, d_v, based.BASED_BF16)
    # room for all that any path lays out, so that a size that is too small shows as a changed guard and not as a stray write
    guard = _laid_out(based.binding.lib(), BH, L, d_v, 256) + 4096
    buf = torch.full((n + guard,), 0xA5, dtype=torch.uint8, device="cuda")
    got = based.based_prefill_backward(*x, workspace=buf[:n], out=based.based_prefill(*x[:3]) if with_out else None)
    for a, b in zip(got, want):
        a = wl.to_f64(a[:, heads])
        assert (np.abs(a - b).max(axis=(0, 2, 3)) <= TOL_BF16 * np.abs(b).max(axis=(0, 2, 3))).all()
    assert bool((buf[n:] == 0xA5).all())
    assert based.based_poll_error() == based.BASED_OK
