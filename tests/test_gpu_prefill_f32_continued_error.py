"""fp32 prompt pieces appended to few sequences: the rounding of the outputs, as a share of them (root of the mean square)."""
import pytest
import torch

import paper_2402_18668_b200 as based

pytestmark = pytest.mark.gpu


def phi(x):
    return torch.cat([torch.ones_like(x[..., :1]), x / 2, (x[..., :, None] * x[..., None, :]).flatten(-2) / 32 ** 0.5], -1)


@pytest.mark.parametrize("d_v", [64, 112])
@pytest.mark.parametrize("L", [5, 96, 188])
def test_error_of_a_continued_piece(d_v, L):
    """The state's 153 terms of an output are summed in sixteen runs of ten and those in pairs: by the rounding of each addition (a random
    walk, checked with the same sums on the CPU) 1.0e-7 to 1.25e-7 and the folding of the state's rows; 1.35e-7 to 1.6e-7 in runs of
    twenty behind the keys, added one after the other."""
    BH = 8
    g = torch.Generator(device="cuda").manual_seed(L)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    error = norm = 0.0
    for _ in range(200 // L + 2):
        q, k, v = rnd(1, BH, L, 16), rnd(1, BH, L, 16), rnd(1, BH, L, d_v)
        f = phi(rnd(1, BH, 64, 16).double())
        kv, z = (f.transpose(-1, -2) @ rnd(1, BH, 64, d_v).double()).float(), f.sum(-2).float()
        fq = phi(q.double())
        s = q.double() @ k.double().transpose(-1, -2)
        w = torch.tril(1 + s / 4 + s * s / 32)
        want = (w @ v.double() + fq @ kv.double()) / (w.sum(-1) + (fq @ z.double()[..., None])[..., 0])[..., None]
        y = based.based_prefill(q, k, v, kv_state=kv, z_state=z, flags=based.BASED_STATE_CONTINUE)
        error += float(((y - want) ** 2).sum())
        norm += float((want ** 2).sum())
    assert (error / norm) ** 0.5 <= 1.4e-7
    assert based.based_poll_error() == based.BASED_OK
