"""One-token steps at the edges of the rule for how many CTAs share a head (8 up to 18 heads, 4 up to 37, 2 up to 74): against
the recurrence in 64 bits, and the fused step of both mixers bit for bit the same."""
import pytest
import torch

import paper_2402_18668_b200 as based

pytestmark = pytest.mark.gpu


def _phi(x, sym):
    o = x[..., :, None] * x[..., None, :]
    if sym:
        m, n = torch.triu_indices(16, 16, device=x.device)
        o = o[..., m, n] * torch.where(m == n, 1 / (4 * 2 ** 0.5), 0.25).to(x)
    else:
        o = o.flatten(-2) / (4 * 2 ** 0.5)
    return torch.cat([torch.ones_like(x[..., :1]), x / 2, o], dim=-1)


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("d_v", [64, 112, 128])
@pytest.mark.parametrize("heads", [1, 18, 19, 37, 38, 74, 75])
def test_heads_shared_by_ctas(heads, d_v, sym):
    g = torch.Generator(device="cuda").manual_seed(heads + d_v)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    kv, z = based.new_state(1, heads, d_v, sym=sym)
    kv.copy_(rnd(*kv.shape))
    z.copy_(rnd(*z.shape).abs()); z[:, :, 0] += 100.0            # (denominators far from zero)
    q, k, v = rnd(1, heads, 16), rnd(1, heads, 16), rnd(1, heads, d_v)
    kc, vc = rnd(1, heads, 16, 64), rnd(1, heads, 16, 64)
    qw, kw, vw = rnd(1, heads, 64), rnd(1, heads, 64), rnd(1, heads, 64)
    kv2, z2 = kv.clone(), z.clone()
    pos = torch.tensor([20, 0], dtype=torch.int32, device="cuda")
    S, Z = kv.double(), z.double()
    pq, pk = _phi(q.double(), sym), _phi(k.double(), sym)
    S, Z = S + pk[..., None] * v.double()[..., None, :], Z + pk
    want = (pq[..., None] * S).sum(-2) / ((pq * Z).sum(-1, keepdim=True) + 1e-12)
    out = (based.based_decode_step_sym if sym else based.based_decode_step)(q, k, v, kv, z)
    # sums of 273 products in fp32: a few roundings of 2^-24 of their absolute sum, which is up to 20 times the result
    assert (out.double() - want).norm() <= 5e-6 * want.norm()
    assert (kv.double() - S).abs().max() <= 2.0 ** -22 * S.abs().max() and (z.double() - Z).abs().max() <= 2.0 ** -22 * Z.abs().max()
    fused, _ = based.based_generation_step(q, k, v, kv2, z2, qw, kw, vw, kc, vc, pos, flags=based.BASED_STATE_SYM if sym else 0)
    assert torch.equal(fused, out) and torch.equal(kv2, kv) and torch.equal(z2, z)
    assert based.based_poll_error() == based.BASED_OK
