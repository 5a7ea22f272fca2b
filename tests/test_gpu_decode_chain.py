"""The one-token steps are programmatic dependent launches: a chain of them without host synchronisation, each on what the
one before wrote, gives the bits of the same chain with a synchronisation after every call."""
import pytest
import torch

import paper_2402_18668_b200 as based

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,d_v,sym", [(1, 2, 64, True), (1, 16, 128, False), (3, 16, 112, False), (20, 16, 128, True), (70, 16, 64, False)])
def test_chain_of_steps_equals_the_synchronised_chain(B, H, d_v, sym):
    window, C, width, T = 16, 512, 3, 25

    def chain(sync):
        g = torch.Generator(device="cuda").manual_seed(B + d_v)
        rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").bfloat16()
        kv, z = based.new_state(B, H, d_v, sym=sym)
        kv.normal_(generator=g); z.fill_(20.0)
        kc, vc, cs = rnd(B, H, window, 64), rnd(B, H, window, 64), rnd(B, width - 1, C)
        h, b2 = torch.randn(width, C, generator=g, device="cuda"), torch.randn(C, generator=g, device="cuda")
        x, w, c = rnd(B, H, d_v), rnd(B, H, 64), rnd(B, C)
        q, k = rnd(B, H, 16), rnd(B, H, 16)
        pos = torch.full((B,), 3, dtype=torch.int32, device="cuda")
        step = based.based_decode_step_sym if sym else based.based_decode_step
        for t in range(T):                                   # every output is the next call's input, buffers reused
            for call in (lambda: step(q, k, x, kv, z, out=x),
                         lambda: based.swa_decode_step(w, w, w, kc, vc, t, out=w) if t % 2 else
                         based.swa_decode_step_ragged(w, w, w, kc, vc, pos, out=w),
                         lambda: based.baseconv_gate_step(c, c, h, b2, cs, out=torch.empty_like(c)),
                         lambda: step(q, k, x, kv, z, out=x)):
                call()
                if sync:
                    torch.cuda.synchronize()
        return x, w, kv, z, kc, vc, cs

    want = chain(True)
    for _ in range(3):
        assert all(torch.equal(a, b) for a, b in zip(chain(False), want))
    assert based.based_poll_error() == based.BASED_OK
