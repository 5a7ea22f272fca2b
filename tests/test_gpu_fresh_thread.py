"""Calls from a host thread that no CUDA runtime call has touched yet (autograd's worker thread is one, when the buffers
of the backward pass come out of torch's allocator cache): the library has to bind the device's context itself."""
import threading

import pytest
import torch

import paper_2402_18668_b200 as based

pytestmark = pytest.mark.gpu


def _in_fresh_thread(fn):
    got = []

    def body():
        try:
            got.append(("ok", fn()))
        except Exception as e:              # noqa: BLE001  (re-raised in the test's own thread)
            got.append(("error", e))
    t = threading.Thread(target=body)
    t.start()
    t.join()
    if got[0][0] == "error":
        raise got[0][1]
    return got[0][1]


@pytest.mark.parametrize("what", ["prefill", "state", "window", "backward", "backward_blocks", "dfeat"])
def test_entry_points_from_a_thread_without_a_context(what):
    g = torch.Generator(device="cuda").manual_seed(3)
    L = 1024 if what == "backward_blocks" else 300
    d = 24 if what == "dfeat" else 16
    q, k = ((torch.randn(1, 3, L, d, generator=g, device="cuda") * 0.4).bfloat16() for _ in range(2))
    v, g_ = (torch.randn(1, 3, L, 64, generator=g, device="cuda").bfloat16() for _ in range(2))
    call = {"prefill": lambda: based.based_prefill(q, k, v), "dfeat": lambda: based.based_prefill(q, k, v),
            "state": lambda: based.based_prefill_state(k, v), "window": lambda: based.swa_forward(v, g_, v),
            "backward": lambda: based.based_prefill_backward(q, k, v, g_),
            "backward_blocks": lambda: based.based_prefill_backward(q, k, v, g_)}[what]
    want = call()
    again = call()                          # leaves blocks of every size in the allocator's cache: no cudaMalloc below
    torch.cuda.synchronize()
    del again
    got = _in_fresh_thread(call)
    assert based.based_poll_error() == based.BASED_OK
    for a, b in zip(*((x,) if isinstance(x, torch.Tensor) else x for x in (got, want))):
        assert torch.equal(a, b)
