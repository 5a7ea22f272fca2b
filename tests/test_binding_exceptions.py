"""Python exceptions that pass through the extension's C++ frames reach the caller as they are."""
import pytest
import torch
from torch.utils._python_dispatch import TorchDispatchMode
from torch.utils.checkpoint import checkpoint

import paper_2402_18668_b200 as based
from paper_2402_18668_b200.autograd import linear_attention
from paper_2402_18668_b200.binding import BasedError


class _Mine(Exception):
    pass


class _Raise(TorchDispatchMode):
    def __torch_dispatch__(self, func, types, args=(), kwargs=None):
        raise _Mine(str(func))


def test_exception_of_a_dispatch_mode():
    q = torch.zeros(1, 4, 2, 16).transpose(1, 2)          # not contiguous: its copy goes through the mode
    with _Raise(), pytest.raises(_Mine):
        linear_attention(q, q, q)


def _inputs(d_feat=16):
    g = torch.Generator(device="cuda").manual_seed(3)
    return [(torch.randn(2, 3, 40, w, generator=g, device="cuda") * 0.5).requires_grad_(True) for w in (d_feat, d_feat, 64)]


@pytest.mark.gpu
@pytest.mark.parametrize("which", ["pack", "unpack"])
def test_exception_of_a_saved_tensor_hook(which):
    def fail(x):
        raise _Mine(which)
    keep = lambda x: x
    with pytest.raises(_Mine, match=which):
        with torch.autograd.graph.saved_tensors_hooks(fail if which == "pack" else keep, fail if which == "unpack" else keep):
            linear_attention(*_inputs()).sum().backward()


@pytest.mark.gpu
@pytest.mark.parametrize("reentrant", [False, True])
def test_activation_checkpointing(reentrant):
    """The recomputation ends by an exception from the saved-tensor hook."""
    t = _inputs()
    want = torch.autograd.grad(linear_attention(*t).square().sum(), t)
    checkpoint(linear_attention, *t, use_reentrant=reentrant).square().sum().backward()
    for a, b in zip(t, want):
        assert torch.equal(a.grad, b)


@pytest.mark.gpu
def test_status_of_the_backward():
    """fp32 at d' 24 has a forward and no backward: the status arrives from autograd's worker thread."""
    out = linear_attention(*_inputs(24))
    with pytest.raises(BasedError, match="based_prefill_backward: unsupported") as e:
        out.sum().backward()
    assert e.value.status == 2
    assert based.based_poll_error() == based.BASED_OK
