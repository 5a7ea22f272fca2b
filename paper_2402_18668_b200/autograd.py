"""torch.autograd glue for the Taylor linear attention (training-time use).

`linear_attention(q, k, v)` returns based_prefill's output from the empty state (fp32: up to rounding, from the
tensor-core form of the pass where that is the faster and the device has room for its scratch) and, under
autograd, routes the output gradient through based_prefill_backward (with the saved forward
output, which lets the bf16 path merge two of its passes).  The node itself is native
(csrc_host/native.cpp), so neither direction waits for the interpreter; both run in the library's
kernels.
"""
from __future__ import annotations

from . import binding as _b


def linear_attention(q, k, v, numerator_only: bool = False):
    """Causal Taylor linear attention of q, k [B,H,L,16] and v [B,H,L,d_v] (bf16 or fp32, CUDA),
    differentiable with respect to q, k and v."""
    return _b.native().linear_attention(q, k, v, _b.BASED_NUMERATOR_ONLY if numerator_only else 0)
