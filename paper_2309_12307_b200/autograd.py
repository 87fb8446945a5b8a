"""torch.autograd front end of S2-Attn (Algorithm 1 of the LongLoRA paper).

`s2_attn(q, k, v, G)` behaves like a differentiable function of q [B,N,H,d] and k, v [B,N,Hkv,d]
(bf16, CUDA, contiguous): the forward runs `s2a_fwd_ex`, the backward `s2a_bwd_ex`.  Everything is
computed by the CUDA library; torch only records the graph (a C++ autograd function in
csrc/torch_binding.cpp, so that the backward does not come back to Python) and owns the tensors.
"""
from __future__ import annotations

import torch

from . import binding


def s2_attn(q: torch.Tensor, k: torch.Tensor, v: torch.Tensor, G: int, *, scale: float | None = None,
            n_unshifted: int | None = None, shift: int | None = None, leak_free: bool = False,
            swap_wrapped: bool = False, fast_backward: bool = True) -> torch.Tensor:
    """Shifted sparse attention: groups of G tokens, second half of the heads shifted by G/2.

    Keyword options as in `s2a_fwd_ex`: softmax scale (default 1/sqrt(d)), number of unshifted heads
    (default H/2), shift in tokens (default G/2), and variants 2 (`leak_free`) and 3 (`swap_wrapped`)
    of the paper's Appendix B.  With n_unshifted = H, shift = 0 and G = N it is ordinary causal attention.
    `fast_backward` chooses the backward's scratch: True allocates room for the spilled dS (2 bytes per
    attended pair of a tile, from what torch's caching allocator holds unused or within half of the free device
    memory) so that dq is a plain product, False the minimum (4 bytes per query row; dq then recomputes the scores).
    """
    hot = binding._hot or binding._hot_for(_check, q, k, v)
    o = hot.s2_attn(q, k, v, G, scale, n_unshifted, shift, binding._flags(leak_free, swap_wrapped), bool(fast_backward))
    if o is None:
        binding._result(o, "s2_attn", _check, q, k, v)
    return o if q.__class__ in binding._PLAIN else binding._typed((o,), (q,))[0]


def _check(q, k, v) -> None:
    for t, name in ((q, "q"), (k, "k"), (v, "v")):
        if not isinstance(t, torch.Tensor):
            raise ValueError(f"{name} must be a torch.Tensor")
    binding._dims(*(t.contiguous() for t in (q, k, v)))
