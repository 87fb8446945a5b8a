"""The workspace that a backward makes for itself: no more than half of the free device memory is taken for it, but
memory that torch's caching allocator holds unused serves without a question."""
import pytest
import torch

from paper_2309_12307_b200 import binding as s2a
from paper_2309_12307_b200.autograd import s2_attn

pytestmark = pytest.mark.gpu
B, N, G, H, d = 1, 8192, 4096, 32, 64
FULL = s2a.bwd_workspace_bytes_fast(B, N, H, H, d, G, 1 << 60) if torch.cuda.is_available() else 0  # 1.1 GB


def fill(leave):
    """Takes the device's free memory but for `leave` bytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


def peak_of(run):
    torch.cuda.synchronize()
    torch.cuda.reset_peak_memory_stats()
    before = torch.cuda.memory_allocated(), torch.cuda.mem_get_info()[0]
    out = run()
    torch.cuda.synchronize()
    return out, torch.cuda.max_memory_allocated() - before[0], before[1] - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("way", ["bwd", "autograd"])
def test_a_backward_leaves_half_of_the_free_memory(way):
    q, k, v, dO = (torch.randn(B, N, H, d, device="cuda").bfloat16() for _ in range(4))
    o, lse = s2a.s2a_fwd(q, k, v, G)
    if way == "bwd":
        run = lambda: s2a.s2a_bwd(q, k, v, o, lse, dO, G)
    else:
        leaves = [t.requires_grad_() for t in (q, k, v)]
        out = s2_attn(*leaves, G)
        run = lambda: torch.autograd.grad(out, leaves, dO, retain_graph=True)
    outputs = 3 * q.numel() * 2
    want, peak, _ = peak_of(run)
    assert peak >= FULL  # there is room
    run()  # beside the first call's outputs
    held = []
    try:
        # the allocator holds the memory of the call before: nothing is taken from the device
        held.append(torch.empty(torch.cuda.mem_get_info()[0] - (256 << 20), dtype=torch.uint8, device="cuda"))
        got, peak, taken = peak_of(run)
        assert peak >= FULL and taken <= 0
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        del held[:], got
        # it holds nothing (or parts of segments in use), and the whole workspace is more than half of what is free
        leave = int(1.5 * FULL)
        held.append(fill(leave))
        got, _, taken = peak_of(run)
        assert taken <= leave // 2 + outputs + (64 << 20)  # outputs and segments in whole 2 or 20 MB
        assert all(torch.equal(a, b) for a, b in zip(got[1:], want[1:]))  # dk, dv; dq to rounding
        assert float((got[0].float() - want[0].float()).norm() / want[0].float().norm()) < 2e-3
        # it holds enough, but in pieces
        del held[:], got
        held.append(fill(leave + 2 * FULL))
        pieces = [torch.empty(FULL // 4, dtype=torch.uint8, device="cuda") for _ in range(8)]
        del pieces
        got, _, taken = peak_of(run)
        assert taken <= leave // 2 + outputs + (64 << 20)
        assert all(torch.equal(a, b) for a, b in zip(got[1:], want[1:]))
    finally:
        del held[:]
        torch.cuda.empty_cache()
    assert s2a.device_status() == (0, 0)
