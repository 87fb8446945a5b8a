"""Calls on a stream that is not torch's current one: what the binding allocates for them must not be shared with
work of the current stream that is still queued, neither before the call nor after it."""
import threading

import pytest
import torch

from paper_2309_12307_b200 import binding as s2a
from paper_2309_12307_b200.inputs import make_inputs

pytestmark = pytest.mark.gpu
LATE = 200_000_000  # clocks: about a tenth of a second


def calls():
    q, k, v, dO = (x.cuda() for x in make_inputs(1, 2048, 4, 4, 128, seed=9))
    qkv = torch.stack((q, k, v), 2)
    o, lse = s2a.s2a_fwd(q, k, v, 512)
    return {
        "fwd": lambda s: s2a.s2a_fwd(q, k, v, 512, stream=s),
        "fwd_ex": lambda s: s2a.s2a_fwd_ex(q, k, v, 512, leak_free=True, stream=s),
        "bwd": lambda s: s2a.s2a_bwd(q, k, v, o, lse, dO, 512, stream=s),
        "bwd_min": lambda s: s2a.s2a_bwd(q, k, v, o, lse, dO, 512, stream=s, fast=False),
        "bwd_ex": lambda s: s2a.s2a_bwd_ex(q, k, v, o, lse, dO, 512, shift=-256, stream=s),
        "fwd_packed": lambda s: s2a.s2a_fwd_packed(qkv, 512, stream=s),
        "bwd_packed": lambda s: (s2a.s2a_bwd_packed(qkv, o, lse, dO, 512, stream=s),),
    }


@pytest.mark.parametrize("call", ["fwd", "fwd_ex", "bwd", "bwd_min", "bwd_ex", "fwd_packed", "bwd_packed"])
def test_memory_of_a_call_on_another_stream_is_its_own(call):
    run = calls()[call]
    want = [t.clone() for t in run(None)]
    sizes = [t.numel() * t.element_size() for t in want] + [s2a.bwd_workspace_bytes(1, 2048, 4, 4, 128, 512),
                                                            s2a.bwd_workspace_bytes_fast(1, 2048, 4, 4, 128, 512, 1 << 40)]
    side = torch.cuda.Stream()
    run(side)  # its blocks are there from now on
    torch.cuda.synchronize()
    # the current stream writes late to memory that it gave back before the call
    torch.cuda._sleep(LATE)
    for n in sizes:
        torch.empty(n, dtype=torch.uint8, device="cuda").fill_(255)
    got = run(side)
    side.synchronize()
    first = [t.clone() for t in got]
    torch.cuda.synchronize()
    for t, f, w in zip(got, first, want):
        assert torch.equal(t, w) and torch.equal(f, w)
    # the kernels run late; the current stream takes and writes memory as soon as the call has returned
    with torch.cuda.stream(side):
        torch.cuda._sleep(LATE)
    got = run(side)
    taken = [torch.empty(n, dtype=torch.uint8, device="cuda").fill_(255) for n in sizes for _ in range(2)]
    torch.cuda.synchronize()
    del taken
    for t, w in zip(got, want):
        assert torch.equal(t, w)
    assert s2a.device_status() == (0, 0)


def test_host_entry_point_from_several_threads():
    """Calls from several threads on streams of their own share the library's copy streams and events."""
    B, N, G, H, Hkv, d = 1, 4096, 1024, 16, 16, 128
    jobs = []
    for seed in range(4):
        host_in = [t.pin_memory() for t in make_inputs(B, N, H, Hkv, d, seed=seed)]
        q, k, v, dO = (t.cuda() for t in host_in)
        ws = torch.empty(s2a.bwd_workspace_bytes(B, N, H, Hkv, d, G), dtype=torch.uint8, device="cuda")
        o, lse = s2a.s2a_fwd(q, k, v, G)
        want = (o, lse, *s2a.s2a_bwd(q, k, v, o, lse, dO, G, workspace=ws))
        host_out = [torch.zeros(t.shape, dtype=t.dtype).pin_memory() for t in want]
        jobs.append((host_in, host_out, [torch.zeros_like(t) for t in (q, k, v, dO, *want)], ws, torch.cuda.Stream(), [t.cpu() for t in want]))
    torch.cuda.synchronize()
    failed = []

    def work(host_in, host_out, dev, ws, stream, want):
        try:
            for _ in range(5):
                for t in host_out:
                    t.zero_()
                s2a.s2a_fwd_bwd_host(host_in, host_out, dev, G, ws, stream=stream)
                stream.synchronize()
                failed.extend(i for i, (a, b) in enumerate(zip(host_out, want)) if not torch.equal(a, b))
        except Exception as e:  # noqa: BLE001 - reported below
            failed.append(e)

    threads = [threading.Thread(target=work, args=job) for job in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed and s2a.device_status() == (0, 0)
