"""The C++ half of the binding (csrc/torch_binding.cpp) reports errors as the Python half names them: ValueError
for tensors the kernels would misread, S2AError with the library's status, also out of an autograd backward."""
import pytest
import torch

from paper_2309_12307_b200 import binding as s2a
from paper_2309_12307_b200.autograd import s2_attn
from paper_2309_12307_b200.inputs import make_inputs


@pytest.mark.parametrize("bad", ["cpu", "dtype", "none"])
def test_s2_attn_names_a_bad_argument(bad):
    q = torch.zeros((1, 256, 2, 64), dtype=torch.float32 if bad == "dtype" else torch.bfloat16)
    with pytest.raises((ValueError, AttributeError)):
        s2_attn(None if bad == "none" else q, q, q, 128)


@pytest.mark.gpu
def test_status_reaches_the_caller_from_forward_and_backward():
    q, k, v, dO = (x.cuda() for x in make_inputs(1, 1024, 4, 2, 64, seed=5))
    with pytest.raises(s2a.S2AError) as e:
        s2_attn(q, k, v, 384)  # N % G
    assert e.value.status == s2a.S2A_ERR_INVALID_ARG
    with pytest.raises(ValueError, match="dq must have shape"):
        o, lse = s2a.s2a_fwd(q, k, v, 256)
        s2a.s2a_bwd(q, k, v, o, lse, dO, 256, dq=torch.empty_like(k))
    for t in (q, k, v):
        t.requires_grad_()
    o = s2_attn(q, k, v, 256)
    s2a.selftest_wait_expiry(1_000_000)  # a bounded wait runs out: entry points refuse until the status is read
    torch.cuda.synchronize()
    with pytest.raises(s2a.S2AError) as e:
        torch.autograd.grad(o, (q, k, v), dO)
    assert e.value.status == s2a.S2A_ERR_TIMEOUT
    assert s2a.device_status()[0] == s2a.S2A_ERR_TIMEOUT and s2a.device_status() == (0, 0)


@pytest.mark.gpu
def test_s2_attn_takes_strided_inputs_and_gradients():
    q, k, v, dO = (x.cuda() for x in make_inputs(2, 512, 4, 2, 128, seed=6))
    o, lse = s2a.s2a_fwd(q, k, v, 256)
    want = (o, *s2a.s2a_bwd(q, k, v, o, lse, dO, 256))
    strided = [t.transpose(1, 2).contiguous().transpose(1, 2).requires_grad_() for t in (q, k, v)]
    o = s2_attn(*strided, 256)
    got = (o.detach(), *torch.autograd.grad(o, strided, dO.transpose(1, 2).contiguous().transpose(1, 2)))
    for a, b in zip(got, want):
        assert torch.equal(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("change", [lambda t: t.half(), lambda t: t[..., ::2], lambda t: t[..., :32].contiguous(), lambda t: t.cpu(),
                                    lambda t: t.transpose(1, 2).contiguous().transpose(1, 2)])
@pytest.mark.parametrize("which", range(5))
def test_backward_refuses_saved_tensors_that_come_back_changed(change, which):
    """q, k, v, o, lse pass through saved-tensor hooks; the kernels read them by their raw pointers."""
    q, k, v, dO = (x.cuda() for x in make_inputs(1, 512, 4, 2, 64, seed=7))
    for t in (q, k, v):
        t.requires_grad_()
    saved = []
    with torch.autograd.graph.saved_tensors_hooks(lambda t: saved.append(t) or len(saved) - 1,
                                                  lambda i: change(saved[i].detach()) if i == which else saved[i]):
        o = s2_attn(q, k, v, 256)
    assert [t.dtype for t in saved] == [torch.bfloat16] * 4 + [torch.float32]
    with pytest.raises(ValueError, match="saved"):
        torch.autograd.grad(o, (q, k, v), dO)
