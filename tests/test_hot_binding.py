"""The C++ half of the binding (csrc/torch_binding.cpp) reports errors as the Python half names them: ValueError
for tensors the kernels would misread, S2AError with the library's status, also out of an autograd backward."""
import pytest
import torch

from paper_2309_12307_b200 import binding as s2a
from paper_2309_12307_b200.autograd import s2_attn
from paper_2309_12307_b200.inputs import make_inputs


@pytest.mark.parametrize("which", range(3))
@pytest.mark.parametrize("bad", [None, 3.0])
def test_s2_attn_names_an_argument_that_is_no_tensor(bad, which):
    args = [torch.zeros((1, 256, 2, 64), dtype=torch.bfloat16)] * 3
    args[which] = bad
    with pytest.raises(ValueError, match=f"{'qkv'[which]} must be a torch.Tensor"):
        s2_attn(*args, 128)


def test_s2_attn_names_a_tensor_on_the_cpu():
    q = torch.zeros((1, 256, 2, 64), dtype=torch.bfloat16)
    with pytest.raises(ValueError, match="q must be a CUDA tensor"):
        s2_attn(q, q, q, 128)


@pytest.mark.gpu
@pytest.mark.parametrize("which", range(3))
@pytest.mark.parametrize("change,message", [(lambda t: t.float(), "must have dtype"), (lambda t: t.cpu(), "must be a CUDA tensor"),
                                            (lambda t: t[0], "must be|must have shape"), (lambda t: t[..., :32], "must be|must have shape")])
def test_s2_attn_names_a_tensor_the_kernels_would_misread(change, message, which):
    args = [torch.zeros((1, 256, 2, 64), dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    args[which] = change(args[which])
    # q sets the sizes: a head of 32 in q alone is told of k
    name = "k" if which == 0 and args[0].dim() == 4 and args[0].shape[-1] == 32 else "qkv"[which]
    with pytest.raises(ValueError, match=f"^{name} ({message})"):
        s2_attn(*args, 128)


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


class Marked(torch.Tensor):
    """What a user's program may mark its tensors with."""


@pytest.mark.gpu
def test_results_have_the_class_of_their_arguments():
    q, k, v, dO = (x.cuda() for x in make_inputs(1, 512, 4, 2, 64, seed=8))
    o, lse = s2a.s2a_fwd(q, k, v, 256)
    want = s2a.s2a_bwd(q, k, v, o, lse, dO, 256, fast=1)
    mq, mk = q.as_subclass(Marked), k.as_subclass(Marked)
    mo, mlse = s2a.s2a_fwd(mq, mk, v, 256)
    assert type(mo) is Marked and type(mlse) is torch.Tensor and torch.equal(mo.as_subclass(torch.Tensor), o)
    assert type(s2a.s2a_fwd_ex(q, mk, v, 256)[0]) is torch.Tensor
    given = torch.empty_like(k)
    got = s2a.s2a_bwd(mq, mk, v, mo, lse, dO, 256, dk=given, fast="yes")
    assert [type(t) for t in got] == [Marked, torch.Tensor, Marked] and got[1] is given
    assert all(torch.equal(a.as_subclass(torch.Tensor), b) for a, b in zip(got, want))
    leaf = mq.detach().requires_grad_()
    out = s2_attn(leaf, k, v, 256, fast_backward="yes")
    assert type(out) is Marked and torch.equal(torch.autograd.grad(out, leaf, dO)[0].as_subclass(torch.Tensor), want[0])
    p = torch.nn.Parameter(q)
    assert type(s2_attn(p, k, v, 256)) is torch.Tensor and type(s2a.s2a_fwd(p.detach(), k, v, 256)[0]) is torch.Tensor
    qkv = torch.stack((q, q, q), 2).as_subclass(Marked)
    po, plse = s2a.s2a_fwd_packed(qkv, 256)
    assert type(po) is torch.Tensor and type(s2a.s2a_bwd_packed(qkv, po, plse, dO, 256)) is Marked
