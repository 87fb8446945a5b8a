"""The work that a user of this library has it do: what is timed when a kernel or the host path changes.

A case is one pass of S2-Attn through a public entry point.  `path` says which one:

  autograd   s2_attn() and torch.autograd.grad: a training step as a model's attention layer makes it
  train      s2a_fwd + s2a_bwd with a workspace that the caller keeps (at most 24 GiB)
  train_min  s2a_fwd + s2a_bwd with the least workspace, which the caller keeps: dq recomputes the scores
  packed     s2a_fwd_packed + s2a_bwd_packed: qkv in one tensor, as Algorithm 1 is called
  noalloc    s2a_bwd_noalloc alone, on the o and lse of an earlier forward pass
  forward    s2a_fwd: evaluation, or a forward pass under activation checkpointing
  causal     s2a_fwd_ex with one group and no shift: the full causal attention a fine-tuned model prefills with
  host       s2a_fwd_bwd_host: pinned host tensors in and out

`variant` is the treatment of the group that wraps around the sequence end: the paper's default, "leak_free" or
"swap_wrapped".  Sizes are the Llama2 attention shapes of inputs.py and of the tests; values are N(0, 1) in bf16,
as everywhere in this repository.
"""
from __future__ import annotations

import math

import torch

from paper_2309_12307_b200 import binding
from paper_2309_12307_b200.autograd import s2_attn

WORKSPACE_BUDGET = 24 << 30


def _case(path, B, N, G, H, Hkv, d, variant="default"):
    return dict(path=path, B=B, N=N, G=G, H=H, Hkv=Hkv, d=d, variant=variant)


def listed():
    cases = {
        # the smallest training step: a few dozen tiles, so launches and host time are what it costs
        "tiny_train": _case("autograd", 1, 1024, 256, 4, 4, 64),
        # short ragged sequences in a batch: 200-token groups on 128-token tiles, grouped KV heads
        "ragged_batch_train": _case("autograd", 4, 2000, 200, 16, 4, 64),
        # variant 2 of the paper's appendix on a mid-sized grouped-query model with head size 64
        "leak_free_gqa_train": _case("autograd", 2, 4096, 1024, 32, 8, 64, "leak_free"),
        # fine-tuning a 7B model at the shortest context length: one attention layer of the step
        "7b_8k_train": _case("autograd", 1, 8192, 2048, 32, 32, 128),
        # the same layer in evaluation
        "7b_8k_forward": _case("forward", 1, 8192, 2048, 32, 32, 128),
        # the fine-tuned model at inference: ordinary causal attention over the whole prompt
        "7b_8k_causal_prefill": _case("causal", 1, 8192, 8192, 32, 32, 128),
        # the same layer by a caller that keeps its tensors on the host
        "7b_8k_host": _case("host", 1, 8192, 2048, 32, 32, 128),
        # Algorithm 1's own calling convention, one packed tensor, twice the context
        "7b_16k_packed_train": _case("packed", 1, 16384, 4096, 32, 32, 128),
        # gradients in a program that has no memory to give
        "7b_16k_backward_noalloc": _case("noalloc", 1, 16384, 4096, 32, 32, 128),
        # the shape that the benchmark quotes
        "7b_32k_train": _case("train", 1, 32768, 8192, 32, 32, 128),
        # a 70B model: eight query heads to a KV head
        "70b_32k_gqa_train": _case("train", 1, 32768, 8192, 64, 8, 128),
        # the longest context, in its literal form: groups of 25,000 tokens, not a multiple of a tile
        "7b_100000_train": _case("train", 1, 100000, 25000, 32, 32, 128),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _pairs(case):
    """(query, key) pairs attended."""
    B, N, G, H = case["B"], case["N"], case["G"], case["H"]
    per_group = G * (G + 1) // 2
    pairs = B * H * (N // G) * per_group
    if case["variant"] == "leak_free":  # the wrapped group of a shifted head is two groups of G / 2
        pairs -= B * (H // 2) * (per_group - 2 * (G // 2 * (G // 2 + 1) // 2))
    return pairs


def _elements(case):
    """Elements of one query-shaped and of one key-shaped tensor, and rows of statistics."""
    rows = case["B"] * case["N"]
    return rows * case["H"] * case["d"], rows * case["Hkv"] * case["d"], rows * case["H"]


LARGEST = _case("train", 1, 100000, 25000, 32, 32, 128)


def draw(rng):
    """One more case: path, model shape, group size, number of groups and batch, sizes spread over their logarithm."""
    while True:
        path = rng.choice(["autograd", "autograd", "train", "train", "train_min", "packed", "noalloc", "forward", "forward", "causal", "host"])
        H, Hkv, d = rng.choice([(4, 4, 64), (8, 2, 64), (16, 4, 64), (32, 32, 64), (8, 8, 128), (32, 32, 128), (32, 32, 128), (40, 40, 128), (64, 8, 128)])
        if path == "packed":
            Hkv = H
        B = rng.choice([1, 1, 1, 2, 4])
        G = int(math.exp(rng.uniform(math.log(128), math.log(25600))))
        # two groups in three are whole tiles, the rest as ragged as the entry points take
        G = G // 256 * 256 if rng.random() < 0.67 else G // 8 * 8
        groups = rng.choice([1, 2, 3, 4, 4, 4, 6, 8, 16])
        if G == 0 or (path == "causal" and groups != 1):
            continue
        variant = rng.choice(["default", "default", "leak_free", "swap_wrapped"]) if path == "autograd" else "default"
        case = _case(path, B, G * groups, G, H, Hkv, d, variant)
        if case["N"] < 1024:
            continue
        q_elements, _, rows = _elements(case)
        most = _elements(LARGEST)[0]
        if path == "noalloc" and rows > binding.bwd_noalloc_max_rows():
            continue
        if path == "host":
            most //= 8
        cost, limit = work(case), work(LARGEST)
        if q_elements > most or cost["flops"] > limit["flops"] or cost["bytes"] > limit["bytes"]:
            continue
        # an autograd call takes its scratch from the free device memory: keep it well inside
        if path == "autograd" and binding.bwd_workspace_bytes_fast(B, case["N"], H, Hkv, d, G, 1 << 60) > WORKSPACE_BUDGET:
            continue
        return case


class State:
    """What the caller holds: inputs, and buffers that its program keeps from step to step."""


def prepare(case, seed):
    s = State()
    s.case = case
    B, N, G, H, Hkv, d = (case[k] for k in ("B", "N", "G", "H", "Hkv", "d"))
    path = case["path"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def normal(*shape):
        return torch.randn(shape, generator=gen, dtype=torch.float32, device="cuda").to(torch.bfloat16)

    if path == "packed":
        s.qkv = normal(B, N, 3, H, d)
    else:
        s.q, s.k, s.v = normal(B, N, H, d), normal(B, N, Hkv, d), normal(B, N, Hkv, d)
    if path not in ("forward", "causal"):
        s.dO = normal(B, N, H, d)

    if path == "autograd":
        for t in (s.q, s.k, s.v):
            t.requires_grad_()
        s.options = {} if case["variant"] == "default" else {case["variant"]: True}
    elif path in ("train", "packed", "train_min"):
        need = binding.bwd_workspace_bytes(B, N, H, Hkv, d, G)
        if path != "train_min":
            need = binding.bwd_workspace_bytes_fast(B, N, H, Hkv, d, G, WORKSPACE_BUDGET)
        s.workspace = torch.empty(need, dtype=torch.uint8, device="cuda")
    elif path == "noalloc":
        s.o, s.lse = binding.s2a_fwd(s.q, s.k, s.v, G)
        s.dq, s.dk, s.dv = torch.empty_like(s.q), torch.empty_like(s.k), torch.empty_like(s.v)
    elif path == "host":
        inputs = (s.q, s.k, s.v, s.dO)
        s.host_in = tuple(torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in inputs)
        lse = torch.empty((B, H, N), dtype=torch.float32, device="cuda")
        outputs = (torch.empty_like(s.q), lse, torch.empty_like(s.q), torch.empty_like(s.k), torch.empty_like(s.v))
        s.host_out = tuple(torch.empty(t.shape, dtype=t.dtype, pin_memory=True) for t in outputs)
        s.device_buffers = inputs + outputs
        need = binding.bwd_workspace_bytes_fast(B, N, H, Hkv, d, G, WORKSPACE_BUDGET)
        s.workspace = torch.empty(need, dtype=torch.uint8, device="cuda")
    return s


def run(s):
    case, path, G = s.case, s.case["path"], s.case["G"]
    if path == "autograd":
        o = s2_attn(s.q, s.k, s.v, G, **s.options)
        return (o.detach(), *torch.autograd.grad(o, (s.q, s.k, s.v), s.dO))
    if path in ("train", "train_min"):
        o, lse = binding.s2a_fwd(s.q, s.k, s.v, G)
        return (o, lse, *binding.s2a_bwd(s.q, s.k, s.v, o, lse, s.dO, G, workspace=s.workspace))
    if path == "packed":
        o, lse = binding.s2a_fwd_packed(s.qkv, G)
        return o, lse, binding.s2a_bwd_packed(s.qkv, o, lse, s.dO, G, workspace=s.workspace)
    if path == "noalloc":
        return binding.s2a_bwd_noalloc(s.q, s.k, s.v, s.o, s.lse, s.dO, G, s.dq, s.dk, s.dv)
    if path == "forward":
        return binding.s2a_fwd(s.q, s.k, s.v, G)
    if path == "causal":
        return binding.s2a_fwd_ex(s.q, s.k, s.v, G, n_unshifted=case["H"], shift=0)
    if path == "host":
        binding.s2a_fwd_bwd_host(s.host_in, s.host_out, s.device_buffers, G, s.workspace)
        return s.host_out
    raise ValueError(path)


def work(case):
    """Every input read once and every output written once; 4 d operations for each attended pair forward, 10 d backward."""
    q, kv, rows = _elements(case)
    path = case["path"]
    forward = 2 * (q + 2 * kv)            # q, k, v
    gradients = 2 * (q + 2 * kv)          # dq, dk, dv
    if path in ("forward", "causal"):
        return {"bytes": forward + 2 * q + 4 * rows, "flops": 4 * case["d"] * _pairs(case)}
    if path == "noalloc":
        return {"bytes": forward + 4 * q + 4 * rows + gradients, "flops": 10 * case["d"] * _pairs(case)}
    lse = 0 if path == "autograd" else 4 * rows
    return {"bytes": forward + 2 * q + 2 * q + lse + gradients, "flops": 14 * case["d"] * _pairs(case)}


def tolerance(case):
    """bf16 results of fp32 sums, with the probabilities and their gradients rounded to bf16 ahead of the second product.

    Against the same operator in 64 bits, groups of 200 to 4096 tokens: o 2.0e-3, dv 2.3e-3, dq and dk 2.5e-3 (2-norm),
    largest single differences 0.07 to 0.09 of the result's root mean square; about four times that is allowed.
    """
    return {"rel": 1e-2, "max": 0.3}
