"""Every wait of a whole warp must end the same way for all its lanes (mbar_wait_uniform): mbar_wait decides lane by
lane, so it may only stand where a single lane runs."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2309_12307_b200", "csrc")


@pytest.mark.parametrize("name", ["fwd_kernel.cu", "bwd_kernels.cu"])
def test_lanes_wait_alone_only_where_one_lane_runs(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    found, single_lane = 0, []  # single_lane: per open brace, whether it opened the body of a one-lane branch
    for m in re.finditer(r"\bif \(lane == 0\) \{|\bif \(elect_one\(\)\) \{|\{|\}|\bmbar_wait\(|\bmbar_wait_drain\(", text):
        token = m.group()
        if token.endswith("{"):
            single_lane.append(token != "{")
        elif token == "}":
            single_lane.pop()
        else:
            found += 1
            assert any(single_lane), f"{name}: {token} of a whole warp in line {text.count(chr(10), 0, m.start()) + 1}"
    assert found > 0 and not single_lane


def _statement_end(text, i):
    """Where the statement at i ends: after its braces, or after its semicolon."""
    depth, brackets = 0, 0
    for x in range(i, len(text)):
        c = text[x]
        depth += (c == "{") - (c == "}")
        brackets += (c in "([") - (c in ")]")
        if brackets == 0 and depth == 0 and c in ";}":
            return x + 1
    raise ValueError(text[i:i + 60])


def _instance(text, constants):
    """The text as one template instance has it: the branches of `if constexpr` that are taken."""
    while m := re.search(r"if constexpr \(([^()]*)\)\s*", text):
        end = _statement_end(text, m.end())
        other = re.compile(r"\s*else\b\s*").match(text, end)
        stop = _statement_end(text, other.end()) if other else end
        taken = eval(m.group(1), {}, constants)
        keep = text[m.end():end] if taken else text[other.end():stop] if other else ""
        text = text[:m.start()] + keep + text[stop:]
    return text


def _inlined(text):
    """The text with every named lambda's body in the place of its calls."""
    while m := re.search(r"\bauto (\w+) = \[[^\]]*\]\s*\([^)]*\)[^{;]*\{", text):
        end = _statement_end(text, m.end() - 1)
        body = text[m.end() - 1:end]
        rest = re.sub(rf"\b{m.group(1)}\([^()]*\)", lambda _: body, text[end:])
        text = text[:m.start()] + rest
    return text


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("name", ["fwd_kernel.cu", "bwd_kernels.cu"])
def test_no_wait_can_give_up_on_stores_to_tensor_memory(name, hd):
    """A warp whose wait runs out leaves for the end of the block, where the tensor memory is given back: its own stores
    must be complete by then.  So no bounded wait stands between a store and the wait for the stores, unless the branch that
    gives up begins with that wait itself."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    constants = dict(kPBufs=2 if hd == 64 else 1, kVInTmem=hd == 64, kSpill=True)
    text = _inlined(_instance(text, constants))
    text = re.sub(r"\bif \(!mbar_wait\w*\([^;{}]*\)\) \{ tmem_wait_st\(\); return false; \}", "", text)
    stores, pending = 0, 0
    for m in re.finditer(r"\btmem_st_\w+\(|\btmem_wait_st\(|\b(?:mbar_wait\w*|next_item)\(|\bnamed_barrier\w*\(", text):
        token = m.group()
        if token.startswith("tmem_st_"):
            stores, pending = stores + 1, pending + 1
        elif token.startswith("tmem_wait_st"):
            pending = 0
        else:
            assert pending == 0, f"{name}, head size {hd}: {token} after stores to tensor memory that are not waited for"
    assert stores > 0 and pending == 0
