"""The kernels' work items at the edges of their tiles, against the CPU oracle: groups of one tile, of an odd
number of tiles (a query tile without a partner), last tiles that end inside, at and just past the 32 rows
that one TMA store covers, more items than blocks and fewer.

Tolerances as everywhere: bf16 results of fp32 sums against fp64 (one bf16 rounding of an o of up to 4 is
8e-3 plus the rounding of the probabilities: 2e-2; 1e-2 relative L2 on the gradients).
"""
import math

import numpy as np
import pytest
import torch

from oracle import s2a_oracle as orc
from paper_2309_12307_b200.inputs import make_inputs

pytestmark = pytest.mark.gpu


def rel_l2(got, want):
    return float(np.linalg.norm(got - want) / max(np.linalg.norm(want), 1e-30))


@pytest.mark.parametrize("B,N,G,H,Hkv,d,kw", [
    (1, 128, 128, 2, 2, 128, {}),                       # the smallest: one group, its shifted heads of two half tiles
    (1, 256, 128, 2, 1, 64, {"n_unshifted": 2}),        # one tile per group, nothing shifted
    (1, 768, 384, 4, 2, 128, {}),                       # three tiles
    (1, 320, 160, 2, 2, 64, {}),                        # 32 rows in the last tile
    (2, 336, 168, 2, 2, 128, {}),                       # 40 rows, 84-row runs where the group wraps
    (1, 384, 192, 2, 2, 128, {"leak_free": True}),      # a cut inside a pair of tiles
    (1, 168, 168, 2, 2, 128, {}),                       # D's last block has half of its rows
    (3, 136, 136, 2, 2, 64, {}),                        # and three quarters
    (1, 1920, 640, 4, 4, 64, {"leak_free": True}),      # five tiles, cut after the third
    (1, 640, 320, 2, 2, 128, {"swap_wrapped": True}),
    (3, 1536, 128, 10, 2, 64, {"n_unshifted": 5}),      # more units than blocks
    (2, 16384, 128, 8, 8, 64, {"n_unshifted": 8}),      # 14 items to a block, none with a second query tile
    (1, 4992, 1664, 12, 12, 64, {}),                    # 13 tiles: more pairs than blocks, the last one single
])
def test_tile_edges_match_oracle(B, N, G, H, Hkv, d, kw):
    from paper_2309_12307_b200 import binding as s2a

    q, k, v, dO = make_inputs(B, N, H, Hkv, d, seed=31)
    o_ref, lse_ref = orc.fwd(q, k, v, G, **kw)
    grads_ref = orc.bwd(q, k, v, dO, G, **kw)
    qd, kd, vd, dOd = (x.cuda() for x in (q, k, v, dO))
    o, lse = (torch.full(s, float("nan"), dtype=t, device="cuda") for s, t in ((qd.shape, torch.bfloat16), ((B, H, N), torch.float32)))
    s2a.s2a_fwd_ex(qd, kd, vd, G, o=o, lse=lse, **kw)
    assert np.abs(o.double().cpu().numpy() - o_ref).max() <= 2e-2
    assert np.abs(lse.double().cpu().numpy() - lse_ref).max() <= 2e-3
    for fast in (False, True):
        grads = tuple(torch.full_like(x, float("nan")) for x in (qd, kd, vd))
        s2a.s2a_bwd_ex(qd, kd, vd, o, lse, dOd, G, fast=fast, dq=grads[0], dk=grads[1], dv=grads[2], **kw)
        for got, want, name in zip(grads, grads_ref, ("dq", "dk", "dv")):
            err = rel_l2(got.double().cpu().numpy(), want)
            assert math.isfinite(err) and err <= 1e-2, (name, fast, err)
    assert s2a.device_status() == (0, 0)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("N,G,kw", [(6144, 384, {}),                          # a pair and a single tile to each group
                                    (6144, 128, {"n_unshifted": 16}),         # single tiles only
                                    (4800, 480, {"leak_free": True})])        # ragged, two to four tiles
def test_forward_items_of_either_parity(N, G, kw, d):
    """The two groups of softmax warps take the later tile of a block's items in turn: several items to a block, with one tile and
    with two in every order.  Tolerance as above."""
    from paper_2309_12307_b200 import binding as s2a

    H = 16
    q, k, v, _ = make_inputs(1, N, H, H, d, seed=43)
    o_ref, lse_ref = orc.fwd(q, k, v, G, **kw)
    o, lse = (torch.full(s, float("nan"), dtype=t, device="cuda") for s, t in ((q.shape, torch.bfloat16), ((1, H, N), torch.float32)))
    s2a.s2a_fwd_ex(q.cuda(), k.cuda(), v.cuda(), G, o=o, lse=lse, **kw)
    assert np.abs(o.double().cpu().numpy() - o_ref).max() <= 2e-2
    assert np.abs(lse.double().cpu().numpy() - lse_ref).max() <= 2e-3
    assert s2a.device_status() == (0, 0)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("N,G,H,kw", [(15360, 384, 32, {}),                   # a pair and a single tile to each group: 17 items to a block
                                      (15360, 128, 32, {"n_unshifted": 32}),  # single tiles only: 26 to a block, 13 to either group of warps
                                      (15360, 640, 32, {"leak_free": True})])  # five tiles, six where a group is cut: 16 items
def test_forward_item_lists_go_round_their_rings(N, G, H, kw, d):
    """More items to a block than its rings of eight hold, where a list's position is not the item's slot: every row against the
    same kernel on a part of the heads, which gives a block a few items (the same sums, so the same bits; see the test above for
    these against the oracle)."""
    from paper_2309_12307_b200 import binding as s2a

    gen = torch.Generator(device="cuda").manual_seed(47)
    q, k, v = (torch.randn(1, N, H, d, generator=gen, device="cuda").bfloat16() for _ in range(3))
    o, lse = (torch.full(s, float("nan"), dtype=t, device="cuda") for s, t in ((q.shape, torch.bfloat16), ((1, H, N), torch.float32)))
    s2a.s2a_fwd_ex(q, k, v, G, o=o, lse=lse, **kw)
    n_unshifted = kw.get("n_unshifted", H // 2)
    for h in range(0, H, 4):
        part = [x[:, :, h:h + 4].contiguous() for x in (q, k, v)]
        want_o, want_lse = s2a.s2a_fwd_ex(*part, G, **{**kw, "n_unshifted": min(4, max(0, n_unshifted - h))})
        assert torch.equal(o[:, :, h:h + 4], want_o) and torch.equal(lse[:, h:h + 4], want_lse)
    assert s2a.device_status() == (0, 0)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("rows", [4, 12, 16, 20, 28, 32, 36, 48, 60, 64, 68, 124])
def test_masked_blocks_of_the_backward(rows, d):
    """dK/dV take the diagonal and the end of a ragged tile in blocks of 32 keys by 16 queries that are visible as a whole, in
    part or not at all.  Two tiles per group, the second of `rows` rows, which is judged by itself as well; tolerance as above."""
    from paper_2309_12307_b200 import binding as s2a

    G, H = 128 + rows, 2
    q, k, v, dO = make_inputs(1, 2 * G, H, H, d, seed=41)
    kw = {"n_unshifted": H, "shift": 0}
    grads_ref = orc.bwd(q, k, v, dO, G, **kw)
    qd, kd, vd, dOd = (x.cuda() for x in (q, k, v, dO))
    o, lse = s2a.s2a_fwd_ex(qd, kd, vd, G, **kw)
    for fast in (False, True):
        grads = tuple(torch.full_like(x, float("nan")) for x in (qd, kd, vd))
        s2a.s2a_bwd_ex(qd, kd, vd, o, lse, dOd, G, fast=fast, dq=grads[0], dk=grads[1], dv=grads[2], **kw)
        for got, want, name in zip(grads, grads_ref, ("dq", "dk", "dv")):
            got, want = (x.reshape(1, 2, G, H, d) for x in (got.double().cpu().numpy(), want))
            for part in (slice(None), slice(128, G)):
                err = rel_l2(got[:, :, part], want[:, :, part])
                assert math.isfinite(err) and err <= 1e-2, (name, fast, part, err)
    assert s2a.device_status() == (0, 0)


@pytest.mark.parametrize("B,N,G,H,Hkv,d", [(1, 8192, 2048, 32, 32, 64),   # groups and heads cut
                                           (1, 6000, 600, 16, 8, 128),    # ragged tiles; two groups in the chunk that wraps
                                           (2, 4096, 4096, 16, 4, 128),   # one group: heads cut only
                                           (1, 8192, 1024, 6, 3, 128),    # a KV head with shifted and unshifted query heads
                                           (20, 1024, 512, 4, 4, 128)])   # several batch items to a chunk, not the same number
@pytest.mark.parametrize("fast", [False, True])
def test_host_chunks_equal_device_path(B, N, G, H, Hkv, d, fast):
    """A chunk of the host entry point cuts its groups into the tiles of the whole job, so nothing differs by a bit."""
    from paper_2309_12307_b200 import binding as s2a
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(5)
    q, dO = (torch.randn(B, N, H, d, generator=gen, device=dev).bfloat16() for _ in range(2))
    k, v = (torch.randn(B, N, Hkv, d, generator=gen, device=dev).bfloat16() for _ in range(2))
    o, lse = s2a.s2a_fwd(q, k, v, G)
    need = s2a.bwd_workspace_bytes_fast(B, N, H, Hkv, d, G, 1 << 40) if fast else s2a.bwd_workspace_bytes(B, N, H, Hkv, d, G)
    ws = torch.empty(need, dtype=torch.uint8, device=dev)
    want = (o, lse, *s2a.s2a_bwd(q, k, v, o, lse, dO, G, workspace=ws))
    host_in = [x.cpu().pin_memory() for x in (q, k, v, dO)]
    host_out = [torch.full(x.shape, float("nan"), dtype=x.dtype).pin_memory() for x in want]
    s2a.s2a_fwd_bwd_host(host_in, host_out, [torch.empty_like(x) for x in (q, k, v, dO, *want)], G, ws)
    torch.cuda.synchronize()
    assert s2a.device_status()[0] == 0
    for got, ref in zip(host_out, want):
        assert torch.equal(got, ref.cpu())


@pytest.mark.parametrize("d", [64, 128])
def test_row_sums_add_neighbouring_columns_first(d):
    """One key with weight 1 ahead of keys with weight 2^-24, half an ulp of it: added one by one to the 1 they are lost, added
    in pairs first they count.  The sum of each half tile is four chains of pairs; l = 1 + x is known, and lse = log(l) to
    1 ulp of log2 and the 2^-22 of an exponential, of x (a chain for each column parity misses x by 1/128 to 1/2)."""
    from paper_2309_12307_b200 import binding as s2a

    N, f = 256, np.float32
    scale = next(x for x in (f(np.log(2)) + f(i) * f(2) ** -25 for i in range(-8, 9)) if f(x) * f(1.4426950408889634) == f(1))
    q, k = torch.zeros(1, N, 2, d), torch.zeros(1, N, 2, d)
    q[..., 0], k[:, 1:, :, 0] = 1, -24
    q, k = q.bfloat16().cuda(), k.bfloat16().cuda()
    _, lse = s2a.s2a_fwd_ex(q, k, k, N, scale=float(scale), n_unshifted=2, shift=0)
    want = np.zeros(N)
    for row in range(N):
        l = [f(0), f(0)]
        for tile in range(row // 128 + 1):
            p = [f(0) if 128 * tile + x > row else f(1) if tile + x == 0 else f(2) ** -24 for x in range(128)]
            for half in range(2):
                chains = [f(0)] * 4
                for pair in range(32):
                    at = 64 * half + 2 * pair
                    chains[pair % 4] = f(chains[pair % 4] + f(p[at] + p[at + 1]))
                l[half] = f(l[half] + f(f(chains[0] + chains[1]) + f(chains[2] + chains[3])))
        want[row] = np.log(np.float64(f(l[0] + l[1])))
    got = lse[0].double().cpu().numpy()
    assert want[-1] > 200 * 2.0 ** -24
    assert np.abs(got - want).max() <= 2e-6 * want.max(), (got[0, :8], want[:8])
