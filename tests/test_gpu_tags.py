"""The tagged words by which the one-launch passes hand expansions on (csrc/lbf_fixed.cuh): the
density's chain and the multiplier potential's share them, at orders of their own, and the
tags come round after 255 launches."""
import numpy as np
import pytest
import torch

import workloads as wl
from gpu_util import L, dev, plan_for, zeros

pytestmark = pytest.mark.gpu
TURN = 255  # launches until a tag comes again


def _plan():
    """600 islands: E y through the chain (too many for a stored E), 32 terms; the density 27."""
    g = wl.star_caps(7, 600, 33)
    return g, plan_for(g, p=26, leaf_size=24)


def test_a_chain_leaves_no_word_of_an_earlier_launch(monkeypatch):
    """After a whole application (a chain of each kind) and one of the density alone, all 64
    words of every box with children carry the last chain's tag, the third (in a workspace of
    zeros, without another plan's words)."""
    monkeypatch.setattr(L, "_allocate", lambda sizes, d: torch.zeros(sizes[0], dtype=torch.uint8, device=d))
    g, plan = _plan()
    v = dev(np.random.default_rng(1).standard_normal(g.N + g.M))
    o = zeros(g.N + g.M)
    L.lbf_apply(plan, L.LBF_OP_FULL, v, o)
    L.lbf_apply(plan, L.LBF_OP_K_ONLY, v[:g.N].contiguous(), o[:g.N].contiguous())
    assert L.lbf_sync_status(plan) == L.LBF_OK
    parents = int((L.lbf_tree_export(plan)[1][:, 5] > 0).sum())
    found = []
    for phase in (0, 256):  # a box's words are 512 bytes at a multiple of 256
        ws = plan.workspace[phase:]
        words = ws[:len(ws) // 512 * 512].view(torch.int64).view(-1, 64)
        top = (words >> 56) & 0xff
        found.append(top[(top[:, :54] == 3).all(dim=1)])
    found = max(found, key=len)
    assert len(found) == parents
    assert bool((found == 3).all())


@pytest.mark.parametrize("between", [TURN - 3, TURN - 2, TURN - 1, 2 * TURN - 2])
def test_applications_across_the_turn_of_the_tags(between):
    """A whole application, then so many of the density alone that the next chain of 32 terms
    has the tag of the last one (TURN - 2 of them) or one beside it: bit for bit a fresh plan's."""
    g, plan = _plan()
    rng = np.random.default_rng(between)
    u, v = (dev(rng.standard_normal(g.N + g.M)) for _ in range(2))
    o, k, ref = zeros(g.N + g.M), zeros(g.N), zeros(g.N + g.M)
    L.lbf_apply(plan, L.LBF_OP_FULL, u, o)
    s = u[:g.N].contiguous()
    for _ in range(between):
        L.lbf_apply(plan, L.LBF_OP_K_ONLY, s, k)
    L.lbf_apply(plan, L.LBF_OP_FULL, v, o)
    assert L.lbf_sync_status(plan) == L.LBF_OK
    L.lbf_apply(_plan()[1], L.LBF_OP_FULL, v, ref)
    assert torch.equal(o, ref)
