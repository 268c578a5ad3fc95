"""Stored leaf rows of the accurate forward operator (csrc/lbf_rows.cu): plans with and
without room for them, against the oracle, where the tiles' edges fall differently."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl
from gpu_util import L, dev, host, plan_for, rel_l2, zeros

pytestmark = pytest.mark.gpu
# the operator's own bound at these orders (p >= 24: truncation below 2e-12; rounding far less)
TOL = 1e-10


def short_plan(monkeypatch, g, **opt):
    """The same plan in a workspace without room for the rows (they come last in it)."""
    full = L.lbf_workspace_size
    with monkeypatch.context() as m:
        m.setattr(L, "lbf_workspace_size", lambda ptr, o: full(ptr, o) - 1024)
        return plan_for(g, **opt)


@pytest.mark.parametrize("fmm64", [0, 1])
@pytest.mark.parametrize("leaf,p,depth", [
    (1, 24, 30),     # one row a leaf, many chunks
    (5, 26, 30),     # two row groups, the second with one row
    (33, 35, 30),    # a leaf of more than 32 rows: two blocks where whole leaves go to a warp
    (48, 63, 30),    # the most local columns
    (1024, 26, 30),  # one or few leaves: every node a column of every row
    (4, 26, 4),      # depth-capped leaves
])
def test_rows_against_the_oracle_and_the_unstored_rows(monkeypatch, leaf, p, depth, fmm64):
    g = wl.star_caps(11, 5, np.array([64, 37, 201, 90, 333]))
    v = np.random.default_rng(leaf).standard_normal(g.N + g.M)
    ref = oracle.apply(g, v, 0)
    opt = dict(leaf_size=leaf, p=p, max_depth=depth, fmm64=fmm64)
    out = []
    for plan in (plan_for(g, **opt), short_plan(monkeypatch, g, **opt)):
        o = zeros(g.N + g.M)
        L.lbf_apply(plan, L.LBF_OP_FULL, dev(v), o)
        assert L.lbf_sync_status(plan) == L.LBF_OK
        assert rel_l2(host(o), ref) < TOL
        out.append(o)
    assert rel_l2(host(out[0]), host(out[1])) < TOL


def test_rows_of_whole_leaves_and_large_w_boxes():
    """Leaves enough for a warp each (not shared by a thread block), with W boxes of more
    than 4 (p + 1) nodes, whose M2P rows are columns: sampled rows against the oracle."""
    g = wl.star_caps(3, 64, np.where(np.arange(64) % 8 == 0, 4096, 300))
    plan = plan_for(g, leaf_size=8, p=26)
    assert L.lbf_plan_info(plan)["nleaf"] > 4864
    v = np.random.default_rng(1).standard_normal(g.N + g.M)
    o = zeros(g.N + g.M)
    L.lbf_apply(plan, L.LBF_OP_FULL, dev(v), o)
    rows = np.random.default_rng(2).choice(g.N, 400, replace=False)
    assert rel_l2(host(o)[rows], oracle.apply_rows(g, v, rows, 0)) < TOL


def test_rows_repeat_and_zero_weights():
    """Two applications agree bit for bit; a zero density gives zero rows."""
    g = wl.star_caps(5, 7, 129)
    plan = plan_for(g)
    v = dev(np.random.default_rng(3).standard_normal(g.N))
    a, b, z = zeros(g.N), zeros(g.N), torch.full((g.N,), 1.0, dtype=torch.float64, device=v.device)
    L.lbf_apply(plan, L.LBF_OP_K_ONLY, v, a)
    L.lbf_apply(plan, L.LBF_OP_K_ONLY, v, b)
    L.lbf_apply(plan, L.LBF_OP_K_ONLY, zeros(g.N), z)
    assert torch.equal(a, b) and torch.count_nonzero(z) == 0


@pytest.mark.parametrize("fmm64", [0, 1])
@pytest.mark.parametrize("leaf,p,depth", [(1, 24, 30), (5, 26, 30), (33, 35, 30), (48, 63, 30),
                                          (1024, 26, 30), (4, 26, 4)])
def test_transposed_rows_against_the_oracle_and_the_unstored_rows(monkeypatch, leaf, p, depth, fmm64):
    g = wl.star_caps(11, 5, np.array([64, 37, 201, 90, 333]))
    v = np.random.default_rng(leaf).standard_normal(g.N + g.M)
    ref = oracle.matrix(g).T @ v
    opt = dict(leaf_size=leaf, p=p, max_depth=depth, fmm64=fmm64)
    for plan in (plan_for(g, **opt), short_plan(monkeypatch, g, **opt)):
        o = zeros(g.N + g.M)
        L.lbf_apply(plan, L.LBF_OP_FULL | L.LBF_OP_TRANSPOSE, dev(v), o)
        assert L.lbf_sync_status(plan) == L.LBF_OK
        assert rel_l2(host(o), ref) < TOL


def test_transposed_rows_of_whole_leaves_and_large_w_boxes():
    """<K x, y> = <x, K^T y> where whole leaves go to a warp, some boxes' M2P rows are columns
    and leaves of more than 32 rows have two blocks."""
    g = wl.star_caps(3, 64, np.where(np.arange(64) % 8 == 0, 4096, 300))
    for leaf in (8, 40):
        plan = plan_for(g, leaf_size=leaf, p=26, border=0)
        rng = np.random.default_rng(leaf)
        x, y = dev(rng.standard_normal(g.N)), dev(rng.standard_normal(g.N))
        kx, ky = zeros(g.N), zeros(g.N)
        L.lbf_apply(plan, L.LBF_OP_K_ONLY, x, kx)
        L.lbf_apply(plan, L.LBF_OP_K_ONLY | L.LBF_OP_TRANSPOSE, y, ky)
        assert abs(float(kx @ y - x @ ky)) < TOL * float(kx.norm() * y.norm())


@pytest.mark.parametrize("M,nodes", [(1, 40), (7, 33), (8, 32), (33, 48), (129, 40)])
def test_stored_multiplier_block_both_ways(M, nodes):
    """E y and E^T tau where the chunks of eight centres and blocks of 32 nodes end differently:
    entries to the rounding of a logarithm, sums of at most 5,160 of them."""
    g = wl.star_caps(17, M, nodes)
    plan = plan_for(g, p=30)
    rng = np.random.default_rng(M)
    E = oracle.matrix(g)[:g.N, g.N:]
    v = np.concatenate([np.zeros(g.N), rng.standard_normal(g.M)])
    o = zeros(g.N + g.M)
    L.lbf_apply(plan, L.LBF_OP_FULL, dev(v), o)
    assert rel_l2(host(o)[:g.N], E @ v[g.N:]) < 1e-13
    tau = rng.standard_normal(g.N)
    L.lbf_apply(plan, L.LBF_OP_FULL | L.LBF_OP_TRANSPOSE, dev(np.concatenate([tau, np.zeros(g.M)])), o)
    assert rel_l2(host(o)[g.N:], E.T @ tau) < 1e-13 * np.sqrt(g.N)


@pytest.mark.parametrize("op", [L.LBF_OP_K_ONLY, L.LBF_OP_K_ONLY | L.LBF_OP_TRANSPOSE])
@pytest.mark.parametrize("leaf", [8, 300])
def test_integer_rows_keep_scale_and_non_finite_values(leaf, op):
    """The densities' integers are relative to the largest: a power of two comes out exactly
    (no step rounds differently), and a value that is not finite reaches every row (through
    the sum over all nodes that each row holds)."""
    g = wl.star_caps(11, 5, np.array([64, 37, 201, 90, 333]))
    plan = plan_for(g, leaf_size=leaf, p=30, border=0)
    v = dev(np.random.default_rng(leaf).standard_normal(g.N))
    o, p = zeros(g.N), zeros(g.N)
    L.lbf_apply(plan, op, v, o)
    for k in (-800, -1, 800):
        L.lbf_apply(plan, op, v * 2.0 ** k, p)
        assert torch.equal(p * 2.0 ** -k, o)
    for bad in (float("nan"), float("inf")):
        w = v.clone()
        w[g.N // 2] = bad
        L.lbf_apply(plan, op, w, p)
        assert not torch.isfinite(p).any()


def test_passes_where_a_warp_takes_several_leaves():
    """More than 16 leaves and boxes for every warp of the upward pass: sampled rows."""
    g = wl.star_caps(5, 1024, 400)
    plan = plan_for(g, leaf_size=8, p=26, border=0)
    assert L.lbf_plan_info(plan)["nleaf"] > 80000
    v = np.random.default_rng(6).standard_normal(g.N)
    o = zeros(g.N)
    L.lbf_apply(plan, L.LBF_OP_K_ONLY, dev(v), o)
    rows = np.random.default_rng(7).choice(g.N, 60, replace=False)
    assert rel_l2(host(o)[rows], oracle.apply_rows(g, np.concatenate([v, np.zeros(g.M)]), rows, 0)) < TOL


@pytest.mark.parametrize("p", [22, 35])  # fewer, more local columns than the multipliers' terms
@pytest.mark.parametrize("leaf", [3, 48, 200])
def test_multiplier_potential_through_the_local_columns(leaf, p):
    """E y of 600 islands (too many for a stored E) at sampled nodes; the expansions' 32 terms
    are worth 1e-12."""
    g = wl.star_caps(7, 600, 33)
    plan = plan_for(g, leaf_size=leaf, p=p)
    v = np.concatenate([np.zeros(g.N), np.random.default_rng(leaf).standard_normal(g.M)])
    o = zeros(g.N + g.M)
    L.lbf_apply(plan, L.LBF_OP_FULL, dev(v), o)
    rows = np.random.default_rng(8).choice(g.N, 100, replace=False)
    assert rel_l2(host(o)[rows], oracle.apply_rows(g, v, rows, 0)) < TOL
