"""Off-curve targets: the pair sums and the tree walk of the evaluation (csrc/lbf_evaluate.cu),
and the sums over targets at the nodes of its adjoint (csrc/lbf_adjoint.cu), against dense
matrices, on both sides of the pair count that divides them (2^24)."""
import numpy as np
import pytest
import torch

import workloads as wl
from gpu_util import L, dev, host, plan_for, rel_l2, zeros
from oracle import adjoint as oadj

pytestmark = pytest.mark.gpu


def spread_targets(g, T, seed):
    """Targets anywhere off the curves, islands included (the sums do not care), among them
    the projection pole."""
    rng = np.random.default_rng(seed)
    t = rng.standard_normal((T, 3))
    t /= np.linalg.norm(t, axis=1, keepdims=True)
    t[T // 2] = (0.0, 0.0, 1.0)
    return t


def dense(g, t):
    c = np.vstack([oadj.evaluation_matrix(g.island_ptr, g.x, g.dx, g.centres, b)
                   for b in np.array_split(t, max(1, len(t) // 300))])
    return c


@pytest.mark.parametrize("T", [1, 5, 2040])
def test_pair_sums_against_the_dense_matrix(T):
    g = wl.config_geometry("C2")  # 8192 nodes: 2048 targets are 2^24 pairs
    plan = plan_for(g, p=30)
    t = spread_targets(g, T, T)
    C = dense(g, t)
    rng = np.random.default_rng(T + 1)
    z = rng.standard_normal(g.N + g.M)
    z[g.N:] -= z[g.N:].mean()  # a target at the pole sees a_m G with sum a = 0
    u = zeros(T)
    L.lbf_evaluate(plan, dev(z[:g.N]), dev(z[g.N:]), dev(t), u)
    # the rounding of sums of 8192 terms
    assert np.max(np.abs(host(u) - C @ z)) < 1e-12 * np.max(np.abs(C) @ np.abs(z))
    ub = rng.standard_normal(T)
    sbar, abar = zeros(g.N), zeros(g.M)
    L.lbf_evaluate_transpose(plan, dev(t), dev(ub), sbar, abar)
    ref, bound = C.T @ ub, np.abs(C.T) @ np.abs(ub)
    assert np.max(np.abs(host(sbar) - ref[:g.N])) < 1e-12 * np.max(bound[:g.N])
    assert np.max(np.abs(host(abar) - ref[g.N:])) < 1e-12 * np.max(bound[g.N:])


@pytest.mark.parametrize("T,leaf,depth", [(2060, 48, 30), (2500, 3, 30), (2500, 48, 3)])
def test_tree_walk_equals_the_pair_sums(T, leaf, depth):
    """Above 2^24 pairs the walk and the targets' expansions, below them the pairs: one call
    over all targets against calls over two halves.  Both take the same node-target
    differences, so what is left is truncation (3^-31, (sqrt 2/3)^48) and the rounding of the
    sums, relative to the sums of magnitudes."""
    g = wl.config_geometry("C2")
    plan = plan_for(g, leaf_size=leaf, max_depth=depth, p=30)
    t = spread_targets(g, T, T)
    C = dense(g, t)
    rng = np.random.default_rng(T + 1)
    z = rng.standard_normal(g.N + g.M)
    z[g.N:] -= z[g.N:].mean()
    ub = rng.standard_normal(T)
    half = T // 2
    whole, parts = zeros(T), zeros(T)
    sig, a = dev(z[:g.N]), dev(z[g.N:])
    L.lbf_evaluate(plan, sig, a, dev(t), whole)
    assert L.lbf_sync_status(plan) == L.LBF_OK
    L.lbf_evaluate(plan, sig, a, dev(t[:half]), parts[:half])
    L.lbf_evaluate(plan, sig, a, dev(t[half:]), parts[half:])
    assert np.max(np.abs(host(whole) - host(parts)) / (np.abs(C) @ np.abs(z))) < 1e-12
    out = []
    for sel in (slice(0, T), slice(0, half), slice(half, T)):
        sbar, abar = zeros(g.N), zeros(g.M)
        L.lbf_evaluate_transpose(plan, dev(t[sel]), dev(ub[sel]), sbar, abar)
        out.append(host(sbar))
    bound = np.abs(C[:, :g.N].T) @ np.abs(ub)
    assert np.max(np.abs(out[0] - out[1] - out[2])) < 1e-12 * np.max(bound)


def test_gradient_over_many_targets_is_the_sum_over_parts():
    """grad is affine in the targets' weights: all 4000 targets at once (by the tree) against
    two halves (pair by pair) less the part without targets."""
    g = wl.config_geometry("C2")
    plan = plan_for(g, p=30)
    t = wl.targets_off_islands(g, 4000, seed=3)
    rng = np.random.default_rng(5)
    sig, a, lam = (dev(rng.standard_normal(n)) for n in (g.N, g.M, g.N + g.M))
    ub = rng.standard_normal(4000)

    def grad(sel):
        o = zeros(2 * g.N)
        w = np.zeros(len(sel)) if sel.dtype == bool else ub[sel]
        tt = t[:len(sel)] if sel.dtype == bool else t[sel]
        L.lbf_gradient_nodes(plan, sig, a, lam, dev(tt), dev(w), o)
        return host(o)

    whole = grad(np.arange(4000))
    parts = grad(np.arange(2000)) + grad(np.arange(2000, 4000)) - grad(np.zeros(1, dtype=bool))
    assert rel_l2(whole, parts) < 1e-12
