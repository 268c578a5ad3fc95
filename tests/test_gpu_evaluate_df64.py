"""Evaluation on default plans (fmm64 = 1) whose multipoles do not come from the stored parts: an
order above theirs, and workspaces without them."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_util import L, dev, host, plan_for, rel_l2, zeros

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rung", [0, 1, 4])
@pytest.mark.parametrize("p", [26, 31, 32, 44])
def test_evaluation_in_double_float_multipoles(monkeypatch, p, rung):
    """Enough targets for the walk; against the oracle, and no kernel of the double upward pass
    where double-float is the plan's arithmetic: the launch before the walk is the widening of
    its multipoles."""
    g = wl.star_caps(9, 40, 200)
    t = wl.targets_off_islands(g, 3000, seed=2)
    rng = np.random.default_rng(p)
    sigma, a = rng.standard_normal(g.N), rng.standard_normal(g.M)
    a -= a.mean()
    sizes = L.lbf_workspace_sizes
    monkeypatch.setattr(L, "lbf_workspace_size", lambda ptr, o: sizes(ptr, o)[rung])
    u, count = {}, {}
    for fmm64 in (0, 1):
        plan = plan_for(g, p=p, fmm64=fmm64)
        u[fmm64] = zeros(len(t))
        n = L.lbf_launch_count()
        L.lbf_evaluate(plan, dev(sigma), dev(a), dev(t), u[fmm64])
        count[fmm64] = L.lbf_launch_count() - n
        assert L.lbf_sync_status(plan) == L.LBF_OK
        ref = oracle.evaluate(g, sigma, a, t)
        assert rel_l2(host(u[fmm64]), ref) < 1e-10
    stored = rung == 0 and p <= 31
    assert count[1] == count[0] + (0 if stored else 1)
