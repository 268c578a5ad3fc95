"""Per-kernel traces of solves: a graph-replayed step leaves no marks, so the steps that are
replayed while kernels are traced are those the header names."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl
from gpu_util import L, dev, plan_for, zeros

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,n,own,graphs,replayed", [
    (8, 100, False, -1, False),      # the default stream
    (8, 100, False, 1, False),
    (8, 100, True, -1, True),        # a stream of its own, few nodes
    (300, 900, True, -1, False),     # and many
    (300, 900, True, 1, True),
])
def test_traced_solves_leave_a_mark_a_step(M, n, own, graphs, replayed):
    g = wl.star_caps(3, M, n)
    plan = plan_for(g, tol=1e-8, graphs=graphs)
    b = dev(oracle.green_sum(g.x, *wl.pair_sources(g, 0, 1)[:2]))
    sigma, a = zeros(g.N), zeros(g.M)
    stream = torch.cuda.Stream() if own else torch.cuda.current_stream()
    stream.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    L.lbf_gmres_solve(plan, b, sigma, a, stream=stream)  # (a step graph kept from an untraced solve)
    ref = sigma.clone()
    L.lbf_profile_reset()
    L.lbf_profile_enable(True)
    try:
        rc, its, _ = L.lbf_gmres_solve(plan, b, sigma, a, stream=stream)
        torch.cuda.synchronize()
        marks = L.lbf_profile_read(L.LBF_KERNEL_UP)[0]
    finally:
        L.lbf_profile_enable(False)
        L.lbf_profile_reset()
    assert rc == L.LBF_OK and torch.equal(sigma, ref)
    assert (marks < its) if replayed else (marks >= its)
