"""Stored rows (csrc/lbf_rows.cu) of a geometry with a self term that is not finite: the integer
entries have no code for it, and its row, and no other, has to say so."""
import numpy as np
import pytest

import workloads as wl
from gpu_util import L, dev, host, plan_for, rel_l2, zeros

pytestmark = pytest.mark.gpu
NODE = 100


@pytest.mark.parametrize("scale", [1.0, 1e-3])
@pytest.mark.parametrize("transpose", [0, L.LBF_OP_TRANSPOSE])
@pytest.mark.parametrize("leaf", [8, 300])
@pytest.mark.parametrize("fmm64", [0, 1])
def test_a_node_where_the_parametrisation_stops(fmm64, leaf, transpose, scale):
    """x' = 0 at one node: its weight is zero and its self term 0/0.  Its own row comes out as NaN,
    every other row as the direct sums give it (p = 30: to 1e-11)."""
    g = wl.star_caps(11, 5, np.array([64, 37, 201, 90, 333]))
    g.dx = g.dx.copy()
    g.dx[NODE] = 0.0
    v = dev(scale * np.random.default_rng(leaf).standard_normal(g.N))
    out = []
    for matvec in (L.LBF_MATVEC_FMM, L.LBF_MATVEC_DIRECT):
        o = zeros(g.N)
        plan = plan_for(g, p=30, leaf_size=leaf, border=0, fmm64=fmm64, matvec=matvec)
        L.lbf_apply(plan, L.LBF_OP_K_ONLY | transpose, v, o)
        assert L.lbf_sync_status(plan) == L.LBF_OK
        out.append(host(o))
    rest = np.arange(g.N) != NODE
    for o in out:
        assert np.isnan(o[NODE]) and np.isfinite(o[rest]).all()
    assert rel_l2(out[0][rest], out[1][rest]) < 1e-11
