"""M2L on the tensor cores (csrc/lbf_m2l.cu) against the double loop of plans without room
for it, and against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl
from gpu_util import L, dev, host, plan_for, rel_l2, zeros

pytestmark = pytest.mark.gpu


def smallest_plan(monkeypatch, g, **opt):
    """The plan in the smallest workspace it accepts: no stored rows, no tensor-core M2L."""
    full = L.lbf_workspace_size
    for f in np.arange(0.05, 1.0, 0.02):
        with monkeypatch.context() as m:
            m.setattr(L, "lbf_workspace_size", lambda ptr, o: int(full(ptr, o) * f))
            try:
                return plan_for(g, **opt)
            except L.LbfError as e:
                assert e.status == L.LBF_EWORKSPACE
    raise AssertionError("no workspace was accepted")


@pytest.mark.parametrize("p", [4, 7, 8, 15, 22, 23, 24, 30, 31])
@pytest.mark.parametrize("transpose", [0, 1])
def test_m2l_equals_the_double_loop(monkeypatch, p, transpose):
    """The same truncated operator up to rounding at every padding of the 2 (p + 1) reals
    (multiples of 8 and 16, the largest of 64): leaves of at most 1024 nodes but cells of one
    level (max_depth 5), so no W or X box separates the two plans' truncations."""
    rng = np.random.default_rng(p)
    g = wl.star_caps(21, 9, rng.integers(200, 700, 9))
    op = L.LBF_OP_K_ONLY | (L.LBF_OP_TRANSPOSE if transpose else 0)
    v = rng.standard_normal(g.N)
    out = []
    opt = dict(p=p, leaf_size=2, max_depth=5, fmm64=0)
    for plan in (plan_for(g, **opt), smallest_plan(monkeypatch, g, **opt)):
        o = zeros(g.N)
        L.lbf_apply(plan, op, dev(v), o)
        assert L.lbf_sync_status(plan) == L.LBF_OK
        out.append(host(o))
    # W and X boxes of shallower leaves may still differ by truncation: at least the rounding
    # bound, or the truncation of an M2P (ratio 1/2 per term after sqrt 2 growth)
    assert rel_l2(out[0], out[1]) < max(1e-13, 0.8 ** (2 * p))


def test_m2l_many_tiles_against_the_oracle():
    """Thousands of translations: several tiles an offset and a CTA, both directions of the
    operator, sampled against the oracle at an order whose truncation is below the bound."""
    g = wl.star_caps(3, 64, 512)
    plan = plan_for(g, leaf_size=16, p=30, fmm64=0)
    v = np.random.default_rng(1).standard_normal(g.N)
    o = zeros(g.N)
    L.lbf_apply(plan, L.LBF_OP_K_ONLY, dev(v), o)
    rows = np.random.default_rng(2).choice(g.N, 300, replace=False)
    assert rel_l2(host(o)[rows], oracle.apply_rows(g, v, rows, 1)) < 1e-11


@pytest.mark.parametrize("scale", [1e-280, 1.0, 1e280])
def test_m2l_scales_and_non_finite_densities(scale):
    """The integers follow each box's exponent; an infinity or NaN reaches every row."""
    g = wl.star_caps(8, 6, 300)
    plan = plan_for(g, leaf_size=16, fmm64=0)
    v = dev(np.random.default_rng(4).standard_normal(g.N))
    ref, o = zeros(g.N), zeros(g.N)
    L.lbf_apply(plan, L.LBF_OP_K_ONLY, v, ref)
    L.lbf_apply(plan, L.LBF_OP_K_ONLY, v * scale, o)
    assert rel_l2(host(o) / scale, host(ref)) < 1e-14
    for bad in (float("nan"), float("inf")):
        w = v.clone()
        w[17] = bad
        L.lbf_apply(plan, L.LBF_OP_K_ONLY, w, o)
        assert not torch.isfinite(o).any()
