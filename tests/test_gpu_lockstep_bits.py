"""lbf_gmres_solve_many against separate solves, bit for bit, where the lockstep group is large
enough to take its stored rows another way than a separate solve does (csrc/lbf_rows.cu)."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_util import L, dev, host, plan_for, zeros

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [L.LBF_PRECISION_FP64, L.LBF_PRECISION_FP32_REFINE])
@pytest.mark.parametrize("fmm64", [0, 1])
@pytest.mark.parametrize("nrhs", [3, 16])  # too few right-hand sides to fill the chip, and enough
def test_lockstep_bits(nrhs, fmm64, precision):
    """10,000 nodes: about 1300 row blocks of eight rows, 64 warps an SM from eight right-hand
    sides on.  sigma, a, iterations and residuals equal those of separate solves."""
    rng = np.random.default_rng(nrhs)
    g = wl.star_caps(31, 24, np.rint(np.exp(rng.uniform(np.log(64), np.log(1021), 24))).astype(int))
    data = np.stack([oracle.green_sum(g.x, *wl.random_pair_sources(g, rng)[:2]) for _ in range(nrhs)])
    p = plan_for(g, tol=1e-11, fmm64=fmm64, precision=precision)
    sig, a = zeros(nrhs * g.N), zeros(nrhs * g.M)
    rc, its, rr = L.lbf_gmres_solve_many(p, dev(data), sig, a)
    assert rc == L.LBF_OK
    sig, a = host(sig).reshape(nrhs, -1), host(a).reshape(nrhs, -1)
    for k in range(nrhs):
        s1, a1 = zeros(g.N), zeros(g.M)
        rc, it, r1 = L.lbf_gmres_solve(p, dev(data[k]), s1, a1)
        assert rc == L.LBF_OK and (its[k], rr[k]) == (it, r1)
        assert np.array_equal(sig[k], host(s1)) and np.array_equal(a[k], host(a1))
