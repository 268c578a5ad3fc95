"""Stored rows (csrc/lbf_rows.cu) where densities or entries of very different size meet: what
their integers' common units may cost, against the sizes of a row's own terms."""
import numpy as np
import pytest

from gpu_util import L, dev, host, zeros

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def circles(parts, gap):
    """Planar circles, parts = (x, nodes): island 0 at the origin, the others of radius 0.1 in a
    row from x on, gap node spacings apart; island_ptr, xi, xi', xi'', sphere centres."""
    c, r, n = [0.0], [0.05], [parts[0][1]]
    for x, m in parts[1:]:
        c.append(x if len(c) == 1 else c[-1] + 0.2 + gap * 2 * np.pi * 0.1 / m)
        r.append(0.1)
        n.append(m)
    t = [2 * np.pi * np.arange(m) / m for m in n]
    z = [np.stack([x + q * np.exp(1j * s), 1j * q * np.exp(1j * s), -q * np.exp(1j * s)])
         for x, q, s in zip(c, r, t)]
    z = np.concatenate(z, axis=1)
    x = np.array(c)
    centres = np.stack([2 * x / (1 + x * x), 0 * x, (x * x - 1) / (1 + x * x)], axis=1)
    ptr = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
    return ptr, [np.stack([v.real, v.imag], axis=1) for v in z], centres


def plan_of(ptr, z, centres, **opt):
    return L.lbf_plan_create_planar(ptr, *(dev(v) for v in z), dev(centres),
                                    opt=L.lbf_default_options(border=0, **opt))


def row_sizes(ptr, z, density, rows):
    """sum_j |2 K_ij density_j| (the off-diagonal ones) of the rows given."""
    xi, d = (v[:, 0] + 1j * v[:, 1] for v in z[:2])
    w = d * np.repeat(2 * np.pi / np.diff(ptr), np.diff(ptr))
    out = []
    for i in rows:
        dz = xi - xi[i]
        dz[i] = 1.0
        k = np.abs((w / dz).imag) / np.pi
        k[i] = 0.0
        out.append(k @ np.abs(density))
    return np.array(out)


@pytest.mark.parametrize("leaf,nodes", [(64, 128), (16, 60000)])  # leaves shared by warps; a warp each
@pytest.mark.parametrize("fmm64", [0, 1])
def test_a_far_large_density_costs_small_rows_nothing(fmm64, leaf, nodes):
    """Two islands a millionth of a node spacing apart (entries of 3e5) with densities of 1e-9, a
    third at a distance with densities of 1.  Rows of the two are linear in the density to the
    rounding of their own terms: 27 coefficients over at most 30 levels."""
    ptr, z, centres = circles([(0, 64), (1.0, nodes), (0, nodes)], 1e-6)
    plan = plan_of(ptr, z, centres, leaf_size=leaf, p=26, fmm64=fmm64)
    assert (L.lbf_plan_info(plan)["nleaf"] > 4864) == (leaf == 16)
    rng = np.random.default_rng(leaf)
    N, far = int(ptr[-1]), int(ptr[1])
    big, small = rng.standard_normal(N), 2.0 ** -30 * rng.standard_normal(N)
    big[far:] = 0.0
    small[:far] = 0.0
    out = []
    for d in (big, small, big + small):
        o = zeros(N)
        L.lbf_apply(plan, L.LBF_OP_K_ONLY, dev(d), o)
        assert L.lbf_sync_status(plan) == L.LBF_OK
        out.append(host(o))
    rows = far + rng.choice(N - far, min(500, N - far), replace=False)
    rows = np.concatenate([rows, [far, int(ptr[2])]])
    # the two nodes that all but meet
    rows = np.unique(np.concatenate([rows, [int(ptr[2]) + nodes // 2]]))
    err = np.abs(out[2] - out[0] - out[1])[rows]
    assert np.all(err <= 27 * 30 * EPS * row_sizes(ptr, z, big + small, rows))


@pytest.mark.parametrize("gap", [1.0, 0.1, 1e-3, 1e-6])
@pytest.mark.parametrize("fmm64", [0, 1])
def test_transposed_rows_beside_islands_that_touch(fmm64, gap):
    """Transposed rows of islands from a node spacing to a millionth of one apart, all pairs near
    (one leaf), against the direct sums: every node but the two that meet has the error that
    coordinates rounded to 2^-53 of the box's half-width (0.68) make at the node spacing, however
    large the entries of the rows that meet."""
    nodes = 200
    ptr, z, centres = circles([(0, 64), (1.0, nodes), (0, nodes)], gap)
    N = int(ptr[-1])
    v = np.random.default_rng(5).standard_normal(N)
    out = []
    for matvec in (L.LBF_MATVEC_FMM, L.LBF_MATVEC_DIRECT):
        plan = plan_of(ptr, z, centres, leaf_size=1024, p=26, fmm64=fmm64, matvec=matvec)
        o = zeros(N)
        L.lbf_apply(plan, L.LBF_OP_K_ONLY | L.LBF_OP_TRANSPOSE, dev(v), o)
        assert L.lbf_sync_status(plan) == L.LBF_OK
        out.append(host(o))
    rest = np.ones(N, dtype=bool)
    rest[[int(ptr[1]), int(ptr[2]) + nodes // 2]] = False
    xi, d = (a[:, 0] + 1j * a[:, 1] for a in z[:2])
    w = d * np.repeat(2 * np.pi / np.diff(ptr), np.diff(ptr))
    dz = xi[:, None] - xi[None, :] + np.eye(N)
    k = np.abs((w[:, None] / dz).imag) / np.pi * (1 - np.eye(N))
    size = np.abs(v) + k @ np.abs(v)
    bound = 4 * 0.68 / (2 * np.pi * 0.1 / nodes) * EPS * size
    assert np.all(np.abs(out[0] - out[1])[rest] <= bound[rest])
