"""The tensor-core translations alone (csrc/lbf_m2l.cu): a geometry in which they are all there is
between islands, and whose truncation is nothing."""
import numpy as np
import pytest

from gpu_util import L, dev, host, zeros

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53
LD, CLD = np.longdouble, np.clongdouble


def _cells():
    """One circle of 40 nodes about the centre of each of 4 x 4 unit cells (radius a fifth of the
    cell's half-width: expansions of 23 terms and more leave 0.1^23), and circles of eight in
    two corners, which make the cells the quadtree's leaves."""
    mid = [(0.5 + i % 4) + 1j * (0.5 + i // 4) for i in range(16)]
    c, r, n = mid + [0.001 + 0.001j, 3.999 + 3.999j], [0.1] * 16 + [0.001] * 2, [40] * 16 + [8] * 2
    t = [2 * np.pi * np.arange(m) / m for m in n]
    z = [np.stack([m + q * np.exp(1j * s), 1j * q * np.exp(1j * s), -q * np.exp(1j * s)])
         for m, q, s in zip(c, r, t)]
    z = np.concatenate(z, axis=1)
    c = np.array(c)
    a = abs(c) ** 2
    centres = np.stack([2 * c.real / (1 + a), 2 * c.imag / (1 + a), (a - 1) / (1 + a)], axis=1)
    ptr = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
    return ptr, z, centres


@pytest.mark.parametrize("p", [22, 26, 30, 31])
def test_translations_to_less_than_a_double_s_rounding(p):
    """A density on one island at a time, the rows of the islands that are not its neighbours, in
    extended precision; what a density's rows have in common (the rounding of the sphere
    correction's sum) is taken out as the median of the islands' means.  Rms over all offsets in
    units of 2^-53 sum |q| / distance: the rounding of the charges, of the local expansion's
    entries and of the row itself make 0.36, translations whose operands are rounded at 2^-54
    0.13, together 0.38; without the digit products of place 7 the translations make 0.6."""
    ptr, z, centres = _cells()
    N = int(ptr[-1])
    pl = [np.stack([v.real, v.imag], axis=1) for v in z]
    plan = L.lbf_plan_create_planar(ptr, *(dev(v) for v in pl), dev(centres),
                                    opt=L.lbf_default_options(border=0, p=p, leaf_size=48))
    level = host(L.lbf_tree_export(plan)[1])[:, 0]
    assert len(level) == 21 and level.max() == 2
    h = np.repeat(2 * np.pi / np.diff(ptr), np.diff(ptr))
    xi, w = z[0].astype(CLD), (h * z[1]).astype(CLD)
    pi = LD("3.14159265358979323846264338327950288")
    beta = -(xi.conj() * w).imag / (2 * pi * (1 + abs(xi) ** 2))
    rng = np.random.default_rng(100 + p)
    out = []
    for k in list(range(16)) * 3:
        s = np.zeros(N)
        s[ptr[k]:ptr[k + 1]] = rng.standard_normal(40)
        o = zeros(N)
        L.lbf_apply(plan, L.LBF_OP_K_ONLY, dev(s), o)
        o = host(o).astype(LD)
        q = (w * s.astype(LD))[ptr[k]:ptr[k + 1]]
        src, sphere = xi[ptr[k]:ptr[k + 1]], 2 * (beta * s.astype(LD)).sum()
        err, size = [], []
        for j in range(16):
            dx, dy = j % 4 - k % 4, j // 4 - k // 4
            if max(abs(dx), abs(dy)) < 2:
                continue
            at = xi[ptr[j]:ptr[j + 1]]
            ref = (q[None, :] / (src[None, :] - at[:, None])).imag.sum(axis=1) / pi + sphere
            err.append((o[ptr[j]:ptr[j + 1]] - ref).astype(float))
            size.append(float(abs(q).sum()) / abs(dx + 1j * dy) / np.pi)
        common = np.median([e.mean() for e in err])
        out += [(e - common) / t for e, t in zip(err, size)]
    assert np.sqrt(np.mean(np.concatenate(out) ** 2)) < 0.45 * EPS
