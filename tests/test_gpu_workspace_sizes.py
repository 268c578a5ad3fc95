"""Plans and batch items in workspaces without some or all of the stored parts, and a batch in
one shared workspace."""
import ctypes as C

import numpy as np
import pytest
import torch

import oracle
import workloads as wl
from gpu_util import L, dev, host, plan_for, rel_l2, zeros

pytestmark = pytest.mark.gpu
PARTS = [15, 7, 3, 1, 0]


@pytest.mark.parametrize("fmm64", [0, 1])
@pytest.mark.parametrize("rung", range(5))
@pytest.mark.parametrize("M", [40, 600])  # E stored; (box, centre) pairs
def test_a_plan_holds_the_parts_its_workspace_has_room_for(monkeypatch, M, rung, fmm64):
    g = wl.star_caps(5, M, 33)
    sizes = L.lbf_workspace_sizes
    monkeypatch.setattr(L, "lbf_workspace_size", lambda ptr, o: sizes(ptr, o)[rung])
    plan = plan_for(g, p=30, fmm64=fmm64)
    has = L.LBF_PART_E if M <= 512 else L.LBF_PART_PAIRS
    assert L.lbf_plan_parts(plan) == PARTS[rung] & (L.LBF_PART_M2L | L.LBF_PART_ROWS | has)
    v = np.random.default_rng(rung).standard_normal(g.N + g.M)
    rows = np.random.default_rng(1).choice(g.N, 100, replace=False)
    o = zeros(g.N + g.M)
    L.lbf_apply(plan, L.LBF_OP_FULL, dev(v), o)
    assert L.lbf_sync_status(plan) == L.LBF_OK
    assert rel_l2(host(o)[rows], oracle.apply_rows(g, v, rows, 0)) < 1e-10


def test_a_plan_asked_to_store_nothing():
    g = wl.star_caps(5, 40, 33)
    args = (g.island_ptr, dev(g.x), dev(g.dx), dev(g.d2x), dev(g.centres))
    assert L.lbf_plan_parts(L.lbf_plan_create(*args, stored=False)) == 0
    assert L.lbf_plan_parts(L.lbf_plan_create(*args)) == 11


def _instances(nrhs):
    out = []
    for k, M in enumerate((3, 9, 1, 6, 14, 2, 5)):
        g = wl.star_caps(50 + k, M, 90 + 10 * k)
        rng = np.random.default_rng(k)
        data = np.stack([oracle.green_sum(g.x, *wl.random_pair_sources(g, rng)[:2]) for _ in range(nrhs)])
        out.append(dict(island_ptr=g.island_ptr, x=dev(g.x), dx=dev(g.dx), d2x=dev(g.d2x),
                        centres=dev(g.centres), g=dev(data)))
    return out


@pytest.mark.parametrize("rung", range(5))
def test_batch_items_of_every_size_run_in_lockstep(monkeypatch, rung):
    """Two workers and seven instances in one workspace: densities as from separate plans to the
    solver's tolerance, and fewer than half the launches of one right-hand side after another."""
    inst, opt = _instances(8), L.lbf_default_options(tol=1e-12, graphs=0)
    sizes = L.lbf_workspace_sizes
    launches = []
    for lock in (True, False):
        with monkeypatch.context() as m:
            m.setattr(L, "lbf_workspace_sizes", lambda p, o, n=0: [sizes(p, o, n)[rung]] * 5)
            n0 = L.lbf_launch_count()
            res = L.lbf_batch_run(inst, opt=opt, nworkers=2, lockstep=lock)
            launches.append(L.lbf_launch_count() - n0)
        for ins, r in zip(inst, res):
            assert r["status"] == L.LBF_OK and r["max_rel_res"] <= 1e-12
            p = L.lbf_plan_create(ins["island_ptr"], ins["x"], ins["dx"], ins["d2x"], ins["centres"], opt=opt)
            for k in (0, 7):
                sig, a = zeros(p.N), zeros(p.M)
                L.lbf_gmres_solve(p, ins["g"].view(8, -1)[k].contiguous(), sig, a)
                assert rel_l2(host(r["sigma"][k]), host(sig)) < 1e-9
    assert 2 * launches[0] < launches[1]


def test_shared_workspace_gives_what_own_workspaces_give():
    """Bit for bit, with more workers than items and fewer; a short workspace is refused."""
    inst, opt = _instances(3), L.lbf_default_options(tol=1e-12)
    lib = L.load()
    items = (L.lbf_batch_item * len(inst))()
    keep = []
    for it, ins in zip(items, inst):
        ptr = np.ascontiguousarray(ins["island_ptr"], dtype=np.int64)
        M, N = len(ptr) - 1, int(ptr[-1])
        sig, a = zeros(3 * N), zeros(3 * M)
        it.M, it.island_ptr, it.nrhs = M, ptr.ctypes.data, 3
        for name in ("x", "dx", "d2x", "centres", "g"):
            setattr(it, name, ins[name].data_ptr())
        it.sigma, it.a = sig.data_ptr(), a.data_ptr()
        it.bytes = L.lbf_batch_workspace_size(ptr, opt, 3)
        ws = torch.empty(it.bytes, dtype=torch.uint8, device=sig.device)
        it.workspace = ws.data_ptr()
        keep.append((ptr, sig, a, ws))
    assert lib.lbf_batch_run(len(inst), items, C.byref(opt), 3) == L.LBF_OK
    torch.cuda.synchronize()
    own = [(host(s).copy(), host(a).copy(), it.iters) for (_, s, a, _), it in zip(keep, items)]
    for workers in (1, 3, 20):
        total = C.c_size_t(0)
        assert lib.lbf_batch_shared_size(len(inst), items, workers, C.byref(total)) == L.LBF_OK
        ws = torch.empty(total.value, dtype=torch.uint8, device="cuda")
        for _, s, a, _ in keep:
            s.zero_()
            a.zero_()
        torch.cuda.synchronize()
        run = lambda n: lib.lbf_batch_run_shared(len(inst), items, C.byref(opt), workers,  # noqa: E731
                                                 C.c_void_p(ws.data_ptr()), n)
        assert run(total.value - 512) == L.LBF_EWORKSPACE
        assert run(total.value) == L.LBF_OK
        torch.cuda.synchronize()
        for (_, s, a, _), it, (s0, a0, n) in zip(keep, items, own):
            assert it.status == L.LBF_OK and it.iters == n
            assert np.array_equal(host(s), s0) and np.array_equal(host(a), a0)


def test_batch_waits_for_its_inputs():
    """Data still being written on the caller's stream (behind a wait of about 50 ms) when the batch
    is called: its own streams read them after that."""
    inst, opt = _instances(2), L.lbf_default_options(tol=1e-12)
    ref = [host(r["sigma"]) for r in L.lbf_batch_run(inst, opt=opt, nworkers=4)]
    data = [ins["g"].clone() for ins in inst]
    for ins in inst:
        ins["g"] = torch.zeros_like(ins["g"])
    torch.cuda.synchronize()
    torch.cuda._sleep(100_000_000)
    for ins, d in zip(inst, data):
        ins["g"].copy_(d)
    res = L.lbf_batch_run(inst, opt=opt, nworkers=4)
    for r, s in zip(res, ref):
        assert np.array_equal(host(r["sigma"]), s)
