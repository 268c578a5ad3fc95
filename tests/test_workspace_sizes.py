"""Workspaces with fewer stored parts, and one shared by a batch (host calls; no GPU needed)."""
import ctypes as C

import numpy as np
import pytest
import torch

GB = 10 ** 9


@pytest.fixture(scope="module")
def L():
    from paper_1306_0612_gb300.build import build

    build()
    from paper_1306_0612_gb300 import lbfmm

    return lbfmm


def _ptr(M, n):
    return np.arange(M + 1, dtype=np.int64) * n


@pytest.mark.parametrize("M,n,opt", [(24, 400, {}), (2048, 1024, dict(p=22, fmm64=0)),
                                     (407, 1024, dict(precision=1)), (64, 512, dict(border=0)),
                                     (16, 512, dict(p=40)), (1, 256, dict(matvec=1))])
@pytest.mark.parametrize("nrhs", [0, 16])
def test_sizes_descend_from_the_whole_one(L, M, n, opt, nrhs):
    o = L.lbf_default_options(**opt)
    s = L.lbf_workspace_sizes(_ptr(M, n), o, nrhs)
    whole = L.lbf_batch_workspace_size(_ptr(M, n), o, nrhs)
    assert s[0] == whole and all(a >= b for a, b in zip(s, s[1:]))
    if opt.get("matvec") == 1:
        assert s[-1] > 0.9 * s[0]  # direct sums: E at most is stored


def test_the_least_size_holds_a_batch_of_many_uneven_instances(L):
    """512 instances of up to 64 islands, 16 right-hand sides, refined: 132.2 GB with nothing stored
    (before any part was), one workspace for 8 workers a few GB with everything."""
    rng = np.random.default_rng(4)
    o = L.lbf_default_options(precision=1, fmm64=0)
    items = (L.lbf_batch_item * 512)()
    keep, least = [], 0
    for it in items:
        n = np.rint(np.exp(rng.uniform(np.log(64), np.log(1024), rng.integers(1, 65)))).astype(np.int64)
        ptr = np.concatenate([[0], np.cumsum(n)])
        s = L.lbf_workspace_sizes(ptr, o, 16)
        least += s[-1]
        it.M, it.island_ptr, it.nrhs, it.bytes = len(n), ptr.ctypes.data, 16, s[0]
        it.g = it.sigma = 256  # (not read)
        keep.append(ptr)
    assert least < 140 * GB
    total = C.c_size_t(0)
    for workers in (1, 8, 600):
        assert L.load().lbf_batch_shared_size(512, items, workers, C.byref(total)) == L.LBF_OK
        most = max(it.bytes for it in items)
        own = sum(it.bytes for it in items)
        assert most <= total.value <= min(workers * (most + 256), own + 512 * 4096) + 256
    assert L.load().lbf_batch_shared_size(512, items, 0, C.byref(total)) == L.LBF_EINVAL


class _Device:
    def __init__(self, L, monkeypatch, free, total=280 * GB):
        self.free, self.asked = free, []

        def empty(n, dtype=None, device=None):
            self.asked.append(n)
            if n > self.free:
                raise torch.cuda.OutOfMemoryError("no room")
            return n

        cuda = torch.cuda
        monkeypatch.setattr(L.torch, "empty", empty)
        monkeypatch.setattr(cuda, "get_device_properties", lambda d: type("P", (), dict(total_memory=total)))
        monkeypatch.setattr(cuda, "mem_get_info", lambda d: (self.free, total))
        monkeypatch.setattr(cuda, "memory_reserved", lambda d: 0)
        monkeypatch.setattr(cuda, "memory_allocated", lambda d: 0)


def test_allocation_leaves_room_and_takes_the_next_size(L, monkeypatch):
    sizes = [74 * GB, 33 * GB, 30 * GB, 28 * GB, 20 * GB]
    d = _Device(L, monkeypatch, 200 * GB)
    assert L._allocate(sizes, 0) == 74 * GB
    d.free = 80 * GB  # the whole one would fit, and leave the caller 6 GB
    assert L._allocate(sizes, 0) == 33 * GB
    d.free = 25 * GB
    assert L._allocate(sizes, 0) == 20 * GB
    d.free = 10 * GB
    with pytest.raises(torch.cuda.OutOfMemoryError):
        L._allocate(sizes, 0)


def test_allocation_of_small_plans_asks_nothing_first(L, monkeypatch):
    d = _Device(L, monkeypatch, 3 * GB)
    monkeypatch.setattr(torch.cuda, "mem_get_info", None)
    assert L._allocate([2 * GB, GB, GB, GB, GB // 2], 0) == 2 * GB and d.asked == [2 * GB]
    d.free = GB
    assert L._allocate([2 * GB, GB, GB, GB, GB // 2], 0) == GB
