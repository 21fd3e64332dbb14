"""Segment lists where memory is short, and what a first guess leaves (GPU)."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.fixture
def scene():
    import paper_1310_1854_gb300 as pkg
    g = gen.make_disk_grid(3000, 111)
    rays = gen.disk_rays(20_000, 112)
    O, D = dev(rays.origin), dev(rays.dir)

    def grid():
        vg = pkg.VoronoiGrid(g.sites, g.box)
        vg.set_density(dev(g.rho))
        return vg

    vg = grid()
    want = vg.trace(O, D, segments=True)
    return pkg, grid, O, D, want


def same(r, q):
    assert torch.equal(r.seg_off, q.seg_off) and torch.equal(r.seg_cell, q.seg_cell)
    assert torch.equal(r.seg_len, q.seg_len) and torch.equal(r.tau, q.tau)
    assert r.seg_cell.numel() == int(r.seg_off[-1])


def test_no_room_to_trim_the_lists(scene, monkeypatch):
    """The traversal has succeeded: lists that cannot be copied down are
    returned as they are."""
    pkg, grid, O, D, want = scene

    def full(self, *a, **k):
        raise torch.cuda.OutOfMemoryError("CUDA out of memory (test)")

    monkeypatch.setattr(torch.Tensor, "clone", full)
    r = grid().trace(O, D, segments=True)
    monkeypatch.undo()
    same(r, want)
    assert r.seg_cell.untyped_storage().nbytes() > 4 * 1.5 * r.seg_cell.numel()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_a_large_first_guess_leaves_no_large_buffers(scene, monkeypatch, precision):
    pkg, grid, O, D, _ = scene
    monkeypatch.setattr(pkg, "_SEG_SMALL", 0)
    vg = grid()
    want = grid().trace(O, D, precision=precision, segments=True, seg_capacity=10 ** 6)
    vg.trace(O, D, precision=precision)             # the buffers of a call without lists
    before = vg.info()["device_bytes"]
    same(vg.trace(O, D, precision=precision, segments=True), want)
    after = vg.info()["device_bytes"]
    assert after - before < 64 * O.shape[0]         # offsets and scans, not the pool
    same(vg.trace(O, D, precision=precision, segments=True), want)
    held = vg.info()["device_bytes"]
    assert held > after                             # the size of the last call: kept
    same(vg.trace(O, D, precision=precision, segments=True), want)
    assert vg.info()["device_bytes"] <= held + 4096


def test_a_first_guess_beyond_the_free_memory_counts_first(scene, monkeypatch):
    pkg, grid, O, D, want = scene
    monkeypatch.setattr(pkg, "_SEG_SMALL", 0)
    monkeypatch.setattr(torch.cuda, "mem_get_info", lambda *a: (1 << 20, 1 << 38))
    asked, empty = [], torch.empty

    def watch(*a, **k):
        if k.get("dtype") == torch.int32 and isinstance(a[0], int):
            asked.append(a[0])
        return empty(*a, **k)

    monkeypatch.setattr(torch, "empty", watch)
    r = grid().trace(O, D, segments=True)
    monkeypatch.undo()
    same(r, want)
    assert max(asked) == r.seg_cell.numel()
