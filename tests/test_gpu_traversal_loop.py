"""The traversal loop's ray queue (GPU).

The queue hands a warp up to 32 rays at a time: that may not change a result,
so every comparison is exact (bit for bit).
"""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("lanes,block,per_sm,order", [(1, 128, 0, -1), (1, 32, 1, 1), (4, 256, 1, -1), (8, 64, 2, 1)])
def test_queue_hands_out_every_ray_once(lanes, block, per_sm, order):
    from paper_1310_1854_gb300 import VoronoiGrid
    g = gen.make_uniform_grid(700, 41)
    vg = VoronoiGrid(g.sites, g.box)
    vg.set_density(dev(g.rho), 1.25)
    rays = gen.uniform_rays(20_011, 42)
    O, D = dev(rays.origin), dev(rays.dir)
    O[::97] += 5.0  # outside the domain
    tint = torch.rand(O.shape[0], device="cuda")
    w = torch.rand(O.shape[0], device="cuda")
    vg.set_launch(order=-1)
    want = {p: vg.trace(O, D, precision=p).tau for p in ("fp32", "fp64")}
    cell, s, _ = vg.interact(O, D, tint, w)
    vg.set_launch(lanes_per_ray=lanes, block=block, blocks_per_sm=per_sm, fp64_lanes_per_ray=lanes, order=order)
    for n in (1, 31, 32, 33, 4097, 20_011):
        for p in want:
            r = vg.trace(O[:n], D[:n], precision=p, stats=True, status=True)
            assert torch.equal(r.tau, want[p][:n]), (n, p)
            out = int((r.status == 1).sum())
            assert out == (n + 96) // 97
            q = vg.trace(O[:n], D[:n], precision=p, segments=True)
            assert torch.equal(q.tau, r.tau)
            st = r.stats
            assert st["rays"] == n and st["outside"] == out
            assert st["crossings"] == q.seg_cell.numel() == q.stats["crossings"]
            assert st["decisions"] == st["crossings"] + st["zero_steps"]  # no step without an exit here
        c, d, _ = vg.interact(O[:n], D[:n], tint[:n], w[:n])
        assert torch.equal(c, cell[:n]) and torch.equal(d, s[:n]), n
