"""One lane per ray, which a shape asks for with blocks_per_sm (GPU): the
default lets calls of few rays take several. Every shape gives the same bits
(float32 atomics apart)."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu

ONE = {"lanes_per_ray": 1, "fp64_lanes_per_ray": 1, "blocks_per_sm": 64}  # more blocks than fit


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _everything(vg, O, D, tint):
    out = [vg.trace(O, D, precision=p, enter=e).tau for p in ("fp32", "fp32_exact", "fp64") for e in (False, True)]
    for p in ("fp32", "fp32_exact", "fp64"):
        r = vg.trace(O, D, precision=p, segments=True, status=True)
        out += [r.tau, r.seg_off, r.seg_cell, r.seg_len, r.status]
    cell, s, _ = vg.interact(O, D, tint)
    return out + [cell, s, vg.trace_host(O.cpu(), D.cpu()).tau.cuda()]


@pytest.mark.parametrize("n", [1, 100, 4_000, 20_000, 75_000, 130_000, 260_000])
@pytest.mark.parametrize("place", ["disk", "ball"])
def test_every_shape_gives_the_same(place, n):
    from paper_1310_1854_gb300 import VoronoiGrid
    if place == "disk":
        g, rays, kw = gen.make_disk_grid(1500, 50), gen.disk_rays(n, 51), {}
    else:
        g, rays, kw = gen.make_ball_grid(1500, 50), gen.ball_rays(n, 51), {"sphere": tuple(gen.UNIT_BALL)}
    O, D = dev(rays.origin), dev(rays.dir)
    tint = dev(gen.rng_for(52).random(n).astype(np.float32))
    want = None
    for shape in (ONE, {}, {"lanes_per_ray": 2, "fp64_lanes_per_ray": 4}, {"lanes_per_ray": 8, "fp64_lanes_per_ray": 2}):
        vg = VoronoiGrid(g.sites, g.box, **kw)
        vg.set_density(dev(g.rho))
        vg.set_launch(**shape)
        got = _everything(vg, O, D, tint)
        want = want or got
        for i, (x, y) in enumerate(zip(got, want)):
            assert torch.equal(x, y), (shape, i)
