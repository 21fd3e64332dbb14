"""Grids in other units of length (GPU): a kiloparsec is 3e19 m or 3e21 cm, an
atom 1e-10 m. Lengths times a power of two are exact, and so is what float64
makes of them: results scale with the unit, bit for bit."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _grid(place):
    if place == "ball":
        g = gen.make_ball_grid(2000, 101)
        return g, gen.ball_rays(5000, 102), np.array(gen.UNIT_BALL)
    if place == "disk":
        g = gen.make_disk_grid(2000, 101)
        return g, gen.disk_rays(5000, 102), None
    g = gen.make_uniform_grid(2000, 101)
    rays = gen.uniform_rays(5000, 102)
    i = np.arange(1500)  # start on walls and next to them, along them and into them
    rays.origin[i, i % 3] = np.where(i % 2, 1.0, -1.0) * (1.0 - np.array([0.0, 1e-14, 1e-7])[i % 5 % 3])
    rays.dir[i[::2], i[::2] % 3] *= 1e-9
    rays.dir /= np.linalg.norm(rays.dir, axis=1, keepdims=True)
    return g, rays, None


@pytest.mark.parametrize("place", ["uniform", "disk", "ball"])
def test_cells_of_points_in_every_unit(place):
    """C(r) where squared distances leave float32's range, in part of a block's
    list or in all of it."""
    from paper_1310_1854_gb300 import VoronoiGrid
    g, rays, sphere = _grid(place)
    rng = gen.rng_for(103)
    P = np.concatenate([rays.origin, g.box[:3] + (g.box[3:] - g.box[:3]) * rng.random((20_000, 3))])
    want = None
    for p in (0, -105, -70, -30, 40, *range(58, 74), 100):
        scale = 2.0 ** p
        kw = {} if sphere is None else {"sphere": tuple(sphere * scale)}
        # few blocks per site make lists that reach across the grid
        for per_site in (8.0, 0.02):
            vg = VoronoiGrid(g.sites * scale, g.box * scale, blocks_per_site=per_site, **kw)
            for prec in ("fp32", "fp64"):
                c = vg.locate(dev(P * scale), precision=prec)
                want = c if want is None else want
                assert torch.equal(c, want), (p, per_site, prec)


@pytest.mark.parametrize("place", ["uniform", "disk", "ball"])
def test_float64_results_scale_with_the_unit(place):
    from paper_1310_1854_gb300 import VoronoiGrid
    g, rays, sphere = _grid(place)
    D = dev(rays.dir)

    def run(scale):
        kw = {} if sphere is None else {"sphere": tuple(sphere * scale)}
        vg = VoronoiGrid(g.sites * scale, g.box * scale, **kw)
        vg.set_density(dev(g.rho))
        O = dev(rays.origin * scale)
        out = []
        for shape in ({"blocks_per_sm": 64}, {}, {"fp64_lanes_per_ray": 4}):
            vg.set_launch(**shape)
            r = vg.trace(O, D, precision="fp64", segments=True, status=True)
            t = vg.trace(O, D, precision="fp64")
            out.append((r.seg_off, r.seg_cell, r.status, r.seg_len / scale, r.tau / scale, t.tau / scale))
        return out

    want = run(1.0)
    for p in (-105, -95, -70, -30, -21, 39, 42, 62, 64, 65, 66, 76, 95, 110):
        for a, b in zip(run(2.0 ** p), want):
            for i, (x, y) in enumerate(zip(a, b)):
                assert torch.equal(x, y), (p, i)
