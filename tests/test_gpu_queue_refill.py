"""The traversal's ray queue where the lanes of a warp are far apart (GPU): a
warp refills its queue while other lanes have only just read their slots, so
rays of very different lengths are dealt out in several orders and over few
warps (many refills each). Each ray's results depend on nothing else: exact."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("lanes,block,per_sm", [(1, 32, 1), (1, 128, 1), (2, 64, 1), (8, 32, 1)])
def test_every_order_of_the_rays(lanes, block, per_sm):
    from paper_1310_1854_gb300 import Batch, VoronoiGrid
    g = gen.make_uniform_grid(3000, 81)
    vg = VoronoiGrid(g.sites, g.box)
    vg.set_density(dev(g.rho), 1.5)
    n = 30_001
    rays = gen.uniform_rays(n, 82)
    # one crossing to a path through the whole box, in any order
    k = np.arange(n) % 5
    near = rays.dir * np.where(k == 0, 0.0, np.where(k == 1, 0.999, 0.0))[:, None]
    edge = near / np.maximum(np.abs(near).max(axis=1, keepdims=True), 1e-30) * 0.999
    rays.origin[:] = np.where((k == 1)[:, None], edge, rays.origin)
    rays.origin[k == 2] += 5.0  # outside
    O, D = dev(rays.origin), dev(rays.dir)
    rng = gen.rng_for(83)
    tint, w = dev(rng.exponential(1.0, n).astype(np.float32)), dev(rng.random(n).astype(np.float32))
    dL = dev(rng.standard_normal(n).astype(np.float32))
    vg.set_launch(lanes_per_ray=lanes, block=block, blocks_per_sm=per_sm, fp64_lanes_per_ray=lanes, order=-1)
    want = None
    for p in (np.arange(n), np.argsort(k, kind="stable"), rng.permutation(n)):
        P = dev(p)
        o, d = O[P], D[P]
        inv = torch.empty_like(P)
        inv[P] = torch.arange(n, device=P.device)
        seg = vg.trace(o, d, segments=True, status=True)
        cell, s, _ = vg.interact(o, d, tint[P], w[P])
        got = [vg.trace(o, d).tau[inv], vg.trace(o, d, precision="fp64").tau[inv],
               vg.trace(o, d, precision="fp32_exact").tau[inv], seg.tau[inv], seg.status[inv],
               torch.diff(seg.seg_off)[inv], cell[inv], s[inv]]
        b = Batch([(vg, o[:n // 3].contiguous(), d[:n // 3].contiguous()),
                   (vg, o[n // 3:].contiguous(), d[n // 3:].contiguous())])
        b.set_launch(lanes, block, per_sm, -1)
        b.run()
        torch.cuda.synchronize()
        got.append(torch.cat(list(b.tau))[inv])
        grad = vg.trace_grad(o, d, dL[P])
        if want is None:
            want, want_grad = got, grad
        for i, (x, y) in enumerate(zip(got, want)):
            assert torch.equal(x, y), i
        # the same float32 terms added in another order: each sum is within
        # count 2^-24 of the sum of the terms' sizes
        size = vg.trace_grad(o, d, dL[P].abs())
        count = torch.bincount(seg.seg_cell, minlength=vg.M)
        assert bool(((grad - want_grad).abs() <= 2.1 * count * 2.0 ** -24 * size).all())
