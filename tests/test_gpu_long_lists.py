"""Block lists longer than a warp orders (GPU), from few blocks per site or sites
crowded into one block. C(r), whose scan relies on the order, against brute
force."""
import numpy as np
import pytest
import torch

import gen

from helpers import nearest_site

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n,per_site", [(257, 0.001), (258, 0.001), (511, 0.001), (512, 0.001), (513, 0.02),
                                        (1025, 0.001), (3000, 8.0), (5000, 0.2)])
@pytest.mark.parametrize("where", ["corner", "clumps"])
def test_nearest_site_from_long_lists(where, n, per_site):
    from paper_1310_1854_gb300 import VoronoiGrid
    rng = gen.rng_for(120 + n)
    if where == "corner":
        S = -1.0 + 0.05 * rng.random((2 * n, 3))
    else:
        S = rng.uniform(-0.9, 0.9, (3, 3))[rng.integers(0, 3, 2 * n)] + 1e-3 * rng.standard_normal((2 * n, 3))
    S = np.unique(np.float32(S).astype(np.float64), axis=0)
    S = S[rng.permutation(len(S))[:n]]
    P = gen.uniform_points(6000, rng)
    P[:3000] = np.clip(S[rng.integers(0, n, 3000)] + 0.01 * rng.standard_normal((3000, 3)), -1.0, 1.0)
    want = nearest_site(S, P, chunk=256)
    for reorder in (True, False):
        vg = VoronoiGrid(S, gen.CUBE_BOX, blocks_per_site=per_site, reorder=reorder)
        for p in ("fp32", "fp64"):
            assert np.array_equal(vg.locate(dev(P), precision=p).cpu().numpy(), want), (reorder, p)


@pytest.mark.parametrize("gpu_build", [False, True])
def test_lists_that_are_refused(gpu_build):
    """2^30 blocks and two entries each exceed what offsets hold: the error, and
    a device that takes the next grid."""
    from paper_1310_1854_gb300 import VGridError, VoronoiGrid
    g = gen.make_uniform_grid(1000, 3)
    rays = gen.uniform_rays(1000, 4)
    with pytest.raises(VGridError, match="2\\^31"):
        VoronoiGrid(g.sites, g.box, gpu_build=gpu_build, blocks_per_site=1.1e6)
    tau = [VoronoiGrid(g.sites, g.box, gpu_build=b).trace(dev(rays.origin), dev(rays.dir)).tau for b in (gpu_build, False)]
    assert torch.equal(*tau)
