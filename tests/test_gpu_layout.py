"""Cell blocks and block lists built on the device: list lengths around the
lanes and buffers of the ordering kernels, and past what they order on the
device. C(r) against brute force, paths against the float64 form (which reads
the absolute blocks) and the same grid in another cell order."""
import numpy as np
import pytest
import torch

import gen

from helpers import nearest_site

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _crowd(n, rng):
    """n sites within 0.01 of a point, 40 around: the lists of the blocks
    there name all n (blocks are larger than the crowd)."""
    c = np.array([0.31, -0.17, 0.05]) + 0.01 * (rng.random((n, 3)) - 0.5)
    return np.concatenate([c, gen.uniform_points(40, rng)])


def _shell(n, rng):
    """One site with n neighbours on a sphere around it, in a sparse box."""
    k = np.arange(n) + 0.5
    th, ph = np.arccos(1.0 - 2.0 * k / n), np.pi * (1.0 + 5.0 ** 0.5) * k
    s = 0.5 * np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], axis=1)
    far = gen.uniform_points(300, rng)
    return np.concatenate([[[0.0, 0.0, 0.0]], s, far[np.linalg.norm(far, axis=1) > 0.8]])


@pytest.mark.parametrize("make,n", [(_crowd, 1), (_crowd, 31), (_crowd, 33), (_crowd, 250), (_crowd, 300), (_crowd, 1200),
                                    (_shell, 34), (_shell, 300), (_shell, 4200)])
def test_lists_of_every_length(make, n):
    from paper_1310_1854_gb300 import VoronoiGrid
    rng = gen.rng_for(70 + n)
    S = np.unique(np.float32(make(n, rng)).astype(np.float64), axis=0)
    rho = rng.uniform(0.5, 2.0, len(S)).astype(np.float32)
    P = gen.uniform_points(3000, rng)
    P[:1500] = S[rng.integers(0, len(S), 1500)] + 0.02 * rng.standard_normal((1500, 3))
    P = np.clip(P, -1.0, 1.0)
    D = gen.isotropic_dirs(3000, rng)
    want = nearest_site(S, P, chunk=256)
    tau = []
    # few blocks per site make the lists long
    for kw in ({"blocks_per_site": 0.05}, {}, {"reorder": False}):
        vg = VoronoiGrid(S, gen.CUBE_BOX, **kw)
        vg.set_density(dev(rho))
        for p in ("fp32", "fp64"):
            assert np.array_equal(vg.locate(dev(P), precision=p).cpu().numpy(), want), (kw, p)
        a = vg.trace(dev(P), dev(D), segments=True)
        b = vg.trace(dev(P), dev(D), precision="fp64", segments=True)
        assert torch.equal(a.seg_off, b.seg_off) and torch.equal(a.seg_cell, b.seg_cell)
        tau.append((a.tau, b.tau))
    for a, b in tau[1:]:
        assert torch.equal(a, tau[0][0]) and torch.equal(b, tau[0][1])
    host = VoronoiGrid(S, gen.CUBE_BOX, host_only=True)
    assert VoronoiGrid(S, gen.CUBE_BOX).info()["block_entries"] == host.info()["block_entries"]
