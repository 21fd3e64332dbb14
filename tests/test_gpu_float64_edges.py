"""The float64 form where a ray starts on a wall or on a face (GPU)."""
import numpy as np
import pytest
import torch

import gen
import oracle

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _segments(r):
    return r.seg_off.cpu().numpy(), r.seg_cell.cpu().numpy(), r.seg_len.cpu().numpy()


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -70, 2.0 ** 40])
@pytest.mark.parametrize("lanes", [1, 4])
def test_a_ray_on_a_wall_ends_there(scale, lanes):
    """A ray that starts on a wall with any outward component ends at once
    (Eq. 5 gives s = 0), also where the component is zero in float32."""
    from paper_1310_1854_gb300 import VoronoiGrid
    g = gen.make_uniform_grid(500, 91)
    rng = gen.rng_for(92)
    n = 3000
    o = gen.uniform_points(n, rng)
    d = gen.isotropic_dirs(n, rng)
    i, ax, side = np.arange(n), rng.integers(0, 3, n), rng.choice([-1.0, 1.0], n)
    out = np.array([1e-250, 1e-200, 1e-100, 7e-46, 1e-45, 1e-40, 1e-17, 1e-5])[i % 8]
    d[i, ax] = 0.0
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    d[i, ax] = side * out
    o[i, ax] = side
    S, box, o = g.sites * scale, g.box * scale, np.ascontiguousarray(o * scale)
    ref = oracle.trace(S, box, g.rho.astype(np.float64), o, d)
    assert np.all(ref.tau == 0.0)
    vg = VoronoiGrid(S, box)
    vg.set_density(dev(g.rho))
    vg.set_launch(fp64_lanes_per_ray=lanes)
    r = vg.trace(dev(o), dev(d), precision="fp64", segments=True, status=True)
    assert not torch.any(r.tau) and r.seg_cell.numel() == 0 and not torch.any(r.status)


@pytest.mark.parametrize("lanes", [1, 4])
def test_a_wall_at_zero(lanes):
    """Next to a wall at coordinate 0 a ray can be off it, and move towards it,
    by less than float32 holds: it ends on that wall at a distance of order 1."""
    from paper_1310_1854_gb300 import VoronoiGrid
    rng = gen.rng_for(93)
    S = np.unique(np.float32(rng.random((400, 3))).astype(np.float64), axis=0)
    box = np.array([0.0, 0.0, 0.0, 1.0, 1.0, 1.0])
    rho = rng.uniform(0.5, 2.0, len(S)).astype(np.float32)
    n = 2000
    o, d = rng.random((n, 3)), gen.isotropic_dirs(n, rng)
    i, ax = np.arange(n), rng.integers(0, 3, n)
    tiny = np.array([1e-300, 1e-60, 3e-46, 1e-42, 1e-30])[i % 5]
    d[i, ax] = 0.0
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    d[i, ax] = -tiny
    o[i, ax] = tiny * rng.uniform(0.05, 0.5, n)
    ref = oracle.trace(S, box, rho.astype(np.float64), o, d)
    vg = VoronoiGrid(S, box)
    vg.set_density(dev(rho))
    vg.set_launch(fp64_lanes_per_ray=lanes)
    r = vg.trace(dev(o), dev(d), precision="fp64", segments=True)
    so, sc, sl = _segments(r)
    # near_tie would leave out every ray that ends on that wall (its numerator is tiny)
    ok = np.nonzero(ref.min_margin > oracle.TIE_REL)[0]
    assert ok.size > 0.95 * n and np.mean(np.abs(ref.length[ok] * tiny[ok] / o[ok, ax[ok]] - 1.0) < 1e-9) > 0.5
    for k in ok:
        rc, rl = ref.segments(k)
        assert np.array_equal(sc[so[k]:so[k + 1]], rc), k
        assert np.all(np.abs(sl[so[k]:so[k + 1]] - rl) <= np.where(rl < 1e-6, 1e-12, 1e-12 * rl)), k


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_a_step_of_no_length_adds_nothing(bad):
    """Rays that start on a face take a step of zero length through the cell
    behind it, whatever that cell's density is."""
    from paper_1310_1854_gb300 import VoronoiGrid
    S = np.stack(np.meshgrid(*[np.arange(-0.75, 1.0, 0.5)] * 3, indexing="ij"), -1).reshape(-1, 3)
    rng = gen.rng_for(94)
    rho = rng.uniform(0.5, 2.0, len(S)).astype(np.float32)
    rho[rng.random(len(S)) < 0.3] = bad
    n = 4000
    o, d = gen.uniform_points(n, rng), gen.isotropic_dirs(n, rng)
    i, ax = np.arange(n), rng.integers(0, 3, n)
    o[i, ax] = rng.choice([-0.5, 0.0, 0.5], n)
    vg = VoronoiGrid(S, gen.CUBE_BOX)
    vg.set_density(dev(rho))
    r = vg.trace(dev(o), dev(d), precision="fp64", segments=True, stats=True)
    assert r.stats["zero_steps"] > n // 4
    so, sc, sl = _segments(r)
    want = np.array([np.sum(rho[sc[a:b]].astype(np.float64) * sl[a:b]) for a, b in zip(so[:-1], so[1:])])
    for lanes in (1, 4):
        vg.set_launch(fp64_lanes_per_ray=lanes)
        for tau in (r.tau, vg.trace(dev(o), dev(d), precision="fp64").tau):
            t = tau.cpu().numpy()
            fine = np.isfinite(want)
            assert fine.sum() > n // 50
            np.testing.assert_allclose(t[fine], want[fine], rtol=1e-12)
            assert np.array_equal(np.isnan(t), np.isnan(want)) and np.array_equal(np.isinf(t), np.isinf(want))
