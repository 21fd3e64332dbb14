"""The traversal loop's ray queue, early stop and float32 search (GPU).

The queue hands a warp up to 32 rays at a time and the search leaves out the
records that lie too far from the site: neither may change a result, so every
comparison is exact (bit for bit). The float64 form searches in float32 with
error bounds and evaluates the exit in float64: its paths are the oracle's.
"""
import numpy as np
import pytest
import torch

import gen
import oracle

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


def _shell(n):
    k = np.arange(n) + 0.5
    th, ph = np.arccos(1.0 - 2.0 * k / n), np.pi * (1.0 + 5.0 ** 0.5) * k
    return np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], axis=1)


def _sites(kind, rng):
    if kind == "few":            # one to three records, all padding behind them
        return rng.uniform(-1.0, 1.0, (3, 3))
    if kind == "equidistant":    # a cell whose 80 neighbours are equally far
        far = rng.uniform(-1.0, 1.0, (1500, 3))
        return np.concatenate([[[0.0, 0.0, 0.0]], 0.5 * _shell(80), far[np.linalg.norm(far, axis=1) > 0.75][:200]])
    if kind == "near and far":   # neighbours at distances over eight decades
        return _shell(120) * (10.0 ** rng.uniform(-8.0, 0.0, 120))[:, None] * 0.99
    return np.stack(np.meshgrid(*[np.linspace(-0.75, 0.75, 7)] * 3, indexing="ij"), -1).reshape(-1, 3)


@pytest.mark.parametrize("kind", ["few", "equidistant", "near and far", "lattice"])
def test_early_stop_takes_the_same_paths(kind):
    """One lane per ray stops early, four lanes read every record, the float64
    form tests every plane in float64."""
    from paper_1310_1854_gb300 import VoronoiGrid
    rng = gen.rng_for(43)
    S = np.unique(np.float32(_sites(kind, rng)).astype(np.float64), axis=0)
    vg = VoronoiGrid(S, gen.CUBE_BOX)
    vg.set_density(dev(rng.uniform(0.5, 2.0, len(S)).astype(np.float32)))
    rays = gen.uniform_rays(4_000, 44)
    k = rng.integers(0, len(S), 1_000)
    rays.origin[:1_000] = np.clip(S[k] + 1e-7 * rng.standard_normal((1_000, 3)), -1.0, 1.0)
    O, D = dev(rays.origin), dev(rays.dir)
    a = vg.trace(O, D, segments=True, stats=True)
    vg.set_launch(lanes_per_ray=4)
    b = vg.trace(O, D, segments=True, stats=True)
    assert a.stats == b.stats
    for x in ("tau", "seg_off", "seg_cell", "seg_len"):
        assert torch.equal(getattr(a, x), getattr(b, x)), x
    vg.set_launch()
    c = vg.trace(O, D, precision="fp64", segments=True)
    if kind != "lattice":        # rays through edges may order ties otherwise
        assert torch.equal(a.seg_off, c.seg_off) and torch.equal(a.seg_cell, c.seg_cell)


@pytest.mark.parametrize("sphere", [None, tuple(gen.UNIT_BALL)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -70, 2.0 ** 40])
def test_float64_form_at_the_boundary(scale, sphere):
    """Rays along the walls, off them by nothing to 1e-3, with direction
    components down to 1e-300, and rays that graze the sphere: the domain's
    exit is where the float32 bounds are widest. Segment lengths to 1e-12 as
    the other float64 tests."""
    from paper_1310_1854_gb300 import VoronoiGrid
    g = gen.make_ball_grid(800, 45) if sphere else gen.make_uniform_grid(800, 45)
    rng = gen.rng_for(46)
    n = 6000
    rays = (gen.ball_rays if sphere else gen.uniform_rays)(n, 47)
    o, d = rays.origin, rays.dir
    ax, side = rng.integers(0, 3, n), rng.choice([-1.0, 1.0], n)
    i = np.arange(n)
    if sphere is None:
        o[i, ax] = side * (1.0 - rng.choice([0.0, 1e-16, 1e-12, 1e-9, 1e-6, 1e-3], n))
        d[i, ax] = side * rng.choice([0.0, 1e-300, 1e-40, 1e-17, 1e-9, 1e-5, 1e-2], n) * rng.choice([-1.0, 1.0], n)
        d[i, (ax + 1) % 3] += 0.25  # not zero
        d /= np.linalg.norm(d, axis=1, keepdims=True)
    else:
        u = gen.isotropic_dirs(n, rng)
        t = np.cross(u, gen.isotropic_dirs(n, rng))
        t /= np.linalg.norm(t, axis=1, keepdims=True)
        o[:] = u * (1.0 - rng.choice([1e-12, 1e-9, 1e-6, 1e-3], n))[:, None]
        d[:] = t + side[:, None] * rng.choice([0.0, 1e-9, 1e-5, 1e-2], n)[:, None] * u
        d /= np.linalg.norm(d, axis=1, keepdims=True)
    S, box = g.sites * scale, g.box * scale
    sp = None if sphere is None else tuple(np.array(sphere) * scale)
    o = np.ascontiguousarray(o * scale)
    off, idx = oracle.csr(oracle.cells(S, box), len(S))
    ref = oracle.trace(S, box, g.rho.astype(np.float64), o, d, off=off, idx=idx, **({"sphere": sp} if sp else {}))
    ok = np.nonzero(ref.near_tie == 0)[0]
    assert ok.size > 0.5 * n
    vg = VoronoiGrid(S, box, sphere=sp)
    vg.set_density(dev(g.rho))
    for lanes in (1, 4):
        vg.set_launch(fp64_lanes_per_ray=lanes)
        r = vg.trace(dev(o), dev(d), precision="fp64", segments=True)
        so, sc, sl = r.seg_off.cpu().numpy(), r.seg_cell.cpu().numpy(), r.seg_len.cpu().numpy()
        diag = np.linalg.norm(box[3:] - box[:3])
        for k in ok:
            rc, rl = ref.segments(k)
            assert np.array_equal(sc[so[k]:so[k + 1]], rc), k
            gl = sl[so[k]:so[k + 1]]
            assert np.all(np.abs(gl - rl) <= np.where(rl < 1e-6 * diag, 1e-12 * diag, 1e-12 * rl)), k
        np.testing.assert_allclose(r.tau.cpu().numpy()[ok], ref.tau[ok], rtol=1e-12, atol=1e-300)


def test_segment_buffers_guessed_counted_and_short_of_memory(monkeypatch):
    """The lists are the same whether the buffers are sized on the first
    guess, on the last call, after a count, or after a guess that is too small
    or does not fit in memory; a generous guess is not kept alive."""
    import paper_1310_1854_gb300 as pkg
    g = gen.make_disk_grid(3000, 48)
    rays = gen.disk_rays(2000, 49)
    O, D = dev(rays.origin), dev(rays.dir)

    def grid():
        vg = pkg.VoronoiGrid(g.sites, g.box)
        vg.set_density(dev(g.rho))
        return vg

    def same(r, q):
        assert torch.equal(r.seg_off, q.seg_off) and torch.equal(r.seg_cell, q.seg_cell)
        assert torch.equal(r.seg_len, q.seg_len) and torch.equal(r.tau, q.tau)
        total = int(r.seg_off[-1])
        assert r.seg_cell.numel() == total == r.stats["crossings"]
        assert r.seg_cell.untyped_storage().nbytes() <= 4 * (1.5 * total + 4096) + 512

    vg = grid()
    want = vg.trace(O, D, segments=True)          # first guess
    same(vg.trace(O, D, segments=True), want)     # from the last call
    vg._seg_per_ray = 0.01
    same(vg.trace(O, D, segments=True), want)     # too small: traced again
    monkeypatch.setattr(pkg, "_SEG_GUESS_MAX", 10)
    same(grid().trace(O, D, segments=True), want)  # counted first
    monkeypatch.undo()
    empty, asked = torch.empty, []

    def tight(*a, **k):
        n = a[0] if isinstance(a[0], int) else 0
        if n > want.seg_cell.numel() and k.get("dtype") == torch.int32:
            asked.append(n)
            raise torch.cuda.OutOfMemoryError("CUDA out of memory (test)")
        return empty(*a, **k)

    monkeypatch.setattr(torch, "empty", tight)
    r = grid().trace(O, D, segments=True)         # the guess does not fit
    monkeypatch.undo()
    assert asked
    same(r, want)
    none = vg.trace(O[:0], D[:0], segments=True)
    assert none.seg_cell.numel() == 0 and int(none.seg_off[0]) == 0


@pytest.mark.parametrize("n", [100, 4_000, 20_000, 100_000, 130_000, 260_000])
def test_default_shape_follows_the_rays(n):
    """Without a shape set, few rays get several lanes each: the results are
    those of one lane per ray, in every form and mode."""
    from paper_1310_1854_gb300 import VoronoiGrid
    g = gen.make_disk_grid(1500, 50)
    rays = gen.disk_rays(n, 51)
    O, D = dev(rays.origin), dev(rays.dir)
    tint = torch.rand(n, device="cuda")

    def everything(vg):
        out = [vg.trace(O, D, precision=p).tau for p in ("fp32", "fp32_exact", "fp64")]
        for p in ("fp32", "fp32_exact", "fp64"):
            r = vg.trace(O, D, precision=p, segments=True, status=True)
            out += [r.tau, r.seg_off, r.seg_cell, r.seg_len, r.status]
        cell, s, _ = vg.interact(O, D, tint)
        return out + [cell, s, vg.trace_host(O.cpu(), D.cpu()).tau.cuda()], vg.trace_grad(O, D, tint)

    auto = VoronoiGrid(g.sites, g.box)
    one = VoronoiGrid(g.sites, g.box)
    one.set_launch(lanes_per_ray=1)
    for vg in (auto, one):
        vg.set_density(dev(g.rho))
    (a, ga), (b, gb) = everything(auto), everything(one)
    for i, (x, y) in enumerate(zip(a, b)):
        assert torch.equal(x, y), i
    # float32 atomics in another order: the same terms, some hundred per cell
    torch.testing.assert_close(ga, gb, rtol=1e-4, atol=1e-6 * float(gb.abs().max()))
