"""Both forms' cell blocks, built on the device, against the oracle with every
site a candidate (GPU).

Every form searches the relative blocks, so comparing forms with each other
holds one set of records against itself. Here the float32 and float64 forms are
held to the oracle, with one lane per ray (which stops early) and with four
(which read every record), and the absolute blocks are read at every crossing:
in units of 2^-110 the float64 form searches each cell in float64."""
import numpy as np
import pytest
import torch

import gen
import oracle

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _shell(n):
    k = np.arange(n) + 0.5
    th, ph = np.arccos(1.0 - 2.0 * k / n), np.pi * (1.0 + 5.0 ** 0.5) * k
    return np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], axis=1)


def _sites(kind, rng):
    if kind == "one":
        return rng.uniform(-1.0, 1.0, (1, 3))
    if kind == "few":                # one to three records, all padding behind them
        return rng.uniform(-1.0, 1.0, (3, 3))
    if kind.startswith("shell"):     # a cell with many neighbours, equally far
        far = rng.uniform(-1.0, 1.0, (300, 3))
        return np.concatenate([[[0.0, 0.0, 0.0]], 0.5 * _shell(int(kind[5:])), far[np.linalg.norm(far, axis=1) > 0.8]])
    if kind == "near and far":       # neighbours at distances over eight decades
        return _shell(120) * (10.0 ** rng.uniform(-8.0, 0.0, 120))[:, None] * 0.99
    if kind == "crowd":
        return np.concatenate([np.array([0.31, -0.17, 0.05]) + 0.01 * (rng.random((1200, 3)) - 0.5),
                               rng.uniform(-1.0, 1.0, (40, 3))])
    if kind == "clumpy":
        return gen.make_clumpy_grid(3000, 133).sites
    return np.stack(np.meshgrid(*[np.linspace(-0.75, 0.75, 7)] * 3, indexing="ij"), -1).reshape(-1, 3)


@pytest.mark.parametrize("gpu_build", [False, True])
@pytest.mark.parametrize("kind", ["one", "few", "shell34", "shell300", "shell4200", "near and far", "crowd", "clumpy",
                                  "lattice"])
def test_paths_are_the_oracles(kind, gpu_build):
    from paper_1310_1854_gb300 import VoronoiGrid
    rng = gen.rng_for(131)
    S = np.unique(np.float32(_sites(kind, rng)).astype(np.float64), axis=0)
    box = gen.make_clumpy_grid(3000, 133).box if kind == "clumpy" else gen.CUBE_BOX
    rho = rng.uniform(0.5, 2.0, len(S)).astype(np.float32)
    n = 1500
    O = box[:3] + (box[3:] - box[:3]) * rng.random((n, 3))
    O[:n // 2] = np.clip(S[rng.integers(0, len(S), n // 2)] + 0.02 * rng.standard_normal((n // 2, 3)), box[:3], box[3:])
    D = gen.isotropic_dirs(n, rng)
    ref = oracle.trace(S, box, rho.astype(np.float64), O, D)
    # (without neighbours the margin has no scale)
    ok = np.nonzero(ref.near_tie == 0)[0] if len(S) > 1 else np.arange(n)
    # neighbours down to 1e-8 apart make many crossings ties against 1e-9
    assert ok.size > (0.5 if kind == "near and far" else 0.9) * n
    diag = np.linalg.norm(box[3:] - box[:3])
    want_off = np.concatenate([[0], np.cumsum([len(ref.segments(k)[0]) for k in ok])])
    want_cell = np.concatenate([ref.segments(k)[0] for k in ok])
    want_len = np.concatenate([ref.segments(k)[1] for k in ok])
    # (the near neighbours' coordinates are not float32 values in the small units)
    for scale in (1.0,) if kind == "near and far" else (1.0, 2.0 ** -110):
        vg = VoronoiGrid(S * scale, box * scale, gpu_build=gpu_build)
        vg.set_density(dev(rho))
        for shape in ({"blocks_per_sm": 64}, {"lanes_per_ray": 4, "fp64_lanes_per_ray": 4}):
            vg.set_launch(**shape)
            for p in ("fp64", "fp32", "fp32_exact") if scale == 1.0 else ("fp64",):
                r = vg.trace(dev(O[ok] * scale), dev(D[ok]), precision=p, segments=True)
                assert np.array_equal(r.seg_off.cpu().numpy(), want_off), (scale, shape, p)
                assert np.array_equal(r.seg_cell.cpu().numpy(), want_cell), (scale, shape, p)
                got = r.seg_len.cpu().numpy().astype(np.float64) / scale
                if p == "fp64":
                    tol = np.where(want_len < 1e-6 * diag, 1e-12 * diag, 1e-12 * want_len)
                    assert np.all(np.abs(got - want_len) <= tol), (scale, shape)
                    np.testing.assert_allclose(r.tau.cpu().numpy() / scale, ref.tau[ok], rtol=1e-12, atol=1e-12 * diag)
