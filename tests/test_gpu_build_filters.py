"""GPU cell construction: the float32 filters and the spreading of few cells
over warps, against the host builder (every list, volume and bounding box)."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 33, 700, 6000])
@pytest.mark.parametrize("shape,scale", [("ball", 1.0), ("corner", 1.0), ("uniform", 2.0 ** -50), ("uniform", 2.0 ** 70)])
def test_filters_drop_only_what_misses(n, shape, scale):
    """Sites in a ball or a corner: cells reach far across empty space, where
    the filters decide most; tiny and huge coordinates take the scaled path."""
    from paper_1310_1854_gb300 import VoronoiGrid
    rng = gen.rng_for(60 + n)
    if shape == "ball":
        S = gen.ball_points(n, rng)
    elif shape == "corner":
        S = -1.0 + 0.05 * rng.random((n, 3))
    else:
        S = gen.uniform_points(n, rng)
    S = np.unique(np.float32(S).astype(np.float64), axis=0) * scale
    box = gen.CUBE_BOX * scale
    a, b = VoronoiGrid(S, box, gpu_build=True), VoronoiGrid(S, box, host_only=True)
    (ao, ai), (bo, bi) = a.neighbors(), b.neighbors()
    for m in range(len(S)):
        p, q = set(ai[ao[m]:ao[m + 1]].tolist()), set(bi[bo[m]:bo[m + 1]].tolist())
        assert len(p ^ q) <= 2, m   # at most planes that only touch the cell
    (av, ab), (bv, bb) = a.cells(), b.cells()
    np.testing.assert_allclose(av, bv, rtol=1e-9, atol=1e-13 * 8.0 * scale ** 3)
    np.testing.assert_allclose(ab, bb, rtol=0, atol=1e-11 * scale)
    np.testing.assert_allclose(av.sum(), 8.0 * scale ** 3, rtol=1e-11)


@pytest.mark.parametrize("n", [3, 6, 7, 1029, 4098])
@pytest.mark.parametrize("stretch", [(1.0, 1.0, 1.0), (1.0, 1.0, 0.004), (0.004, 1.0, 0.004), (0.004, 1.0, 1.0)])
def test_bucket_rows_in_thin_boxes(n, stretch):
    """Boxes one bucket thin along any axis, sizes off the multiples of four, and
    sites crowded at one end, so that rows of buckets are skipped or ragged: the
    lists of the host builder (no face of random sites is degenerate), volumes
    to the rounding of a cell's cuts (1e-9)."""
    from paper_1310_1854_gb300 import VoronoiGrid
    rng = gen.rng_for(70 + n)
    box = np.float32(gen.CUBE_BOX * np.tile(stretch, 2)).astype(np.float64)
    u = rng.random((n, 3))
    u[:, 1] **= 3.0
    S = np.float32(box[:3] + (0.001 + 0.998 * u) * (box[3:] - box[:3])).astype(np.float64)
    S = np.unique(S, axis=0)
    a, b = VoronoiGrid(S, box, gpu_build=True), VoronoiGrid(S, box, host_only=True)
    (ao, ai), (bo, bi) = a.neighbors(), b.neighbors()
    for m in range(len(S)):
        assert set(ai[ao[m]:ao[m + 1]].tolist()) == set(bi[bo[m]:bo[m + 1]].tolist()), m
    np.testing.assert_allclose(a.cells()[0], b.cells()[0], rtol=1e-9)
