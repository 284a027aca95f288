"""Hulls of few survivors (one block: sort, repeated points, elimination
passes per side) and the copy of the chains to the hull, at the sizes where
they change over, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402
import pointgen  # noqa: E402

pytestmark = pytest.mark.gpu


def hull(p):
    d = torch.from_numpy(np.ascontiguousarray(p, np.float32)).cuda()
    ws = ch.Workspace(len(p))
    idx, cnt = ch.convex_hull(d, ws)
    ws.check()
    return idx[: int(cnt.item())].cpu().numpy().view(np.uint32)


def points(kind, n):
    rng = np.random.default_rng(n)
    if kind == "circle":
        return pointgen.make_points("circle", n, seed=n)
    if kind == "lattice":   # repeated points, equal x, collinear runs
        return rng.integers(-3, 4, (n, 2)).astype(np.float32)
    if kind == "vertical":
        return np.stack([np.ones(n), rng.integers(0, 9, n)], 1).astype(np.float32)
    if kind == "parabola":  # every point a vertex of one side
        x = rng.permutation(n).astype(np.float64)
        return np.stack([x, x * x], 1).astype(np.float32)
    return np.stack([np.linspace(-1, 1, n), rng.standard_normal(n) * 1e-7], 1).astype(np.float32)   # near a line


@pytest.mark.parametrize("kind", ["circle", "lattice", "vertical", "parabola", "line"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 31, 32, 33, 64, 65, 127, 128, 129, 511, 512, 513, 1025, 4095, 4097])
def test_few_survivors(kind, n):
    p = points(kind, n)
    assert np.array_equal(hull(p), oracle.convex_hull(p)[2])


@pytest.mark.parametrize("n", [2048, 8191, 8192, 8193, 33_000])
def test_many_vertices_per_chunk(n):
    # nearly every point of a small circle is a vertex: ranges longer than
    # one copied part, on one, two and several super-chunks
    p = pointgen.make_points("circle", n, seed=n)
    assert np.array_equal(hull(p), oracle.convex_hull(p)[2])
