"""The polygon test's affine forms (with the exact test behind them) where
they can go wrong: thin rotated sets, sets far from the origin (differences
to the centre that lose bits), huge and tiny scales (forms switched off or
near under- and overflow), points on and next to the edges, caller-supplied
vertices with repeated points -- survivor lists against the oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402
import pointgen  # noqa: E402

pytestmark = pytest.mark.gpu


def survivors(p, ext, fused):
    d = torch.from_numpy(p).cuda()
    ws = ch.Workspace(len(p))
    if fused:
        _, idx, _, cnt = ch.extremes_and_filter(d, ws)
    else:
        idx, _, cnt = ch.filter_points(d, torch.from_numpy(ext.astype(np.int32)).cuda(), ws)
    ws.check()
    return idx[: int(cnt.item())].cpu().numpy().view(np.uint32)


def make(case, rng, n=20_011):
    if case == "thin":
        return pointgen.make_family("ellipse", n, seed=5)
    base = pointgen.make_points("displaced", n, seed=6).astype(np.float64)
    if case == "far":
        return (base + [1.0e6, -3.0e5]).astype(np.float32)
    if case == "tiny":
        return (base * 1e-41).astype(np.float32)
    if case == "huge":
        return (base * 3.3e38).astype(np.float32)
    if case == "flat":
        return (base * [1.0, 1e-30]).astype(np.float32)
    assert case == "edges"   # the octagon's own edges: points on them and an ulp to either side
    v = np.array([[4, 1], [3, 3], [1, 4], [-2, 3], [-4, 1], [-3, -3], [1, -4], [3, -2]], np.float32)
    t = rng.integers(0, 65, n) / 64.0
    k = rng.integers(0, 8, n)
    p = (v[k] * (1 - t[:, None]) + v[(k + 1) % 8] * t[:, None]).astype(np.float32)
    p = np.nextafter(p, p + rng.integers(-1, 2, p.shape).astype(np.float32), dtype=np.float32)
    p[:8] = v
    return p


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("case", ["thin", "far", "tiny", "huge", "flat", "edges"])
def test_survivors(case, fused):
    p = make(case, np.random.default_rng(3))
    ext = oracle.extremes(p)
    assert np.array_equal(survivors(p, ext, fused), oracle.filter_points(p, ext))


def test_callers_vertices():
    # repeated vertices, a clockwise stretch, points far outside the vertices' box
    p = pointgen.make_points("normal", 20_011, seed=8)
    rng = np.random.default_rng(9)
    for _ in range(6):
        ext = rng.integers(0, len(p), 8).astype(np.uint32)
        ext[3] = ext[2]
        assert np.array_equal(survivors(p, ext, False), oracle.filter_points(p, ext))
    ext = oracle.extremes(p)
    ext[5:7] = ext[4]
    assert np.array_equal(survivors(p, ext, False), oracle.filter_points(p, ext))
