"""The merge tree over super-chunks where its tangent search can go wrong:
chains that lose nothing, a few vertices, most of them or whole chunks in one
merge, on both sides -- hulls of one set and of a batch against the
oracle's.  (Fewer than 65536 points: the octagon's survivors are sorted as
they are.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402
import pointgen  # noqa: E402

pytestmark = pytest.mark.gpu


def points(kind, n):
    rng = np.random.default_rng(n)
    if kind == "circle":
        return pointgen.make_points("circle", n, seed=n)
    if kind == "diamond":      # collinear sides: every inner chunk goes
        t = rng.integers(-(1 << 20), (1 << 20) + 1, n) * 2.0 ** -20
        return np.stack([t, (1 - np.abs(t)) * rng.choice([-1.0, 1.0], n)], 1).astype(np.float32)
    th = rng.uniform(0, 2 * np.pi, n)
    if kind == "ellipse":      # steep ends: long walks between unequal chains
        p = np.stack([np.cos(th), np.sin(th) / 19.0], 1) @ np.array([[0.8, 0.6], [-0.6, 0.8]])
    elif kind == "dents":      # stretches of the circle that sink below their chord
        p = np.stack([np.cos(th), np.sin(th)], 1) * (1 - 1e-4 * (np.sin(37 * th) > 0.3))[:, None]
    else:                      # one far point on either side: nearly all of the other chunks go
        p = np.stack([np.cos(th), 0.5 * np.sin(th)], 1)
        p[:2] = [[3.0, 40.0], [-2.0, -40.0]]
        p[2:, 0] *= 50.0
    return p.astype(np.float32)


KINDS = ["circle", "diamond", "ellipse", "dents", "far"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [4097, 8193, 20_000, 65_535])
def test_single(kind, n):
    p = points(kind, n)
    ws = ch.Workspace(n)
    idx, cnt = ch.convex_hull(torch.from_numpy(p).cuda(), ws)
    ws.check()
    assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), oracle.convex_hull(p)[2])


def test_batch():
    sets = [points(k, n) for n in (9001, 300, 40_000) for k in KINDS]
    off = np.concatenate([[0], np.cumsum([len(p) for p in sets])]).astype(np.int64)
    ws = ch.Workspace(int(off[-1]), num_sets=len(sets))
    idx, ho = ch.convex_hull_batched(torch.from_numpy(np.concatenate(sets)).cuda(), torch.from_numpy(off).cuda(), ws)
    ws.check()
    ho, idx = ho.cpu().numpy(), idx.cpu().numpy().view(np.uint32)
    for b, p in enumerate(sets):
        assert np.array_equal(idx[ho[b]: ho[b + 1]], oracle.convex_hull(p)[2]), b
