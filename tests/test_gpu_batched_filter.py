"""The batched filter against the oracle at its changes of path: sets around
the sizes that get a fan (16384 points; 65536 on a circle) and its bins, fans
that are dropped (a square's boundary, a ring of few directions), sets at even
and odd positions (16- and 8-byte loads), sets without a fan between them, and
a workspace that a single-set call has used before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle_par  # noqa: E402
import oracle  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402
import pointgen  # noqa: E402

pytestmark = pytest.mark.gpu


def want(p):
    return oracle_par.hull(p, oracle_par.filter_points(p, oracle.extremes(p)))


def check(sets, ws=None):
    off = np.cumsum([0] + [len(s) for s in sets]).astype(np.int64)
    pts = torch.from_numpy(np.concatenate(sets)).cuda()
    ws = ws or ch.Workspace(int(off[-1]), num_sets=len(sets))
    idx, hoff = ch.convex_hull_batched(pts, torch.from_numpy(off).cuda(), ws)
    ws.check()
    idx, hoff = idx.cpu().numpy().view(np.uint32), hoff.cpu().numpy()
    for b, p in enumerate(sets):
        assert np.array_equal(idx[hoff[b]:hoff[b + 1]], want(p)), (b, len(p))
    return ws


def family(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "square":
        t = rng.uniform(-1, 1, n)
        s = rng.integers(0, 4, n)
        x = np.where(s < 2, t, np.where(s == 2, 1.0, -1.0))
        y = np.where(s < 2, np.where(s == 0, 1.0, -1.0), t)
        return np.stack([x, y], 1).astype(np.float32)
    if kind == "spokes":
        th = rng.integers(0, 40, n) * (2 * np.pi / 40)
        r = 1.0 - np.abs(rng.normal(0, 0.05, n))
        return np.stack([r * np.cos(th), r * np.sin(th)], 1).astype(np.float32)
    if kind in ("gaussians", "ellipse"):
        return pointgen.make_family(kind, n, seed=seed)
    return pointgen.make_points(kind, n, seed=seed)


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("kind", ["circle", "displaced", "normal", "ellipse", "gaussians", "square", "spokes"])
def test_sizes(kind, shift):
    sizes = [16_383, 16_384, 16_385, 20_480, 65_535, 65_536, 65_537, 131_071, 131_073, 4097, 300_001]
    sets = [pointgen.make_points("normal", 4 + shift, seed=1)]
    sets += [family(kind, n, 100 * shift + k) for k, n in enumerate(sizes)]
    check(sets)


def test_workspace_used_by_a_single_set():
    p = pointgen.make_points("circle", 900_001, seed=3)
    ws = ch.Workspace(900_001, num_sets=12)
    d = torch.from_numpy(p).cuda()
    for _ in range(2):
        idx, cnt = ch.convex_hull(d, ws)
        ws.check()
        assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), want(p))
        check([family(("circle", "displaced", "ellipse")[k % 3], 70_000 + 13 * k, k) for k in range(12)], ws)
