"""The hull step's fan around a centre that sees most points within a small
angle: a cloud with a few far points.  Consecutive vertices half a turn apart
cost the points of their wedge only, in one set (both levels) and per set of a
batch.  The hulls are the oracle's, and the points to sort stay a fraction of
what the octagon leaves: at least half of them go even from a circle, whose
points lie next to the fan's chords, and three quarters from a displaced one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import fan_query  # noqa: E402
import oracle  # noqa: E402
import oracle_par  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402
import pointgen  # noqa: E402

pytestmark = pytest.mark.gpu


def cloud(dist, n, seed, far, at):
    """n points of a distribution, those from index `at` on replaced by the far ones."""
    p = pointgen.make_points(dist, n, seed=seed)
    p[at:at + len(far)] = far
    return p


ONE = np.array([[10.0, 0.0]], np.float32)                                    # in an axis direction: the end of a bin
OFF = np.array([[9.0, 3.25]], np.float32)
THREE = np.array([[10.0, 0.0], [11.0, 0.25], [12.0, 0.5]], np.float32)


@pytest.mark.parametrize("dist,n,far,at,most", [
    ("displaced", 300_007, ONE, 100_000, 0.25),
    ("displaced", 300_007, OFF, 100_000, 0.25),
    ("displaced", 65_536 * 3, THREE, 5, 0.25),
    ("displaced", 13_000_003, THREE, 4096 + 70, 0.25),   # in a tile that the bins do not sample
    ("circle", 4_200_001, ONE, 4_200_000, 0.75),         # the second level's wedges
    ("circle", 13_000_003, THREE, 4096 + 70, 0.75),
])
def test_single(dist, n, far, at, most):
    p = cloud(dist, n, n % 97, far, at)
    d = torch.from_numpy(p).cuda()
    ws = ch.Workspace(n)
    idx, cnt = ch.convex_hull(d, ws)
    ws.check()
    want = oracle_par.filter_points(p, oracle.extremes(p))
    s_oct, t, _, _ = ch.ch_hull_counts(ws.buf, n)
    assert s_oct == len(want)
    assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), oracle_par.hull(p, want))
    assert t <= most * s_oct, (t, s_oct)


def test_batch():
    cases = [(60_001, ONE), (60_001, OFF), (400_003, ONE), (400_003, THREE), (400_003, OFF), (20_000, THREE)]
    sets = [cloud("displaced", n, 31 + i, far, n // 3) for i, (n, far) in enumerate(cases)]
    sets.append(pointgen.make_points("displaced", 60_001, seed=38))
    off = np.concatenate([[0], np.cumsum([len(p) for p in sets])]).astype(np.int64)
    d, o = torch.from_numpy(np.concatenate(sets)).cuda(), torch.from_numpy(off).cuda()
    ws = ch.Workspace(int(off[-1]), len(sets))
    idx = torch.zeros(int(off[-1]), dtype=torch.int32, device="cuda")
    ho = torch.zeros(len(sets) + 1, dtype=torch.int64, device="cuda")
    ch.ch_hull_batched(d, o, idx, ho, ws.buf)
    ws.check()
    at = fan_query.query(ws.buf.numel(), len(sets))[2]
    kept = ws.buf[at:at + 4 * len(sets)].cpu().numpy().view(np.uint32)
    h = ho.cpu().numpy()
    for i, p in enumerate(sets):
        want = oracle_par.filter_points(p, oracle.extremes(p))
        got = idx[int(h[i]): int(h[i + 1])].cpu().numpy().view(np.uint32)
        assert np.array_equal(got, oracle_par.hull(p, want)), i
        assert kept[i] <= 0.25 * len(want), (i, kept[i], len(want))
