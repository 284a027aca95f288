"""Points in the directions of the fan's bin ends and an ulp beside them, seen
from a box centre at the origin, with the library's own bin counts: the first
level, the second one (eight times as many bins) and a batch's sets, whose
bins go by their size.  A vertex near an end of its bin, or a pseudo-angle
rounded into the wrong bin, would drop hull points; and the fan must be at
work: it drops at least half of the octagon's survivors."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import fan_query  # noqa: E402
import oracle  # noqa: E402
import oracle_par  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402

pytestmark = pytest.mark.gpu


def ends(bins, n, seed, spread):
    """n points: pseudo-angles that are multiples of 4 / bins, or next to them, and (every fourth, as such points
    are never vertices) any."""
    rng = np.random.default_rng(seed)
    a = rng.integers(0, bins, n) * (4.0 / bins)   # (from -y counter-clockwise; the set is symmetric)
    a[::4] = rng.uniform(0, 4, len(a[::4]))
    q, t = np.floor(a).astype(int), a % 1.0
    x = np.where(q % 2 == 0, 1 - t, -t) * np.where(q < 2, 1, -1)
    y = np.where(q % 2 == 0, t, 1 - t) * np.where(q < 2, 1, -1)
    r = 1.0 - np.abs(rng.normal(0, spread, n))
    p = (np.stack([x, y], 1) * (r / np.hypot(x, y))[:, None]).astype(np.float32)
    p = np.nextafter(p, p + rng.integers(-1, 2, p.shape).astype(np.float32), dtype=np.float32)
    p[:4] = [[1.03, 0], [0, 1.03], [-1.03, 0], [0, -1.03]]   # the box's centre at the origin
    return p


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("level", [1, 2])
def test_single(level, shift):
    n = 200_003 if level == 1 else (1 << 19) + 77
    p = ends(fan_query.query()[level - 1], n, 61 + level, 0.02 if level == 1 else 0.002)
    d = torch.from_numpy(np.concatenate([np.zeros((shift, 2), np.float32), p])).cuda()[shift:]
    ws = ch.Workspace(n)
    ch.ch_tune_set("fan2_min_log2", 10)
    try:
        idx, cnt = ch.convex_hull(d, ws)
        ws.check()
    finally:
        ch.ch_tune_set("fan2_min_log2", 0)
    want = oracle_par.filter_points(p, oracle.extremes(p))
    c = ch.ch_hull_counts(ws.buf, n)
    assert c[0] == len(want) and c[1] <= 0.5 * c[0], list(c)
    assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), oracle_par.hull(p, want))


def test_batch():
    # bins by a set's tiles, 256 a tile in runs of 512, at most 8192
    sizes = [20_000, 60_001, 131_073, 300_001]
    sets = [ends(min(-(-(-(-n // 4096) * 256) // 512) * 512, 8192), n, 71 + i, 0.02) for i, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    d, o = torch.from_numpy(np.concatenate(sets)).cuda(), torch.from_numpy(off).cuda()
    ws = ch.Workspace(int(off[-1]), len(sets))
    idx, ho = ch.convex_hull_batched(d, o, ws)
    ws.check()
    at = fan_query.query(ws.buf.numel(), len(sets))[2]
    kept = ws.buf[at:at + 4 * len(sets)].cpu().numpy().view(np.uint32)
    h = ho.cpu().numpy()
    for i, p in enumerate(sets):
        want = oracle_par.filter_points(p, oracle.extremes(p))
        assert kept[i] <= 0.5 * len(want), (i, kept[i], len(want))
        assert np.array_equal(idx[int(h[i]): int(h[i + 1])].cpu().numpy().view(np.uint32), oracle_par.hull(p, want)), i
