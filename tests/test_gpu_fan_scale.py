"""The hull step's fan at any scale: a power-of-two scale keeps the structure of
the binary32 points, so the points that reach the sort are those of the plain
set (within a hundredth), up to boxes whose width overflows binary32.  Hulls
are the oracle's; one set with both fan levels, and a batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import fan_query  # noqa: E402
import oracle  # noqa: E402
import oracle_par  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402
import pointgen  # noqa: E402

pytestmark = pytest.mark.gpu

SCALES = [2.0 ** 21, 2.0 ** 100, 2.0 ** 126, 2.0 ** -21, 2.0 ** -50, 2.0 ** -100]


def scaled(p, s):
    return (p.astype(np.float64) * s).astype(np.float32)


def hull(p):
    d = torch.from_numpy(p).cuda()
    ws = ch.Workspace(len(p))
    idx, cnt = ch.convex_hull(d, ws)
    ws.check()
    return idx[: int(cnt.item())].cpu().numpy().view(np.uint32), ch.ch_hull_counts(ws.buf, len(p))


@pytest.mark.parametrize("dist", ["circle", "displaced"])
def test_single(dist):
    ch.ch_tune_set("fan2_min_log2", 16)
    try:
        p = pointgen.make_points(dist, (1 << 20) + 13, seed=41)
        want = oracle_par.hull(p, oracle_par.filter_points(p, oracle.extremes(p)))
        h, plain = hull(p)
        assert np.array_equal(h, want)
        assert plain[1] <= 0.3 * plain[0]
        for s in SCALES:
            h, c = hull(scaled(p, s))
            assert np.array_equal(h, want), s
            assert c[0] == plain[0] and abs(int(c[1]) - int(plain[1])) <= 0.01 * plain[1] + 8, (s, list(c), list(plain))
    finally:
        ch.ch_tune_set("fan2_min_log2", 0)


@pytest.mark.parametrize("s", [2.0 ** 127, 2.0 ** -138])
def test_ends_of_the_range(s):
    # a box whose width overflows; subnormal coordinates
    p = scaled(pointgen.make_points("displaced", 300_007, seed=43), s)
    h, c = hull(p)
    want = oracle_par.filter_points(p, oracle.extremes(p))
    assert c[0] == len(want) and np.array_equal(h, oracle_par.hull(p, want))
    assert c[1] <= 0.25 * c[0], list(c)


def test_batch():
    plain = [pointgen.make_points(d, n, seed=51 + i) for i, (d, n) in
             enumerate([("displaced", 60_001), ("circle", 200_003), ("displaced", 20_000), ("displaced", 300_001)])]
    sets = [q for p in plain for q in [p] + [scaled(p, s) for s in SCALES]]
    off = np.concatenate([[0], np.cumsum([len(p) for p in sets])]).astype(np.int64)
    d, o = torch.from_numpy(np.concatenate(sets)).cuda(), torch.from_numpy(off).cuda()
    ws = ch.Workspace(int(off[-1]), len(sets))
    idx, ho = ch.convex_hull_batched(d, o, ws)
    ws.check()
    at = fan_query.query(ws.buf.numel(), len(sets))[2]
    kept = ws.buf[at:at + 4 * len(sets)].cpu().numpy().view(np.uint32).astype(np.int64)
    h, k = ho.cpu().numpy(), 1 + len(SCALES)
    for i, p in enumerate(plain):
        want = oracle_par.hull(p, oracle_par.filter_points(p, oracle.extremes(p)))
        assert kept[i * k] <= 0.6 * len(p)
        for j in range(i * k, i * k + k):
            assert np.array_equal(idx[int(h[j]): int(h[j + 1])].cpu().numpy().view(np.uint32), want), (i, j)
            assert abs(kept[j] - kept[i * k]) <= 0.01 * kept[i * k] + 8, (i, j)
