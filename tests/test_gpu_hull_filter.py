"""The hull step's one-pass filter (octagon and fan) against the oracle where
it can go wrong: sets around the size that gets a fan and around a tile,
bins without samples, vertices at the ends of their bins, gaps of half a
turn, rings of repeated points, both alignments, the second level on few
directions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import oracle_par  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402
import pointgen  # noqa: E402

pytestmark = pytest.mark.gpu


def check(p, shift=0):
    buf = torch.from_numpy(np.concatenate([np.zeros((shift, 2), np.float32), p])).cuda()
    d = buf[shift:]
    ws = ch.Workspace(len(p))
    idx, cnt = ch.convex_hull(d, ws)
    ws.check()
    want = oracle_par.filter_points(p, oracle.extremes(p))
    c = ch.ch_hull_counts(ws.buf, len(p))
    assert c[0] == len(want) and c[1] <= c[0]
    assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), oracle_par.hull(p, want))
    return c


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [65_535, 65_536, 65_537, 69_631, 69_632, 69_633, 262_147])
def test_sizes(n, shift):
    check(pointgen.make_points("displaced", n, seed=n), shift)


def ring(angles, r=1.0, centre=(0.0, 0.0)):
    return np.stack([centre[0] + r * np.cos(angles), centre[1] + r * np.sin(angles)], 1).astype(np.float32)


CASES = ["few_directions", "bin_ends", "half_turn_gap", "arc_and_cluster", "repeated", "thin", "offset", "spiral"]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("case", CASES)
def test_cases(case, shift):
    rng = np.random.default_rng(11)
    n = 200_003
    r = 1.0 - np.abs(rng.normal(0, 0.02, n))
    if case == "few_directions":      # 97 directions: nearly every bin is empty
        p = ring(rng.integers(0, 97, n) * (2 * np.pi / 97), r)
    elif case == "bin_ends":          # directions of the bins' ends (pseudo-angles k * 4 / 28672) and next to them
        a = rng.integers(0, 28672, n) * (4.0 / 28672)
        q, t = np.floor(a).astype(int), a % 1.0
        x = np.where(q % 2 == 0, 1 - t, -t) * np.where(q < 2, 1, -1)
        y = np.where(q % 2 == 0, t, 1 - t) * np.where(q < 2, 1, -1)
        s = (r / np.hypot(x, y))[:, None]
        p = (np.stack([x, y], 1) * s).astype(np.float32)
        p = np.nextafter(p, p + rng.integers(-1, 2, p.shape).astype(np.float32), dtype=np.float32)
    elif case == "half_turn_gap":     # a half ring: a gap of half a turn seen from near its centre
        p = ring(rng.uniform(0, np.pi, n), r)
    elif case == "arc_and_cluster":   # an arc of a tenth of a turn and a far cluster
        p = np.concatenate([ring(rng.uniform(0, 0.6, n - 500), r[500:]), rng.normal(-3, 0.01, (500, 2)).astype(np.float32)])
    elif case == "repeated":          # 700 points, each many times
        p = ring(np.linspace(0, 6.28, 700))[rng.integers(0, 700, n)]
    elif case == "thin":              # a thin rotated ellipse
        p = pointgen.make_family("ellipse", n, seed=12)
    elif case == "offset":            # far from the origin: differences to the centre lose bits
        p = ring(rng.uniform(0, 2 * np.pi, n), r, (3.0e4, -7.0e3))
    else:                             # radii grow with the angle: long radial edges
        th = rng.uniform(0, 2 * np.pi, n)
        p = ring(th, 0.3 + th / 7)
    check(p, shift)


def test_second_level_with_few_directions():
    rng = np.random.default_rng(13)
    n = (1 << 19) + 77
    p = ring(rng.integers(0, 5000, n) * (2 * np.pi / 5000) + 1e-9 * rng.normal(0, 1, n))
    ch.ch_tune_set("fan2_min_log2", 10)
    try:
        check(p)
    finally:
        ch.ch_tune_set("fan2_min_log2", 0)
