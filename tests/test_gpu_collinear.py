"""Points that are exactly collinear, or an ulp off: on lines y = s x, on the
sides of rectangles, on coarse grids, also at scales where the products of the
exact tiers come near under- and overflow.  Survivors and hulls against the
oracle, in one set and in a batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402

pytestmark = pytest.mark.gpu

N = 20_011


def make(case, scale, nudge):
    rng = np.random.default_rng(17)
    kind, _, arg = case.partition("=")
    if kind == "line":
        x = rng.uniform(-1, 1, N) * 2.0 ** rng.integers(-8, 1, N)
        x = x.astype(np.float32).astype(np.float64)
        p = np.stack([x, float(arg) * x], 1)
    elif kind == "grid":
        m = int(arg)
        p = rng.integers(-m, m + 1, (N, 2)).astype(np.float64) + [0.0, 3.0 * m]
    else:   # a rectangle's sides
        t, k = rng.uniform(0, 1, N), rng.integers(0, 4, N)
        x = np.where(k < 2, t, k - 2.0)
        y = np.where(k < 2, k * 1.0, t)
        p = np.stack([x * 1.5 - 0.25, y * 0.75], 1)
    p = (p * scale).astype(np.float32)
    if nudge:
        q = np.nextafter(p, p + rng.integers(-1, 2, p.shape).astype(np.float32) * np.float32(scale), dtype=np.float32)
        p = np.where(rng.uniform(0, 1, (N, 1)) < 0.3, q, p)
    return p


CASES = ["line=1", "line=-1", "line=0.5", "line=4", "line=3", "line=0.37", "grid=3", "grid=100", "sides"]


@pytest.mark.parametrize("nudge", [False, True])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -70, 2.0 ** -120, 2.0 ** 62, 2.0 ** 118])
@pytest.mark.parametrize("case", CASES)
def test_filter_and_hull(case, scale, nudge):
    p = make(case, scale, nudge)
    ext = oracle.extremes(p)
    want = oracle.filter_points(p, ext)
    d = torch.from_numpy(p).cuda()
    ws = ch.Workspace(N, 2)
    idx, _, cnt = ch.filter_points(d, torch.from_numpy(ext.astype(np.int32)).cuda(), ws)
    ws.check()
    assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), want)
    _, _, hull = oracle.convex_hull(p)
    idx, cnt = ch.convex_hull(d, ws)
    ws.check()
    assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), hull)
    off = torch.tensor([0, 5000, N], dtype=torch.int64, device="cuda")
    idx, ho = ch.convex_hull_batched(d, off, ws)[:2]
    ws.check()
    h = ho.cpu().numpy()
    for b, (lo, hi) in enumerate([(0, 5000), (5000, N)]):
        _, _, hull = oracle.convex_hull(p[lo:hi])
        assert np.array_equal(idx[int(h[b]): int(h[b + 1])].cpu().numpy().view(np.uint32), hull)
