"""Extremes that many points share: the lowest index whatever the tied points'
places in a sweep's tiles (2048 pairs of 512 threads), and the time of sets
whose points share them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402

pytestmark = pytest.mark.gpu

N = 700_001   # (more than one tile for some blocks)
PAIR, ROW, TILE = 2, 1024, 4096


def agree(p):
    for shift in (0, 1):   # 16- and 8-byte alignment
        b = torch.zeros((len(p) + shift, 2), device="cuda")
        b[shift:] = torch.from_numpy(p)
        ws = ch.Workspace(len(p))
        ext = torch.zeros(8, dtype=torch.int32, device="cuda")
        ch.ch_extremes(b[shift:], ext, ws.buf)
        ws.check()
        assert np.array_equal(ext.cpu().numpy().view(np.uint32), oracle.extremes(p))


@pytest.mark.parametrize("at", [
    [0, 1], [1, 0], [3, 2], [64, 2], [66, ROW], [2 * ROW + 4, ROW + 6], [3 * ROW, 62], [63, ROW - 1, 2 * ROW - 1],
    [TILE, TILE + 2, 5 * TILE], [TILE + 64, 7], [N - 1, 0], [N - 1, N - 2], [N - 3 * ROW, N - 1],
    [100 * TILE + 2, 100 * TILE + 4, 100 * TILE + 3 * ROW], [100 * TILE + 3 * ROW, 100 * TILE + 66],
    list(range(0, 64)), list(range(3 * ROW, 3 * ROW + 64)) + [2 * ROW + 63], list(range(5, N, 997)),
])
@pytest.mark.parametrize("slot", range(8))
def test_lowest_index(at, slot):
    rng = np.random.default_rng(slot)
    p = rng.uniform(-0.25, 0.25, (N, 2)).astype(np.float32)
    a = slot * np.pi / 4
    p[at] = np.round([np.cos(a), np.sin(a)]).astype(np.float32)
    agree(p)


@pytest.mark.parametrize("kind", ["equal", "horizontal", "vertical", "grid", "sides"])
@pytest.mark.parametrize("n", [5, 4095, 4097, N])
def test_sets(kind, n):
    rng = np.random.default_rng(n)
    p = rng.uniform(0, 1, (n, 2))
    if kind == "equal":
        p[:] = 0.25
    elif kind in ("horizontal", "vertical"):
        p[:, kind == "horizontal"] = 0.3
    elif kind == "grid":
        p = np.floor(3 * p)
    else:
        p[np.arange(n), rng.integers(0, 2, n)] = rng.integers(0, 2, n)
    agree(p.astype(np.float32))


def test_time():
    """3 10^6 equal points against as many normal ones: 1.9 when every lane
    that holds an extreme had its tile read again, 1.3 before that, 1.1
    measured; the limit is the 1.3 and a quarter more."""
    n = 3_000_001
    us = []
    for p in (torch.randn((n, 2), device="cuda"), torch.full((n, 2), 0.25, device="cuda")):
        ws, ext = ch.Workspace(n), torch.zeros(8, dtype=torch.int32, device="cuda")
        best = np.inf
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                ch.ch_extremes(p, ext, ws.buf)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        us.append(best)
    assert us[1] <= 1.63 * us[0], us
