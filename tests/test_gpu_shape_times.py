"""Inputs whose shape once cost a stage far more than its points: the call's
time against that of the same call on as many points of a circle.  A case's
factor is the ratio of the time that the call took before the stage was made
for other shapes, and a quarter more; what it guards took 1.3 to 3 times the
factor."""
import math

import pytest

torch = pytest.importorskip("torch")

import paper_2303_10581_gb300 as ch  # noqa: E402

pytestmark = pytest.mark.gpu


def points(shape, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    th = 2 * math.pi * u
    if shape == "circle":
        x, y = torch.cos(th), torch.sin(th)
    elif shape == "horizontal":
        x, y = u, torch.full_like(u, 0.3)
    elif shape == "cauchy":   # a heavy-tailed cloud: its box's centre is far from nearly all points
        z = torch.randn((4, n), generator=g, device="cuda", dtype=torch.float64)
        x, y = z[0] / z[1], z[2] / z[3]
    elif shape == "diagonal":
        x = y = u
    elif shape == "grid":
        x = torch.floor(16 * u)
        y = torch.floor(16 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64))
    elif shape == "sides":
        k, t = torch.floor(4 * u), torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        x, y = torch.where(k < 2, t, k - 2), torch.where(k < 2, k, t)
    return torch.stack([x, y], 1).float().contiguous()


def call_us(call, p):
    n = len(p)
    ws = ch.Workspace(n)
    idx = torch.zeros(n, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    if call == "hull":
        def run():
            ch.ch_hull(p, idx, cnt, ws.buf)
    elif call == "filter":
        ext, sp = ch.extremes(p, ws), torch.zeros((n, 2), device="cuda")

        def run():
            ch.ch_filter(p, ext, idx, sp, cnt, ws.buf)
    else:   # a batch: sets of that many points
        m = int(call[5:])
        sets = -(-n // m)
        off = torch.clamp(torch.arange(sets + 1, device="cuda") * m, max=n)
        ws, ho = ch.Workspace(n, sets), torch.zeros(sets + 1, dtype=torch.int64, device="cuda")

        def run():
            ch.ch_hull_batched(p, off, idx, ho, ws.buf)
    for _ in range(3):
        run()
    best = math.inf
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            run()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 100)
    ws.check()
    return best


@pytest.mark.parametrize("call,shape,n,factor", [
    # all bins but two are empty: their neighbours are not searched for through the whole table
    ("hull", "horizontal", 300_007, 2.5),
    # nearly all points in a few bins: those inside the octagon are not binned
    ("hull", "cauchy", 3_000_001, 0.9),
    # points on the polygon's edges: exact signs without binary64
    ("filter", "sides", 300_007, 2.9),
    ("hull", "diagonal", 300_007, 4.0),
    ("batch60001", "sides", 12_000_200, 2.1),
    ("batch150001", "grid", 9_000_060, 1.4),
    ("batch150001", "diagonal", 9_000_060, 6.2),
])
def test_time(call, shape, n, factor):
    base, us = call_us(call, points("circle", n)), call_us(call, points(shape, n))
    assert us <= factor * base, (us, base)
