"""Chains of many survivors: runs of equal x about the ends of 32 points and
sequences about the ends of a warp's share, hulls against the oracle; and the
time of the chain stage against that of the sort's passes where nothing thins
the points out (8 10^6 circle points: 1.40 when every warp worked on a short
sequence too, 1.28 is what the stage took before both sides of a super-chunk
went at once)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402
from paper_2303_10581_gb300 import learned  # noqa: E402

pytestmark = pytest.mark.gpu


def hulls_agree(p):
    ws = ch.Workspace(len(p))
    d = torch.from_numpy(p).cuda()
    want = oracle.convex_hull(p)[2]
    idx, cnt = ch.convex_hull(d, ws)
    ws.check()
    assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), want)
    ws = ch.Workspace(3 * len(p), num_sets=3)
    off = torch.arange(4, device="cuda") * len(p)
    idx, ho = ch.convex_hull_batched(d.repeat(3, 1), off, ws)
    ws.check()
    ho, idx = ho.cpu().numpy(), idx.cpu().numpy().view(np.uint32)
    for b in range(3):
        assert np.array_equal(idx[ho[b]: ho[b + 1]], want), b


@pytest.mark.parametrize("run", [1, 2, 3, 4, 5, 8, 16, 17, 31, 32, 33, 63, 65, 100, 255, 257])
@pytest.mark.parametrize("n", [4001, 20_011])
def test_runs_of_equal_x(run, n):
    """A parabola's columns of `run` points, some equal, in any order: all of
    them beyond the polygon's chords."""
    rng = np.random.default_rng(run * n)
    x = np.arange(n) // run * run / n * 2 - 1
    p = np.stack([x, x * x + rng.integers(-2, 3, n) * 2.0 ** -20], 1).astype(np.float32)
    hulls_agree(rng.permutation(p))


@pytest.mark.parametrize("m", [1, 2, 3, 62, 63, 64, 65, 66, 127, 128, 129, 511, 512, 513, 1024, 1025])
@pytest.mark.parametrize("side", [1, -1])
def test_lengths_of_a_side(m, side):
    """m vertices on one side of a chord and a cloud next to its other side."""
    rng = np.random.default_rng(m)
    x = np.linspace(-1, 1, m + 2)
    arc = np.stack([x, side * (1 - x * x)], 1)
    low = np.stack([rng.uniform(-1, 1, 3000), -side * rng.uniform(0, 1e-3, 3000)], 1)
    hulls_agree(rng.permutation(np.concatenate([arc, low]).astype(np.float32)))


def test_time():
    n = 8_000_001
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    th = 2 * torch.pi * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    p = torch.stack([torch.cos(th), torch.sin(th)], 1).float().contiguous()
    dirs = torch.from_numpy(learned.directions(8)).cuda()
    ws = ch.Workspace(n)
    idx = torch.zeros(n, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    best = np.inf
    for _ in range(4):   # (the first one warms up)
        ch.ch_probe_start(max_launches=64)
        for _ in range(5):
            ch.ch_hull_kgon(p, dirs, idx, cnt, ws.buf)
        torch.cuda.synchronize()
        t = ch.ch_probe_stop()
        best = min(best, t["chain"][0] / t["sort_pass"][0])
    assert best <= 1.28, best
