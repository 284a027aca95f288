"""The two-pass filter's shares of tiles and its block-wide scatter where they
can go wrong: one tile and its edges, a share per block that differs by one
tile (2432 tiles are four for each of 608 blocks), rows that are empty, full
or ragged, both alignments of the points -- survivor lists against the
oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402
import pointgen  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [8, 31, 4095, 4096, 4097, 3 * 4096 + 1, 608 * 4096 - 1, 609 * 4096 + 2])
@pytest.mark.parametrize("dist", ["circle", "stripes"])
def test_survivors(dist, n, shift):
    rng = np.random.default_rng(n)
    p = pointgen.make_points("circle", n, seed=n)
    if dist == "stripes":   # whole rows, warps and tiles inside the polygon
        i = np.arange(n)
        p[((i // 512) % 3 == 0) | ((i // 32) % 5 == 1) | ((i // 4096) % 7 == 2)] *= 0.25
        p[rng.integers(0, n, n // 9)] *= 0.5
    buf = torch.zeros(n + 1, 2, device="cuda")
    d = buf[shift: shift + n]
    d.copy_(torch.from_numpy(p))
    ws = ch.Workspace(n)
    ext = oracle.extremes(p)
    want = oracle.filter_points(p, ext)
    for fused in (False, True):
        if fused:
            _, idx, pts, cnt = ch.extremes_and_filter(d, ws)
        else:
            idx, pts, cnt = ch.filter_points(d, torch.from_numpy(ext.astype(np.int32)).cuda(), ws)
        ws.check()
        m = int(cnt.item())
        got = idx[:m].cpu().numpy().view(np.uint32)
        assert np.array_equal(got, want)
        assert np.array_equal(pts[:m].cpu().numpy(), p[want])
