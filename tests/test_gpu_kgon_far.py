"""The K-direction polygon of a heavy-tailed cloud: binary32 cannot place most
of its points, next to the centre of a polygon of four far vertices.  Vertices
and survivors against the oracle, and the time of the test against that of the
polygon's sweep (4.2 with the tiers after binary32 in line at every edge, 3.4
before that, 3.6 measured; the limit is the 3.4 and 15 percent)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402
from paper_2303_10581_gb300 import learned  # noqa: E402

pytestmark = pytest.mark.gpu


def cauchy(n):
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    torch.rand((2, n), generator=g, device="cuda", dtype=torch.float64)   # (this cloud's polygon has four vertices)
    z = torch.randn((4, n), generator=g, device="cuda", dtype=torch.float64)
    return torch.stack([z[0] / z[1], z[2] / z[3]], 1).float().contiguous()


def filter_call(p, K):
    n = len(p)
    ws = ch.Workspace(n)
    idx = torch.zeros(n, dtype=torch.int32, device="cuda")
    cnt, ext = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(K, dtype=torch.int32, device="cuda")
    sp = torch.zeros((n, 2), device="cuda")
    dirs = torch.from_numpy(learned.directions(K)).cuda()
    return lambda: ch.ch_filter_kgon(p, dirs, ext, idx, sp, cnt, ws.buf), ext, idx, cnt


@pytest.mark.parametrize("K", [8, 16, 64])
def test_survivors(K):
    p = cauchy(30_011)
    call, ext, idx, cnt = filter_call(p, K)
    call()
    h, dirs = p.cpu().numpy(), learned.directions(K)
    assert np.array_equal(ext.cpu().numpy().view(np.uint32), oracle.kgon_extremes(h, dirs))
    assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), oracle.kgon_filter(h, dirs))


def test_time():
    call = filter_call(cauchy(3_000_001), 64)[0]
    best = np.inf
    for _ in range(4):   # (the first one warms up)
        ch.ch_probe_start(max_launches=64)
        for _ in range(5):
            call()
        torch.cuda.synchronize()
        t = ch.ch_probe_stop()
        best = min(best, t["filter"][0] / t["extremes"][0])
    assert best <= 3.9, best
