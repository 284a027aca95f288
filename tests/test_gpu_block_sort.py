"""Survivor sets that one block sorts as it builds their chains: the merge
rounds' ends (32, 64, ... 4096 and one off), keys that repeat, -0 beside +0,
sets of one and of several super-chunks in one batch, and calls whose later
kernels are not launched reporting a bad input -- hulls against the
oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402
import pointgen  # noqa: E402

pytestmark = pytest.mark.gpu


def ring(kind, n):
    rng = np.random.default_rng(n)
    if kind == "circle":      # every point survives the filter
        return pointgen.make_points("circle", n, seed=n)
    t = rng.integers(0, 64, n) / 64.0
    v = np.array([[4, 1], [3, 3], [1, 4], [-2, 3], [-4, 1], [-3, -3], [1, -4], [3, -2]], np.float64)
    k = rng.integers(0, 8, n)   # on the octagon's edges: runs of equal x, repeated points
    p = (v[k] * (1 - t[:, None]) + v[(k + 1) % 8] * t[:, None]).astype(np.float32)
    p[rng.integers(0, n, n // 8 + 1), 0] *= -0.0
    return p


@pytest.mark.parametrize("kind", ["circle", "edges"])
@pytest.mark.parametrize("n", [513, 543, 544, 545, 1023, 1024, 1025, 2047, 2049, 3333, 4064, 4095, 4096, 4097])
def test_single(kind, n):
    p = ring(kind, n)
    ws = ch.Workspace(n)
    idx, cnt = ch.convex_hull(torch.from_numpy(p).cuda(), ws)
    ws.check()
    assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), oracle.convex_hull(p)[2])


@pytest.mark.parametrize("kind", ["circle", "edges"])
def test_batch(kind):
    sizes = [1, 0, 5, 31, 32, 33, 4097, 64, 65, 511, 9000, 512, 513, 0, 1024, 2048, 4095, 4096, 12289, 2]
    sets = [ring(kind, n) if n else np.zeros((0, 2), np.float32) for n in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    ws = ch.Workspace(int(off[-1]), num_sets=len(sizes))
    idx, ho = ch.convex_hull_batched(torch.from_numpy(np.concatenate(sets)).cuda(), torch.from_numpy(off).cuda(), ws)
    ws.check()
    ho, idx = ho.cpu().numpy(), idx.cpu().numpy().view(np.uint32)
    for b, p in enumerate(sets):
        want = oracle.convex_hull(p)[2] if len(p) else np.zeros(0, np.uint32)
        assert np.array_equal(idx[ho[b]: ho[b + 1]], want), sizes[b]


@pytest.mark.parametrize("n", [3, 512, 513, 4096, 4097])
def test_bad_input_count(n):
    p = pointgen.make_points("circle", n, seed=1)
    p[n // 2, 1] = np.nan
    ws = ch.Workspace(n)
    idx = torch.zeros(n, dtype=torch.int32, device="cuda")
    cnt = torch.full((1,), 7, dtype=torch.int32, device="cuda")
    ch.ch_hull(torch.from_numpy(p).cuda(), idx, cnt, ws.buf)
    assert int(cnt.item()) == 0
    with pytest.raises(ch.CHError):
        ws.check()
