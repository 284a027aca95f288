"""The sort's ranking where a digit of the keys has few values (one, the most
that go by match.any, one more, a full digit), in one set and in a batch:
hulls against the oracle, on sets that no fan thins out."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2303_10581_gb300 as ch  # noqa: E402

pytestmark = pytest.mark.gpu

FEW = 8   # kFewDigits


def arc(values, n, seed):
    """Points of a circle's right third whose x has `values` values in its low 8 bits and one in the next 8."""
    rng = np.random.default_rng(seed)
    base = np.floor(rng.uniform(0.5, 1.0, n) * 256) / 256
    x = (base + rng.integers(0, values, n) * 2.0 ** -24).astype(np.float32)
    y = (np.sqrt(np.maximum(0.0, 1 - x.astype(np.float64) ** 2)) * rng.choice([-1, 1], n)).astype(np.float32)
    assert len(np.unique(x.view(np.uint32) & 255)) == values
    return np.stack([x, y], 1)


@pytest.mark.parametrize("values", [1, FEW, FEW + 1, 256])
def test_hulls(values):
    sizes = [12_000, 4_097, 16_000, 5_000]
    sets = [arc(values, n, n) for n in sizes]
    p = arc(values, 30_001, 5)
    want = oracle.convex_hull(p)[2]
    idx, cnt = ch.convex_hull(torch.from_numpy(p).cuda())
    assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), want)
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)).cuda()
    idx, ho = ch.convex_hull_batched(torch.from_numpy(np.concatenate(sets)).cuda(), off)
    h = ho.cpu().numpy()
    for b, q in enumerate(sets):
        want = oracle.convex_hull(q)[2]
        assert np.array_equal(idx[int(h[b]): int(h[b + 1])].cpu().numpy().view(np.uint32), want), b
