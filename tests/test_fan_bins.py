"""Points straight below the centre of a set: their pseudo-angle may round to
the bin before the first.  The rule for the table reads on the CPU
(tests/fan_bins.cu), what the bin is by the same arithmetic, and hulls of such
sets against the oracle."""
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="needs nvcc (host compilation only)")
def test_inner_bins(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "fan_bins")
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"), "-x", "cu",
                    os.path.join(HERE, "fan_bins.cu"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and "bins ok" in r.stdout, r.stdout


def test_bin_before_the_first():
    """A reciprocal within its documented one ulp leads to bin -1, and the
    sample of a batch's fan proofs asks inner_bin before it reads the table."""
    f = np.float32
    t = -f(1.5) * np.nextafter(f(1) / f(1.5), f(2))
    assert t < -1
    for q in (256, 2048, 6912):
        exact = float(t) * q + 2.0**23 + q
        v = f(exact)
        v = np.nextafter(v, f(0)) if float(v) > exact else v
        assert int(v.view(np.uint32)) - 0x4B000000 == -1
    src = open(os.path.join(ROOT, "paper_2303_10581_gb300", "csrc", "kgon.cu")).read()
    assert "return V + (int)(biased - kBinBias);" in src   # (a table in global memory: signed)
    assert len(re.findall(r"fan_bin_biased\(.*- kBinBias;", src)) == len(re.findall(r"= inner_bin\(b, ", src)) == 1


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1.0, 0.37, 2.0**100])
def test_second_level(scale):
    """Straight below the centre, within the circle's rounding: first-level
    survivors that the second level's table is read for."""
    torch = pytest.importorskip("torch")

    import oracle
    import paper_2303_10581_gb300 as ch

    rng = np.random.default_rng(3)
    th = rng.uniform(0, 2 * np.pi, 700_001)
    p = np.stack([np.cos(th), np.sin(th)], 1)
    k = np.arange(5000)
    p[7:5007] = np.stack([0.0 * k, -(1 - k * 2.0**-24)], 1)
    p[1:5] = [[1, 0], [-1, 0], [0, 1], [0, -1]]
    p = (scale * p).astype(np.float32)
    ws = ch.Workspace(len(p))
    ch.ch_tune_set("fan2_min_log2", 10)
    try:
        idx, cnt = ch.convex_hull(torch.from_numpy(p).cuda(), ws)
        ws.check()
    finally:
        ch.ch_tune_set("fan2_min_log2", 0)
    octs, kept, _, first = ch.ch_hull_counts(ws.buf, len(p))
    assert kept < first < octs   # both levels are at work
    assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), oracle.convex_hull(p)[2])


@pytest.mark.gpu
@pytest.mark.parametrize("n", [16_384, 20_011, 70_003])
@pytest.mark.parametrize("scale", [1.0, 0.37])
def test_hulls(n, scale):
    torch = pytest.importorskip("torch")

    import oracle
    import paper_2303_10581_gb300 as ch

    rng = np.random.default_rng(n)
    sets = []
    for _ in range(24):
        th, r = rng.uniform(0, 2 * np.pi, n), 1 - np.abs(rng.normal(0, 0.003, n))
        p = np.stack([r * np.cos(th), r * np.sin(th)], 1)
        below = n * np.arange(0, 256, 2) // 256   # half of the points that decide on the fan
        p[below] = np.stack([0 * below, -rng.uniform(0.25, 0.999, len(below))], 1)
        p[1:5] = [[1, 0], [-1, 0], [0, 1], [0, -1]]   # the centre is the origin
        sets.append((scale * p).astype(np.float32))
    d = torch.from_numpy(np.concatenate(sets)).cuda()
    ws = ch.Workspace(len(d), num_sets=len(sets))
    idx, ho = ch.convex_hull_batched(d, torch.arange(len(sets) + 1, device="cuda") * n, ws)
    ws.check()
    ho, idx = ho.cpu().numpy(), idx.cpu().numpy().view(np.uint32)
    for b, p in enumerate(sets):
        want = oracle.convex_hull(p)[2]
        assert np.array_equal(idx[ho[b]: ho[b + 1]], want), b
        if b < 4:
            one = ch.Workspace(n)
            i1, c1 = ch.convex_hull(torch.from_numpy(p).cuda(), one)
            one.check()
            assert np.array_equal(i1[: int(c1.item())].cpu().numpy().view(np.uint32), want)
