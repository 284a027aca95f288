"""One workspace for calls on different n: the counters that kernels leave
zeroed for the next call stay where the next call looks for them (host check,
tests/reuse_check.cu), and the speculative sweep serves a set after the
workspace has held larger and smaller ones."""
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="needs nvcc (host compilation only)")
def test_self_resetting_records_do_not_move(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "reuse_check")
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"), "-x", "cu",
                    os.path.join(HERE, "reuse_check.cu"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and "reuse ok" in r.stdout, r.stdout


@pytest.mark.gpu
def test_speculation_on_a_used_workspace():
    import oracle
    import oracle_par
    import paper_2303_10581_gb300 as ch
    import pointgen

    sizes = [1 << 24, (1 << 22) + 3, 10_000_019, 1 << 22, 6_000_001]
    ws, served = ch.Workspace(max(sizes)), []
    for n, dist in zip(sizes, ("circle", "normal", "normal", "displaced", "normal")):
        p = pointgen.make_points(dist, n, seed=n % 1000)
        d = torch.from_numpy(p).cuda()
        idx, cnt = ch.convex_hull(d, ws)
        ws.check()
        want = oracle_par.hull(p, oracle_par.filter_points(p, oracle.extremes(p)))
        assert np.array_equal(idx[: int(cnt.item())].cpu().numpy().view(np.uint32), want), n
        fresh = ch.Workspace(n)
        ch.convex_hull(d, fresh)
        fresh.check()
        counts = ch.ch_hull_counts(fresh.buf, n)
        assert list(ch.ch_hull_counts(ws.buf, n)) == list(counts), n
        served.append(int(counts[2]))
    assert any(served), served
