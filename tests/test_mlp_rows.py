"""Batches of more than 2^31 / 68 samples: the MLP's kernels address their rows
in 64 bits (host check, tests/mlp_rows.cu), and by that function alone."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="needs nvcc (host compilation only)")
def test_row_offsets(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "mlp_rows")
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"), "-x", "cu",
                    os.path.join(HERE, "mlp_rows.cu"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and "rows ok" in r.stdout, r.stdout


def test_kernels_use_them():
    src = open(os.path.join(ROOT, "paper_2303_10581_gb300", "csrc", "mlp.cu")).read()
    assert not re.search(r"\[b \* ", src)
