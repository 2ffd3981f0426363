"""The FP32 kernels' sums of squares (csrc/common.cuh, compiled for the host): a thread's plain
accumulator is folded before it has added more rows than FP64-summed threads of 108 rows
have, and pairs of FP32 across threads lose nothing beside what a thread's FP32 products do."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("sums") / "sums_check")
    subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2211_15383_gb300", "csrc"),
                    os.path.join(HERE, "sums_check.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return [[float(v) for v in line.split()] for line in out.splitlines()]


def test_accuracy(rows):
    assert [r[0] for r in rows] == [1, 63, 64, 65, 216, 862]
    for n, folded, plain, split in rows:
        # up to 64 rows the two forms add alike, and differ by the pairs' rounding only; beyond,
        # an RMS over 96 trials is known to 1 / sqrt(2 96) = 7 %: three of these
        assert folded <= plain * (1.001 if n <= 64 else 1.22), (n, folded, plain)
        # 84 additions of a pair with 2^-48 each; FP32 accumulators leave 1e-9 and more of the sum
        assert split < 84 * 2.0 ** -48 and split < 1e-3 * plain, (n, split, plain)
