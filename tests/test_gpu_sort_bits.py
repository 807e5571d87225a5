"""The library's stable sort orders by key bits [0, end_bit) alone and keeps the
others in their keys, whatever form the number of items selects (block up to
4,096 where the position fits beside the bits, cluster up to 98,304, whole
GPU)."""
import os
import subprocess

import pytest

from paper_2609_07577_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))
SIZES = [2, 65, 1000, 2048, 2049, 4096, 4097, 98304, 98305]


@pytest.mark.gpu
def test_bits_above_the_order(tmp_path):
    out = str(tmp_path / "sort_bits_check")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", _build.CSRC, os.path.join(HERE, "sort_bits_check.cu"),
                    os.path.join(_build.CSRC, "prims.cu"), "-o", out],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([out, *map(str, SIZES)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    lines = r.stdout.split("\n")[:-1]
    assert len(lines) == 5 * len(SIZES)
    assert [x for x in lines if not x.endswith(" ok")] == []
