"""The library's prefix sums and stable sort (csrc/scan.cuh, csrc/prims.cu)
against the standard library's, at the sizes where the form changes (one
block, one cluster, whole GPU) and around the edges of their tiles."""
import os
import subprocess

import pytest

from paper_2609_07577_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))

# warp, block and sweep edges; 4096 / 4097 block sort, 98304 / 98305 cluster
# sort, 131072 / 131073 cluster scan; two levels of block sums
SIZES = [1, 2, 31, 33, 64, 65, 1000, 1024, 1025, 2048, 4096, 4097, 8192, 8193, 65536, 65537,
         98304, 98305, 131072, 131073, 300001]


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("prims") / "prims_check")
    cmd = [_build.nvcc(), *_build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
           "-I", _build.CSRC, os.path.join(HERE, "prims_check.cu"),
           os.path.join(_build.CSRC, "prims.cu"), "-o", out]
    subprocess.run(cmd, check=True, capture_output=True, text=True)
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("sizes", [SIZES, [20_000_003]], ids=["edges", "large"])
def test_scans_and_sort(harness, sizes):
    r = subprocess.run([harness, *map(str, sizes)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    lines = r.stdout.split("\n")[:-1]
    assert len(lines) == 8 * len(sizes)
    assert [x for x in lines if not x.endswith(" ok")] == []
