"""Connection rows that cannot grow on the way down: a pass goes on with
histograms from there when their memory ran out (the same partition as the
oracle's), returns any other failure, and leaves the handle usable."""
import os
import subprocess

import numpy as np
import pytest

import oracle
import snngen

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
OOM, CUDA = 3, 5


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    from paper_2609_07577_gb300 import _build
    _build.build()
    out = str(tmp_path_factory.mktemp("rows") / "rows_check")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    "-cudart", "shared", "-I", _build.CSRC, "-I", os.path.join(_build.ROOT, "include"),
                    os.path.join(HERE, "rows_check.cu"), _build.OUT,
                    "-Xlinker", "-rpath," + os.path.dirname(_build.OUT), "-o", out],
                   check=True, capture_output=True, text=True)
    return out


@pytest.mark.parametrize("name, code, nth", [(n, c, k) for n in ("cfg1s", "cfg2s") for c in (OOM, CUDA)
                                             for k in (0, 1, -1)] + [("cfg3s", OOM, -1)])
def test_rows_refused(harness, tmp_path, name, code, nth):
    """Rows are refused from the coarsest, the next and the finest level that
    has them on (cfg3s: after rounds on rows that enacted moves)."""
    hg = snngen.by_name(name)
    rho, cost, *_ = oracle.partition(hg, oracle.params_of(hg))
    net = str(tmp_path / "net")
    with open(net, "wb") as f:
        for a, t in ((hg.off, np.int64), (hg.pins, np.int32), (hg.w, np.int32)):
            f.write(np.ascontiguousarray(a, t).tobytes())
    size = os.path.getsize(net)
    r = subprocess.run([harness, *map(str, (hg.V, hg.E, hg.P, hg.omega, hg.delta, hg.phi)), net,
                        str(nth), str(code)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    whole, cut, again = ([int(x) for x in line.split()] for line in r.stdout.split("\n")[:3])
    got = np.fromfile(net, np.int32, offset=size).reshape(-1, hg.V)
    assert whole == again and whole[:2] == [0, cost] and whole[2] > 2
    if code == CUDA:
        assert cut[0] == CUDA and len(got) == 2
    else:
        # rows above, histograms from the refused level down
        assert cut == [0, cost, nth % whole[2], whole[3] + whole[2] - nth % whole[2]] and len(got) == 3
    assert all(np.array_equal(g, rho) for g in got)
