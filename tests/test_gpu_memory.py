"""Device memory of a job: the peak it reports counts everything its handle
holds (the library's pool never had more in use), and the footprint it was
admitted by bounds that peak."""
import os
import subprocess

import numpy as np
import pytest

import snngen

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    from paper_2609_07577_gb300 import _build
    _build.build()
    out = str(tmp_path_factory.mktemp("mem") / "mem_check")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    "-cudart", "shared", "-I", _build.CSRC, "-I", os.path.join(_build.ROOT, "include"),
                    os.path.join(HERE, "mem_check.cu"), _build.OUT,
                    "-Xlinker", "-rpath," + os.path.dirname(_build.OUT), "-o", out],
                   check=True, capture_output=True, text=True)
    return out


def _pairs(V, E, omega):
    rng = np.random.default_rng(V + E)
    a = rng.integers(0, V, E)
    b = (a + 1 + rng.integers(0, V - 1, E)) % V
    return snngen.Hypergraph("pairs", V, 2 * np.arange(E + 1, dtype=np.int64),
                             np.stack([a, b], 1).astype(np.int32).ravel(),
                             rng.integers(1, 9, E).astype(np.int32), omega, 1 << 28, 1 << 28)


# many vertices, many hyperedges, no pair that can merge (a partition a
# vertex), and jobs of the batched workload's families
NETS = {
    "vertices": lambda: _pairs(1_000_000, 1000, 64),
    "hyperedges": lambda: _pairs(2000, 1_000_000, 64),
    "cores_of_one": lambda: _pairs(100_000, 500_000, 1),
    "cores_of_two": lambda: _pairs(300_000, 1_000_000, 2),
    "layered": lambda: snngen.batch_jobs_one(0),
    "powerlaw": lambda: snngen.powerlaw(100_000, 65536, 8, 16384, 2.1, 0.7, seed=2, omega=4096, delta=16384,
                                        phi=65536, name="pl100k"),
    "conv": lambda: snngen.by_name("cfg2m"),
}


@pytest.mark.parametrize("name", sorted(NETS))
def test_peak_and_footprint(harness, tmp_path, name):
    hg = NETS[name]()
    net = str(tmp_path / "net")
    with open(net, "wb") as f:
        for a, t in ((hg.off, np.int64), (hg.pins, np.int32), (hg.w, np.int32)):
            f.write(np.ascontiguousarray(a, t).tobytes())
    r = subprocess.run([harness, *map(str, (hg.V, hg.E, hg.P, hg.omega, hg.delta, hg.phi)), net],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    footprint, peak, used = (int(x) for x in r.stdout.split())
    assert used <= peak + (1 << 20) and peak <= footprint
