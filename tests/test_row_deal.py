"""The dealing of a connection row's marked chunks to a warp's lanes that
k_dense_best runs (csrc/row_items.cuh), on the host: every quad of a marked
chunk goes to exactly one lane, each lane's in increasing order, none outside;
and the proposal found that way equals the whole row's
(tests/test_row_scan_host.py's scan)."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_row_scan_host import _lane_visit, _reduce, chunk_width, scan_full

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_07577_gb300", "csrc")


@pytest.fixture(scope="module")
def deal(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    out = str(tmp_path_factory.mktemp("row") / "librow.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "row_steps.cpp"), "-o", out], check=True)
    L = C.CDLL(out)
    L.row_deal.argtypes = [C.c_uint64, C.c_int32, C.c_int, C.c_void_p, C.c_int]

    def f(mask, cw):
        buf = np.zeros(64 * max(1, cw // 4), np.int64)
        return [buf[:L.row_deal(mask, cw, lane, buf.ctypes.data, buf.size)].tolist() for lane in range(32)]
    return f


# chunks of 8, 16, 32, 64 and 256 quads: four, two and one a step, two and
# eight steps a chunk
@pytest.mark.parametrize("cw", [32, 64, 128, 256, 1024])
def test_every_marked_quad_once(deal, cw):
    rng = np.random.default_rng(cw)
    cq = cw // 4
    masks = [0, 1, 1 << 63, (1 << 64) - 1, 0b1011] + \
        [int(rng.integers(0, 1 << 62)) & int(rng.integers(0, 1 << 62)) for _ in range(50)]
    for mask in masks:
        lanes = deal(mask, cw)
        want = [c * cq + q for c in range(64) if mask >> c & 1 for q in range(cq)]
        assert sorted(q for qs in lanes for q in qs) == want
        assert all(a < b for qs in lanes for a, b in zip(qs, qs[1:]))


@pytest.mark.parametrize("K", [1, 31, 200, 1000, 2052, 4536, 9011, 20000])
@pytest.mark.parametrize("nonpos", [0, 1])
def test_dealt_scan_equals_full_scan(deal, K, nonpos):
    rng = np.random.default_rng(2 * K + nonpos)
    Kp = (K + 3) & ~3
    cw = chunk_width(Kp)
    for _ in range(15):
        row = np.zeros(Kp, np.int64)
        for _ in range(int(rng.integers(0, 5))):
            a = int(rng.integers(0, K))
            b = min(K, a + int(rng.integers(1, 12)))
            row[a:b] = rng.integers(0, 6, size=b - a)
        T = int(rng.integers(-2, 5))
        ok = rng.random(Kp) < 0.8
        mask = 0
        for c in {int(p) // cw for p in np.flatnonzero(row)} | {int(rng.integers(0, (Kp + cw - 1) // cw))}:
            mask |= 1 << c
        lanes = []
        for qs in deal(mask, cw):
            bs, bk = 0, -1
            for q in qs:
                for p in range(4 * q, min(4 * q + 4, K)):
                    bs, bk = _lane_visit(bs, bk, p, row[p], T, ok[p], nonpos)
            lanes.append((bs, bk))
        assert _reduce(lanes) == scan_full(row, K, T, ok, nonpos)
