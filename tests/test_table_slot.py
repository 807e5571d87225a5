"""Where the histograms' tables put keys (csrc/table_slot.cuh): inserting
structured sets of ids by linear probing takes about as many probes as random
ids do, 1/2 (1 + 1/(1 - load)) on average (at most half as many again and 0.2),
and no key needs the 64 probes at which a block hands its vertex on."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_07577_gb300", "csrc")

SRC = r"""
#include "table_slot.cuh"
#include <vector>
// probes of all keys together, -1 when one needs more than 64
extern "C" int64_t insert_all(const int32_t* key, int n, uint32_t cap)
{
    std::vector<int32_t> t(cap, -1);
    int64_t probes = 0;
    for (int i = 0; i < n; i++) {
        uint32_t s = snn::table_slot(key[i], cap - 1);
        int p = 1;
        for (; t[s] != -1; p++, s = (s + 1) & (cap - 1))
            if (p > 64) return -1;
        t[s] = key[i];
        probes += p;
    }
    return probes;
}
"""


@pytest.fixture(scope="module")
def insert(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("slot")
    (d / "slot.cpp").write_text(SRC)
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "slot.cpp"),
                    "-o", str(d / "libslot.so")], check=True)
    L = C.CDLL(str(d / "libslot.so"))
    L.insert_all.restype = C.c_int64
    L.insert_all.argtypes = [C.c_void_p, C.c_int, C.c_uint32]

    def f(ids, cap):
        ids = np.ascontiguousarray(np.unique(ids), np.int32)
        got = L.insert_all(ids.ctypes.data, ids.size, cap)
        mean = 0.5 * (1 + 1 / (1 - ids.size / cap))
        return ids.size <= got <= (1.5 * mean + 0.2) * ids.size
    return f


# ids a stride apart: small ones, products of image sides and channels, and
# the Fibonacci numbers, whose multiples of the golden ratio are near whole
STRIDES = [1, 2, 3, 5, 7, 8, 13, 21, 27, 34, 55, 64, 89, 112, 144, 224, 233, 256, 377, 512, 610, 784, 987,
           1000, 1024, 1597, 1792, 2048, 2584, 3136, 4096, 4181, 6765, 10946, 12544, 16384, 17711, 28657,
           46368, 50176, 65536, 75025]


@pytest.mark.parametrize("cap, n", [(2048, 300), (2048, 1000), (16384, 3000), (16384, 8000)])
def test_progressions(insert, cap, n):
    bad = [(s, b) for s in STRIDES for b in (0, 1, 77777, 1 << 20)
           if not insert(b + s * np.arange(n, dtype=np.int64) % (1 << 30), cap)]
    assert bad == []


@pytest.mark.parametrize("channels_first", [False, True])
@pytest.mark.parametrize("side", [16, 28, 32, 47, 56, 64, 76, 89, 112, 128, 144, 224, 233, 256])
def test_image_windows(insert, side, channels_first):
    """Windows of 9 x 9 cells and 8 channels of a layer, channels last or first."""
    rng = np.random.default_rng(side)
    for _ in range(20):
        y, x, layer = rng.integers(0, side, 3)
        yy = (y + np.arange(9)) % side
        xx = (x + np.arange(9)) % side
        cell = (yy[:, None] * side + xx).ravel()
        c = np.arange(8)
        ids = c[:, None] * side * side + cell if channels_first else cell[:, None] * 8 + c
        assert insert(int(layer % 8) * 8 * side * side + ids.ravel(), 2048)
