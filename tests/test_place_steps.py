"""The arithmetic that the placement kernels run (csrc/place_items.cuh:
side_forces, on_lattice, reeval_cells, trd_cells; csrc/initial_items.cuh:
gain_corr_hedge) on the host, against the same sums pin by pin, which
tests/test_place_emul.py compares with the oracle: random lattices with empty
cores and one-row ones, pins repeated within a hyperedge, swaps ranked before
and after."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_07577_gb300", "csrc")


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    out = str(tmp_path_factory.mktemp("steps") / "libplace_steps.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "place_steps.cpp"), "-o", out], check=True)
    L = C.CDLL(out)
    i32, i64, vp = C.c_int32, C.c_int64, C.c_void_p
    L.steps_force.argtypes = [i32] + [vp] * 5 + [i32] * 3 + [vp] * 3
    L.steps_reeval_trd.argtypes = [vp, i64, i64, i64, i32, i32, i32, vp, vp, vp, i32, vp, vp]
    L.steps_gain.argtypes = [i32] + [vp] * 6 + [i32] * 3 + [vp] * 4
    for f in (L.steps_force, L.steps_reeval_trd, L.steps_gain):
        f.restype = None
    return L


def ptr(a):
    return a.ctypes.data_as(C.c_void_p)


def case(rng, repeats):
    n = int(rng.integers(2, 30))
    width, height = int(rng.integers(1, 9)), 1
    while width * height < n + int(rng.integers(0, 6)):
        height += 1
    ne = int(rng.integers(1, 25))
    pins = [rng.choice(n, int(rng.integers(1, min(n, 9) + 1)), replace=repeats) for _ in range(ne)]
    off = np.concatenate([[0], np.cumsum([len(p) for p in pins])]).astype(np.int64)
    hid = np.repeat(np.arange(ne), np.diff(off))
    pins = np.concatenate(pins).astype(np.int32)
    order = np.argsort(pins, kind="stable")
    voff = np.concatenate([[0], np.cumsum(np.bincount(pins, minlength=n))]).astype(np.int64)
    return n, width, height, off, pins, voff, hid[order].astype(np.int32), \
        rng.integers(0, 1 << 40, ne).astype(np.int64)


@pytest.mark.parametrize("repeats", [False, True])
def test_forces(steps, repeats):
    rng = np.random.default_rng(int(repeats))
    for _ in range(200):
        n, width, height, off, pins, voff, vinc, eta = case(rng, repeats)
        g = rng.choice(width * height, n, replace=False).astype(np.int32)
        for p in range(n):
            got, want = np.zeros(4, np.int64), np.zeros(4, np.int64)
            steps.steps_force(p, ptr(voff), ptr(vinc), ptr(off), ptr(pins), ptr(eta), n, width, height,
                              ptr(g), ptr(got), ptr(want))
            assert np.array_equal(got, want)


@pytest.mark.parametrize("repeats", [False, True])
def test_reevaluation_and_distances(steps, repeats):
    rng = np.random.default_rng(10 + int(repeats))
    for _ in range(200):
        n, width, height, off, pins, voff, vinc, eta = case(rng, repeats)
        nh = width * height
        g = rng.choice(nh, n, replace=False).astype(np.int32)
        rank = np.full(nh, 0x7fffffff, np.int32)
        mate = np.full(nh, -1, np.int32)
        p = rng.permutation(nh)   # disjoint swaps (any two cores), ranked in turn
        for r in range(int(rng.integers(1, nh // 2 + 1)) if nh > 1 else 0):
            a, b = p[2 * r], p[2 * r + 1]
            rank[a] = rank[b] = r
            mate[a], mate[b] = b, a
        for q in range(n):
            if mate[g[q]] < 0:
                continue
            for t in range(voff[q], voff[q + 1]):
                a = vinc[t]
                got, want = np.zeros(2, np.int64), np.zeros(2, np.int64)
                steps.steps_reeval_trd(ptr(pins), off[a], off[a + 1], int(rng.integers(off[a], off[a + 1])),
                                       n, nh, width, ptr(g), ptr(rank), ptr(mate), q, ptr(got), ptr(want))
                assert np.array_equal(got, want)


def test_gains_and_corrections(steps):
    rng = np.random.default_rng(20)
    for _ in range(300):
        n, _, _, off, pins, voff, vinc, eta = case(rng, False)
        pos = rng.permutation(n).astype(np.int32)
        lo, hi = sorted(int(x) for x in rng.choice(n + 1, 2, replace=False))
        mid = lo + (hi - lo + 1) // 2
        for x in range(n):
            if not lo <= pos[x] < hi:
                continue
            gg, gw = np.zeros(1, np.int64), np.zeros(1, np.int64)
            rg, rw = np.zeros(n, np.int64), np.zeros(n, np.int64)
            steps.steps_gain(x, ptr(voff), ptr(vinc), ptr(off), ptr(pins), ptr(eta), ptr(pos), lo, mid, hi,
                             ptr(gg), ptr(gw), ptr(rg), ptr(rw))
            assert gg[0] == gw[0] and np.array_equal(rg, rw)
