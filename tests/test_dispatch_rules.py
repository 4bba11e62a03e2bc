"""Rules of dispatch on the CPU: the header that holds them, compiled by the
host compiler, against the times that the lines were drawn from."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2205_14503_gb300", "csrc")

# (arcs, seeds, band width, largest weight): query times in ms on a GB300 with
# the full scan and with the tree-only scan; R-MAT graphs of degree 8 to 16
TREE_SCAN = [
    ((520 << 20, 182, 517, 1000), 6.19, 5.51), ((520 << 20, 2000, 129, 1000), 4.69, 3.28),
    ((520 << 20, 10000, 129, 1000), 5.68, 4.52), ((520 << 20, 10000, 32, 1000), 5.60, 4.15),
    ((520 << 20, 10000, 10, 20), 8.11, 9.21), ((520 << 20, 20000, 10, 20), 15.72, 19.15),
    ((520 << 20, 700, 2, 20), 4.30, 5.26), ((520 << 20, 10000, 2, 20), 6.92, 8.34),
    ((520 << 20, 300, 1, 20), 10.14, 10.73), ((520 << 20, 10000, 21, 40), 8.33, 9.70),
    ((520 << 20, 700, 5, 40), 4.42, 3.00), ((520 << 20, 10000, 5, 40), 6.08, 4.25),
    ((520 << 20, 10000, 41, 80), 8.42, 9.45), ((520 << 20, 10000, 10, 80), 5.94, 4.97),
    ((520 << 20, 10000, 83, 160), 8.84, 9.52), ((520 << 20, 10000, 83, 320), 6.64, 6.07),
    ((155 * 10**6, 10000, 10, 20), 4.65, 5.82), ((155 * 10**6, 10000, 41, 80), 3.99, 5.20),
    ((155 * 10**6, 10000, 20, 80), 3.32, 3.89), ((155 * 10**6, 10000, 82, 320), 3.21, 3.68),
    ((155 * 10**6, 182, 10, 80), 1.89, 1.60), ((155 * 10**6, 700, 41, 320), 2.20, 1.99),
    ((142 * 10**6, 2000, 253, 1000), 2.86, 2.61), ((142 * 10**6, 2000, 63, 1000), 2.32, 2.01),
    ((1060 << 20, 10000, 63, 1000), 11.01, 7.60), ((1060 << 20, 10000, 253, 1000), 13.11, 10.61),
    ((1060 << 20, 182, 1, 20), 12.81, 14.21), ((1060 << 20, 10000, 3, 60), 24.28, 26.43),
    ((1060 << 20, 10000, 5, 20), 12.98, 9.10), ((1060 << 20, 10000, 10, 160), 12.00, 8.46),
]


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, lib = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write('#include "rules.h"\nextern "C" int pays(uint64_t m, uint32_t k, uint32_t delta, uint32_t w) '
                "{ return stn::tree_scan_pays(m, k, delta, w); }\n"
                'extern "C" uint32_t step(uint32_t delta, uint32_t delta0, uint32_t w, int even) '
                "{ return stn::first_step(delta, delta0, w, even != 0); }\n")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", lib], check=True)
    so = ctypes.CDLL(lib)
    so.pays.argtypes = [ctypes.c_uint64, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_uint32]
    so.step.argtypes = [ctypes.c_uint32, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_int]
    so.step.restype = ctypes.c_uint32
    return so


@pytest.fixture
def pays(rules):
    return rules.pays


@pytest.mark.parametrize("call,full,tree", TREE_SCAN, ids=[str(c[0]) for c in TREE_SCAN])
def test_tree_scan_is_taken_where_it_is_the_faster_one(pays, call, full, tree):
    assert bool(pays(*call)) == (tree < full)


def test_tree_scan_lines(pays):
    assert not pays((1 << 27) - 1, 300, 50, 1000) and pays(1 << 27, 300, 50, 1000)
    assert not pays(1 << 32, 300, 3, 60) and pays(1 << 32, 300, 4, 60)
    assert not pays(1 << 32, 300, 1000, 1000)            # every arc light: nothing to spare
    assert not pays(1 << 32, 23000, 2**32 - 2, 2**32 - 1)


@pytest.mark.parametrize("delta0", [2, 64, 500, 2191])
def test_first_band_steps(rules, delta0):
    """The first band of even rows is reached in one step once it is narrower
    than an eighth of the default; without the split there is no step."""
    for delta in (1, delta0 // 16, delta0 // 8, delta0 // 8 + 1, delta0, 4 * delta0):
        if delta == 0:
            continue
        for even in (0, 1):
            assert rules.step(delta, delta0, delta - 1, even) == 0
            got = rules.step(delta, delta0, 10**6, even)
            if delta > delta0 // 8:
                assert got == max(2, delta0 // 64)
            else:
                assert got == (0 if even else max(2, delta // 8))
