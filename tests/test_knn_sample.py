"""How knn_exact samples rows and sizes its lists (csrc/knn_sample.h), compiled for the host: the rows at or below
the threshold fit the list of nearly every query wherever the filter is taken, simulated on random rows."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """#include "knn_sample.h"
extern "C" void plan(int64_t n, int64_t nq, int32_t dim, int32_t k, int64_t* out, double* expected) {
    const deg::SamplePlan p = deg::sample_plan(n, nq, dim, k);
    out[0] = p.stride, out[1] = p.ns, out[2] = p.ng, out[3] = p.group, out[4] = p.cap, out[5] = p.filter;
    *expected = p.expected;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("knn_sample")
    (d / "plan.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", os.path.join(ROOT, "paper_2307_10479_gb300", "csrc"),
                    str(d / "plan.cpp"), "-o", str(d / "plan.so")], check=True)
    lib = ctypes.CDLL(str(d / "plan.so"))

    def call(n, k, nq=200, dim=128):
        out, expected = (ctypes.c_int64 * 6)(), ctypes.c_double()
        lib.plan(ctypes.c_int64(n), ctypes.c_int64(nq), ctypes.c_int32(dim), ctypes.c_int32(k), out, ctypes.byref(expected))
        return dict(zip(("stride", "ns", "ng", "group", "cap", "filter"), out), expected=expected.value)
    return call


SIZES = [(16_400, 1_024), (20_000, 1_000), (40_000, 1_001), (66_000, 700), (300_000, 1_024), (1_000_000, 10), (1_000_000, 256),
         (4_000_000, 1_001), (6_000_000, 1_001), (8_000_000, 1_024), (12_000_000, 600), (12_000_000, 1_024), (30_000_000, 1_024)]


@pytest.mark.parametrize("n,k", SIZES)
def test_lists_hold_what_passes_the_threshold(plan, n, k):
    p = plan(n, k)
    rng = np.random.default_rng(n + k)
    over, counts = 0, []
    for _ in range(20):
        u = rng.random(p["ns"], dtype=np.float32)             # a sampled row's rank among all rows, as a share
        minima = np.minimum.reduceat(u, np.arange(0, p["ns"], p["group"]))
        t = np.partition(minima, k - 1)[k - 1]
        counts.append(t * n)
        over += counts[-1] > p["cap"]
    assert abs(np.mean(counts) / p["expected"] - 1) < 0.1
    if p["filter"]:
        assert over <= 10
        if p["cap"] < 8_192 or p["expected"] < 7_000:
            assert over == 0
    else:
        assert over >= 10 or p["expected"] > n / 4


@pytest.mark.parametrize("k", [1, 10, 100, 256, 257, 600, 1_001, 1_024])
def test_limits_over_all_sizes(plan, k):
    for n in sorted({int(1.07**e) + d for e in range(10, 310) for d in (-1, 0, 1)}):
        if not k <= n < 2**31 - 256:
            continue
        p = plan(n, k)
        assert p["ns"] == -(-n // p["stride"]) and p["ng"] == -(-p["ns"] // p["group"]) and p["group"] in (16, 64)
        assert p["ng"] <= 49_152 and 1_024 <= p["cap"] <= 8_192
        if p["filter"] and p["ng"] < k:
            assert n <= p["cap"]
        if 40 * k <= n <= 20_000_000:
            assert p["filter"]                                 # the usual sizes stay on the tensor cores
        few = plan(n, k, nq=1)
        assert few["filter"] == (p["filter"] and (k <= 256 or n > 65_536))
        assert {f: v for f, v in few.items() if f != "filter"} == {f: v for f, v in p.items() if f != "filter"}
        if k <= 256 and n <= 1_024:
            assert p["filter"]
