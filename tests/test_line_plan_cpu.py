"""The division of a 1-D line among the CTAs of the cooperative stepping kernel: the cuts a walk over every node
gives, for plasma anywhere and rows of any weight, and in no time for lines that are much too long to fit."""
import ctypes
import os
import subprocess
import time

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2211_05647_gb300", "csrc")
SHIM = """#include "line_plan.cuh"
extern "C" int plan(int64_t nz, const int32_t *cells, int64_t ns, int ctas, double cost, int32_t *cut, int32_t *slot)
{
    const fp::LinePlan p = fp::line1d_plan(nz, std::vector<int32_t>(cells, cells + ns), ctas, cost);
    std::copy(p.cut.begin(), p.cut.end(), cut);
    std::copy(p.slot_cut.begin(), p.slot_cut.end(), slot);
    return (int)p.cut.size();
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)

    def call(nz, cells, ctas, cost):
        cells = np.ascontiguousarray(cells, dtype=np.int32)
        out = np.zeros((2, ctas + 1), dtype=np.int32)
        ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        n = lib.plan(ctypes.c_int64(nz), ptr(cells), ctypes.c_int64(len(cells)), ctas, ctypes.c_double(cost),
                     ptr(out[0]), ptr(out[1]))
        return out[0][:n].tolist(), out[1][:n].tolist()
    return call


def _walk(nz, cells, ctas, cost):
    n, ns = nz + 1, len(cells)
    want = max(1, min(ctas, n // 4))
    total = n + cost * ns
    cut, slot, acc, s = [0], [0], 0.0, 0
    for c in range(1, n + 1):
        acc += 1.0
        if s < ns and cells[s] == c - 1:
            acc += cost
            s += 1
        if len(cut) < want and acc >= total * len(cut) / want and 2 <= c <= nz - 1:
            cut.append(c)
            slot.append(s)
    return cut + [n], slot + [ns]


@pytest.mark.parametrize("seed", range(6))
def test_cuts_of_a_walk_over_the_nodes(plan, seed):
    rng = np.random.default_rng(seed)
    for _ in range(60):
        nz = int(rng.choice([3, 4, 7, 8, 9, int(rng.integers(10, 3000))]))
        inner = np.arange(1, nz)
        kind = rng.integers(4)
        cells = [inner[:0], inner, inner[rng.random(len(inner)) < 0.3], inner[len(inner) // 2:len(inner) // 2 + 9]][kind]
        ctas, cost = int(rng.choice([1, 2, 5, 152])), float(rng.choice([1, 4, 64, 1024]))
        assert plan(nz, cells, ctas, cost) == _walk(nz, cells.tolist(), ctas, cost), (nz, kind, ctas, cost)


def test_long_lines_are_planned_at_once(plan):
    plan(3, [1], 1, 1.0)
    t0 = time.perf_counter()
    cut, _ = plan(10 ** 9, np.arange(1, 1000), 152, 64.0)
    dt = time.perf_counter() - t0
    assert len(cut) == 153 and dt < 0.1, dt
