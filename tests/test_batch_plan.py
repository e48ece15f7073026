"""The plan of a batched Krylov launch (host code, compiled here with g++):
every problem's blocks once, on different blocks of the launch; the blocks of
a problem of several blocks have the same problems before it (they meet at
its barriers and must reach it together); and no block with far more than its
share of the points, also where the problems outnumber the blocks or one is
much larger than the rest."""

import ctypes
import pathlib
import shutil
import subprocess

import numpy as np
import pytest

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_1604_08159_gb300" / "csrc"
SRC = '''
#include "batch_plan.h"
extern "C" int plan(const long long* n, int M, long long least, int sms, int* items, int* off) {
    std::vector<int> i, o;
    wrc::krylov_batch_plan(std::vector<long long>(n, n + M), least, sms, i, o);
    std::copy(i.begin(), i.end(), items);
    std::copy(o.begin(), o.end(), off);
    return (int)o.size() - 1;
}
'''


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(d / "plan.cpp"), "-o",
                    str(d / "plan.so")], check=True)
    lib = ctypes.CDLL(str(d / "plan.so"))

    def call(n, least=128, sms=152):
        n = np.ascontiguousarray(n, dtype=np.int64)
        items = np.zeros(3 * (n.size + 8 * sms + 8 * n.size), dtype=np.int32)
        off = np.zeros(sms + 1, dtype=np.int32)
        blocks = lib.plan(n.ctypes.data_as(ctypes.c_void_p), n.size, ctypes.c_longlong(least), sms,
                          items.ctypes.data_as(ctypes.c_void_p), off.ctypes.data_as(ctypes.c_void_p))
        assert 1 <= blocks <= sms
        return [[tuple(items[3 * i:3 * i + 3]) for i in range(off[b], off[b + 1])] for b in range(blocks)]

    return call


def check(blocks, n):
    at = {}
    for b, work in enumerate(blocks):
        assert work
        for pos, (q, i, nb) in enumerate(work):
            at.setdefault(q, []).append((i, nb, [w[0] for w in work[:pos]]))
    assert sorted(at) == list(range(len(n)))
    for q, parts in at.items():
        nb = parts[0][1]
        assert sorted(p[0] for p in parts) == list(range(nb)) and all(p[1] == nb for p in parts)
        assert all(p[2] == parts[0][2] for p in parts)
    return max(sum(n[q] / nb for q, _, nb in work) for work in blocks)


@pytest.mark.parametrize("n,most", [
    ([5000], 1.05), ([66000, 66000], 1.05), (list(range(9000, 17000, 170)), 1.5),
    ([2800] * 152, 1.05), ([2800] * 153, 1.7), ([9100] * 160, 1.5), ([2800] * 400, 1.2),
    ([72000] + [2800] * 199, 1.6), ([72000] + [2800] * 151, 1.6), ([30000, 28000, 72000] + [1200] * 600, 1.6),
])
def test_balanced(plan, n, most):
    assert check(plan(n, 128), n) <= most * max(sum(n) / 152, 128)   # (no share below 128 points)


def test_any_sizes(plan):
    rng = np.random.default_rng(0)
    for _ in range(200):
        m, sms = int(rng.integers(1, 500)), int(rng.choice([1, 2, 7, 132, 152]))
        n = np.exp(rng.uniform(np.log(16), np.log(1e5), m)).astype(np.int64)
        check(plan(n, int(rng.choice([64, 128, 1024, 1 << 20])), sms), n)
    check(plan([0, 0, 5]), [0, 0, 5])
