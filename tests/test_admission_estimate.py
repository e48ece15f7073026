"""The admission estimate is a figure that callers set their budgets by: a
request that fitted a budget fits it with every later form of the kernels, and
one that did not does not.  Bytes for lattices of 8^2 to 4096^2 (n0, J), both
precisions, Krylov dimensions and DD orders (half the order)."""

import pytest

from paper_1604_08159_gb300 import binding as B
from paper_1604_08159_gb300 import build as BLD
from paper_1604_08159_gb300 import workloads as W

# (n0, J, prec, m, p): bytes
EST = {
    (4, 1, 0, 20, 2): 3451308.0,
    (4, 1, 0, 30, 2): 3660188.0,
    (4, 1, 0, 31, 4): 6630284.0,
    (4, 1, 1, 20, 2): 3198508.0,
    (4, 1, 1, 30, 2): 3304988.0,
    (4, 1, 1, 31, 4): 6264844.0,
    (16, 3, 0, 20, 2): 12880940.0,
    (16, 3, 0, 30, 2): 14441500.0,
    (16, 3, 0, 31, 4): 30522892.0,
    (16, 3, 1, 20, 2): 10434604.0,
    (16, 3, 1, 30, 2): 11216924.0,
    (16, 3, 1, 31, 4): 27220492.0,
    (32, 3, 0, 20, 2): 19728940.0,
    (32, 3, 0, 30, 2): 21740060.0,
    (32, 3, 0, 31, 4): 41995276.0,
    (32, 3, 1, 20, 2): 15323692.0,
    (32, 3, 1, 30, 2): 16331292.0,
    (32, 3, 1, 31, 4): 36486156.0,
    (32, 5, 0, 20, 2): 159019564.0,
    (32, 5, 0, 30, 2): 170246684.0,
    (32, 5, 0, 31, 4): 279897100.0,
    (32, 5, 1, 20, 2): 115249708.0,
    (32, 5, 1, 30, 2): 120865308.0,
    (32, 5, 1, 31, 4): 229954572.0,
    (32, 7, 0, 20, 2): 2387227180.0,
    (32, 7, 0, 30, 2): 2545910300.0,
    (32, 7, 0, 31, 4): 4085883916.0,
    (32, 7, 1, 20, 2): 1713771052.0,
    (32, 7, 1, 30, 2): 1793114652.0,
    (32, 7, 1, 31, 4): 3325154316.0,
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    BLD.build()


@pytest.mark.parametrize("key", EST)
def test_estimate(key):
    n0, J, prec, m, p = key
    cfg = B.make_config(W.RunParams(n0=n0, J=J, eps=1e-4, re=5000.0, m=m, p=p, prec=prec))
    assert B.wrc_server_estimate(cfg) == EST[key]
