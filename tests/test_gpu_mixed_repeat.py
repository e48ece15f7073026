"""Mixed runs on the lattices whose solve follows the level-by-level
reconstruction (beyond 1024^2), repeated on memory that earlier runs have
used: the same grid and values every time, bit for bit."""

import numpy as np
import pytest

from paper_1604_08159_gb300 import binding as B
from paper_1604_08159_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_08159_gb300 import build
    build.build()
    B.load()


@pytest.mark.parametrize("n0,J,tile", [(16, 5, "0"), (32, 6, None), (32, 7, None)])
def test_repeated_runs_are_bit_identical(n0, J, tile, monkeypatch):
    if tile is not None:
        monkeypatch.setenv("WRC_RECON_TILE", tile)
    v = W.fujiwhara_small().vortices
    prm = W.RunParams(n0=n0, J=J, eps=1e-4, re=5000.0, prec=W.PREC_MIXED, sgs=W.SGS_DYNAMIC, cs=0.17)
    out = []
    for _ in range(4):
        with B.Run(prm) as run:
            run.init_vortices(v)
            run.step(3)
            run.sync()
            out.append(run.active())
    for idx, om in out[1:]:
        assert np.array_equal(idx, out[0][0]) and np.array_equal(om, out[0][1])
