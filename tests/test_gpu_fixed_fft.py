"""The FP64 streamfunction solve's block floating point: every value of a
transform shares one exponent, so a field times a power of two must give psi
times that power, bit for bit (each rounding commutes with the scaling as
long as nothing underflows), also where the exponents leave the range that an
addition to the exponent field serves; and a zero field gives psi = 0.  Sizes:
every first radix (none, 2, 4) at 4 and at 8 values per thread."""

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


def psi_of(n0, J, f):
    with B.Run(W.RunParams(n0=n0, J=J, eps=0.0, re=5000.0)) as run:
        run.init_field(f)
        run.freeze()
        return run.field(B.FIELD_PSI)


@pytest.mark.parametrize("n0,J", [(4, 1), (16, 2), (16, 3), (16, 5), (32, 5), (32, 6), (32, 7)])
def test_solve_scales_by_powers_of_two(n0, J):
    n = n0 << J
    f = np.random.default_rng(n).normal(size=(n, n))
    psi = psi_of(n0, J, f)
    assert np.isfinite(psi).all() and np.abs(psi).max() > 0
    for k in (400, -400, -880):
        assert np.array_equal(psi_of(n0, J, f * 2.0 ** k), psi * 2.0 ** k), k
    assert not psi_of(n0, J, np.zeros((n, n))).any()


@pytest.mark.parametrize("case,tile", [(dict(n0=8, J=4, eps=1e-3, p=4), "0"), (dict(n0=16, J=5, eps=1e-4, p=2), "0"),
                                       (dict(n0=16, J=7, eps=1e-4, p=2), None)])
def test_repeated_runs_are_bit_identical(case, tile, monkeypatch):
    """The solve right after the level-by-level reconstruction (the default
    beyond 1024^2), on memory that earlier runs have used: the same values
    every time."""
    if tile is not None:
        monkeypatch.setenv("WRC_RECON_TILE", tile)
    v = W.fujiwhara_small().vortices
    out = []
    for _ in range(4):
        with B.Run(W.RunParams(re=5000.0, **case)) as run:
            run.init_vortices(v)
            run.step(3)
            run.sync()
            out.append(run.active())
    for idx, om in out[1:]:
        assert np.array_equal(idx, out[0][0]) and np.array_equal(om, out[0][1])
