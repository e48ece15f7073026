"""The sampled initial condition on a full grid (eps = 0) against the oracle's
vortex field, at the edges of the kernel's tiles: lattices below, at and
above the 256 columns of a tile, each row height, vortex counts around the
eight held at once, cores that wrap both seams.  Bound: a value's two
exponentials have arguments of at most 37 where the vorticity is above 1e-16
of a peak, so 37 * 2^-52 plus a few roundings, 1e-14, of the sum of the
peaks."""

import numpy as np
import pytest

from oracle import wrc_oracle as O
from paper_1604_08159_gb300 import binding as B
from paper_1604_08159_gb300 import workloads as W

from helpers import small_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_08159_gb300 import build
    build.build()
    B.load()


@pytest.mark.parametrize("n0,J,n", [(4, 1, 1), (16, 4, 8), (32, 4, 9), (32, 5, 3), (32, 6, 64)])
@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_MIXED])
def test_sampled_field_matches_oracle(n0, J, n, prec):
    prm = small_params(n0=n0, J=J, eps=0.0, prec=prec)
    rng = np.random.default_rng(n)
    v = W.Vortices(rng.uniform(-np.pi, np.pi, n), rng.uniform(-np.pi, np.pi, n), rng.uniform(-1.2, 1.2, n),
                   rng.uniform(0.1, 0.5, n))
    ref = O.vortex_field(prm.NJ, v.xc, v.yc, v.gamma, v.s).ravel()
    with B.Run(prm) as run:
        run.init_vortices(v)
        idx, om = run.active()
    assert np.array_equal(idx, np.arange(prm.NJ * prm.NJ))
    peak = np.sum(np.abs(v.gamma) / (np.pi * v.s ** 2))
    assert np.abs(om - ref).max() <= (1e-14 if prec == W.PREC_FP64 else 1e-14 + 2.0 ** -24) * peak
