"""A flow with every velocity times c, the viscosity times c and the time step
over c is the same flow: one step must give omega times c, for c = 2^140 and
2^-140 too, where the operator's and the vectors' magnitudes lie outside what
FP32 holds (the FP64 kernels use FP32 beside for what is small enough, and
fast paths for mid-range exponents).  Forms: few and many columns a block,
halves and words, the streaming one.  Bound: 1e-12 relative, the roundings of
a step whose intermediate paths differ."""

import numpy as np
import pytest

from paper_1604_08159_gb300 import binding as B
from paper_1604_08159_gb300 import workloads as W

from helpers import rel_l2, small_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_08159_gb300 import build
    build.build()
    B.load()


def step(c, **kw):
    v = W.random_field_params(11, 5)
    v = W.Vortices(v.xc, v.yc, v.gamma * c, v.s)
    prm = small_params(re=2000.0 / c, dt=1e-2 / c, **kw)
    prm.eps *= c
    with B.Run(prm) as run:
        run.init_vortices(v)
        run.step(1)
        run.sync()
        idx, om = run.active()
        return idx, om / c, run.krylov()


@pytest.mark.parametrize("kw", [dict(n0=16, J=3, eps=1e-3, m=20), dict(n0=16, J=4, eps=1e-4, m=31),
                                dict(n0=32, J=3, eps=0.0, m=10), dict(n0=32, J=3, eps=0.0, m=31),
                                dict(n0=32, J=4, eps=0.0, m=18)],
                         ids=["narrow", "ghosts", "halves", "words", "streaming"])
def test_step_scales(kw):
    idx, om, kr = step(1.0, **kw)
    for c in (2.0 ** 140, 2.0 ** -140):
        i2, o2, k2 = step(c, **kw)
        assert np.array_equal(i2, idx) and k2["k"] == kr["k"]
        assert rel_l2(o2, om) <= 1e-12
