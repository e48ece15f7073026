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


FORMS = [dict(n0=16, J=3, eps=1e-3, m=20), dict(n0=32, J=3, eps=0.0, m=31), dict(n0=32, J=4, eps=0.0, m=18)]


@pytest.mark.parametrize("kw", FORMS, ids=["narrow", "words", "streaming"])
def test_far_first_vector(kw):
    """u.z of the unscaled first vector would have the scale c^5."""
    idx, om, kr = step(1.0, **kw)
    for c in (2.0 ** 230, 2.0 ** -230):
        i2, o2, k2 = step(c, **kw)
        assert np.array_equal(i2, idx) and k2["k"] == kr["k"]
        assert abs(k2["beta"] / (c * c) - kr["beta"]) <= 1e-12 * kr["beta"]
        assert rel_l2(o2, om) <= 1e-12


@pytest.mark.parametrize("kw", FORMS, ids=["narrow", "words", "streaming"])
def test_mixed_step_scales(kw):
    """z = A u of the unscaled first vector, c^3, would leave FP32; 2^-55 still
    keeps b's largest entries normal.  Bound: the mixed mode's 1e-6."""
    idx, om, kr = step(1.0, prec=W.PREC_MIXED, **kw)
    for c in (2.0 ** 55, 2.0 ** -55):
        i2, o2, k2 = step(c, prec=W.PREC_MIXED, **kw)
        common, ia, ib = np.intersect1d(i2, idx, assume_unique=True, return_indices=True)
        assert i2.size + idx.size - 2 * common.size <= max(2, 0.002 * idx.size)
        assert k2["k"] == kr["k"]
        assert rel_l2(o2[ia], om[ib]) <= 1e-6


def test_one_block_members_scale():
    """Members of one block each, whose sums stay within the block."""
    v = W.random_field_params(11, 5)

    def members(c):
        prm = small_params(re=2000.0 / c, dt=1e-2 / c, n0=8, J=3, eps=1e-3 * c, prec=W.PREC_MIXED)
        with B.Ensemble([prm] * 160) as ens:
            for mem in ens.members:
                mem.init_vortices(W.Vortices(v.xc, v.yc, v.gamma * c, v.s))
            ens.step(1)
            ens.sync()
            return [mem.active() for mem in ens.members[::40]]

    for (i0, o0), (i1, o1) in zip(members(1.0), members(2.0 ** -55)):
        common, ia, ib = np.intersect1d(i1, i0, assume_unique=True, return_indices=True)
        assert i1.size + i0.size - 2 * common.size <= 2
        assert rel_l2(o1[ia] * 2.0 ** 55, o0[ib]) <= 1e-6
