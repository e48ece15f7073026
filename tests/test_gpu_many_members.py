"""Ensembles of more members than the device has SMs: blocks that take several
members in turn, groups of blocks that share them, and one member much larger
than the rest, on blocks of its own.  Every member after three steps is the
member run alone: the same grid, omega to 1e-10 (the parity bound)."""

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


def pair(r):
    return W.Vortices(np.array([-0.6, 0.6]), np.zeros(2), np.array([1.0, r]), np.full(2, 0.3))


SMALL = [(small_params(n0=8, J=3), pair(r)) for r in (1.0, 0.8, 0.6)]
EQUAL = [(small_params(n0=16, J=3), pair(r)) for r in (1.0, 0.8, 0.6)]
LARGE = (small_params(n0=32, J=4, eps=1e-6), W.random_field_params(11, 6))


@pytest.mark.parametrize("kinds,count,large", [(EQUAL, 153, False), (SMALL, 400, False), (SMALL, 199, True)])
def test_every_member_as_alone(kinds, count, large):
    kinds = kinds + [LARGE] if large else kinds
    which = [q % 3 for q in range(count)] + ([3] if large else [])
    alone = []
    for prm, v in kinds:
        with B.Run(prm) as run:
            run.init_vortices(v)
            run.step(3)
            run.sync()
            alone.append(run.active())
    with B.Ensemble([kinds[w][0] for w in which]) as ens:
        for mem, w in zip(ens.members, which):
            mem.init_vortices(kinds[w][1])
        ens.step(3)
        ens.sync()
        for mem, w in zip(ens.members, which):
            idx, om = mem.active()
            assert np.array_equal(idx, alone[w][0])
            assert rel_l2(om, alone[w][1]) <= 1e-10
