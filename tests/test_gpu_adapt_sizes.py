"""The adaptation's passes over the lattice's flags on both sides of each
launch rule (one flag per thread up to 256^2, four beyond; the smallest
lattice), for every DD order: grid, ghosts and stencil levels bit-exact with
the oracle given the same field, and so the reconstruction through the
default tiles."""

import numpy as np
import pytest

from oracle import wrc_oracle as O
from paper_1604_08159_gb300 import binding as B
from paper_1604_08159_gb300 import workloads as W

from helpers import oracle_config, small_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_08159_gb300 import build
    build.build()
    B.load()


@pytest.mark.parametrize("n0,J,p", [(n0, J, p) for n0, J in [(4, 1), (16, 4), (4, 7), (16, 6)] for p in (2, 3, 4)] +
                         [(32, 6, 2)])   # several turns of every thread, and the reconstruction level by level
def test_grid_bit_exact(n0, J, p):
    prm = small_params(n0=n0, J=J, eps=1e-3, p=p)
    cfg = oracle_config(prm)
    v = W.random_field_params(seed=5, n=3)
    field = O.vortex_field(cfg.NJ, v.xc, v.yc, v.gamma, v.s)
    st = O.state_from_field(cfg, field)
    lev = O.levels(cfg.n0, cfg.J)
    jx, jy = O.stencil_levels(st.active, lev, cfg.J)
    with B.Run(prm) as run:
        run.init_field(field)
        act, gho, _ = run.masks()
        assert np.array_equal(act, st.active)
        assert np.array_equal(gho, O.ghost_set(st.active, jx, jy, cfg.J, cfg.p))
        gjx, gjy = run.stencil_levels()
        assert np.array_equal(gjx, jx[st.active]) and np.array_equal(gjy, jy[st.active])
        assert np.array_equal(run.field(B.FIELD_OMEGA), O.reconstruct(st.omega, st.active, cfg.J, p))
