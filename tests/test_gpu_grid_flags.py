"""wrc_set_grid takes any non-zero byte as an active point, on lattices whose
flag passes take one flag a thread (up to 256^2) and four: the grid, its
ghosts and stencil levels and a step from it are those of flags 0 and 1, bit
for bit."""

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


def stepped(prm, flags, omega):
    with B.Run(prm) as run:
        B.wrc_set_grid(run.h, np.ascontiguousarray(flags), np.ascontiguousarray(omega))
        act, gho, _ = run.masks()
        levels = run.stencil_levels()
        run.step(1)
        run.sync()
        return (act, gho, *levels, *run.active())


@pytest.mark.parametrize("n0,J", [(4, 2), (16, 3), (16, 5)])
def test_nonzero_flags_are_active_points(n0, J):
    prm = small_params(n0=n0, J=J, eps=1e-3)
    cfg = oracle_config(prm)
    v = W.fujiwhara_small().vortices
    st = O.initial_state(cfg, v.xc, v.yc, v.gamma, v.s)
    ones = st.active.astype(np.uint8)
    ref = stepped(prm, ones, st.omega)
    mixed = ones * np.random.default_rng(1).integers(1, 256, ones.shape).astype(np.uint8)
    for flags in (ones * np.uint8(255), ones * np.uint8(128), mixed):
        for got, want in zip(stepped(prm, flags, st.omega), ref):
            assert np.array_equal(got, want)
