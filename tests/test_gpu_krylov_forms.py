"""The single-run Krylov launch in each of its forms (digit tables of at most
128 columns a block, wider ones as halves and as 64-bit integers, and the
FP64 kernel beyond) against the FP64 oracle: one step from the same state at
the sizes where the forms and their edges lie -- Krylov dimensions 1, 15 to
17 and 31 (row tiles of 8 and 16, one and two product depths), grids without
ghosts, blocks with ragged points and ghosts, every DD order, the mixed
mode.  Bounds as in the step parity tests: the grid and k equal, beta to
1e-12, omega to 1e-10 (mixed: omega 1e-6)."""

import numpy as np
import pytest

from oracle import wrc_oracle as O
from paper_1604_08159_gb300 import binding as B
from paper_1604_08159_gb300 import workloads as W

from helpers import oracle_config, rel_l2, small_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_08159_gb300 import build
    build.build()
    B.load()


CASES = [
    # n0, J, eps, m, p
    (4, 1, 0.0, 7, 2),         # 64 points, no ghost, two blocks
    (8, 3, 1e-3, 1, 2),        # one Krylov vector
    (16, 3, 1e-3, 15, 2),
    (16, 3, 1e-3, 16, 2),
    (16, 3, 1e-3, 17, 3),
    (16, 4, 1e-4, 31, 2),      # the largest dimension; ragged points and ghosts
    (16, 4, 1e-4, 31, 4),
    (32, 2, 0.0, 31, 2),       # 16384 points, 108 a block, no ghosts
    (32, 4, 1e-5, 23, 2),      # wide, digits as halves
    (32, 3, 0.0, 31, 2),       # 65536 points: 64-bit integers
    (32, 4, 0.0, 5, 2),        # 262144 points: integers, few rows
    (32, 4, 0.0, 18, 2),       # beyond the table: the FP64 kernel
]


@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_MIXED])
@pytest.mark.parametrize("n0,J,eps,m,p", CASES)
def test_step_matches_oracle(n0, J, eps, m, p, prec):
    prm = small_params(n0=n0, J=J, eps=eps, m=m, p=p, prec=prec, re=2000.0)
    cfg = oracle_config(prm)
    v = W.random_field_params(11, 5)
    st = O.initial_state(cfg, v.xc, v.yc, v.gamma, v.s)
    if prec == W.PREC_MIXED:   # FP32 values to start from
        st.omega = st.omega.astype(np.float32).astype(np.float64)
    with B.Run(prm) as run:
        run.set_grid(st.active, st.omega)
        st2, info = O.step(cfg, st)
        run.step(1)
        run.sync()
        kr = run.krylov()
        assert kr["k"] == info.k
        idx, om = run.active()
        ref = np.flatnonzero(st2.active.ravel())
        if prec == W.PREC_FP64:
            assert abs(kr["beta"] - info.beta) <= 1e-12 * info.beta
            assert np.array_equal(idx, ref)
            assert rel_l2(om, st2.omega[st2.active]) <= 1e-10
        else:
            common, ia, ib = np.intersect1d(idx, ref, assume_unique=True, return_indices=True)
            assert idx.size + ref.size - 2 * common.size <= max(2, 0.002 * ref.size)
            assert rel_l2(om[ia], st2.omega[st2.active][ib]) <= 1e-6
