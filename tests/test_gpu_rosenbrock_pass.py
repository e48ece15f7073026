"""The Rosenbrock step's reductions at their edges (blocks of 128 points, at
most 304 of them): fewer points than a block, whole blocks, more points than
one turn of all blocks, and one to the largest number of vectors.  One step
against the FP64 oracle with the bounds of the form's other parity tests:
1e-10 on the field, 1e-12 on beta, the Krylov dimension equal."""

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


@pytest.mark.parametrize("n0,J,eps,m", [(4, 1, 0.0, 5), (16, 1, 0.0, 1), (16, 3, 1e-3, 31), (32, 3, 0.0, 4)])
def test_one_step(n0, J, eps, m):
    prm = small_params(n0=n0, J=J, eps=eps, m=m, scheme=W.SCHEME_ROSENBROCK)
    cfg = oracle_config(prm)
    v = W.fujiwhara_small().vortices
    st = O.initial_state(cfg, v.xc, v.yc, v.gamma, v.s)
    with B.Run(prm) as run:
        run.set_grid(st.active, st.omega)
        st, info = O.step_rosenbrock(cfg, st)
        run.step(1)
        run.sync()
        kr = run.krylov()
        assert kr["k"] == info.k
        assert abs(kr["beta"] - info.beta) <= 1e-12 * info.beta
        act, _, _ = run.masks()
        assert np.array_equal(act, st.active)
        idx, om = run.active()
        assert rel_l2(om, st.omega[st.active]) <= 1e-10
