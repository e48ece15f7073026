"""The mixed mode's streamfunction solve in a step, on lattices where each
output has blocks of its own (up to 512^2) and beyond, with and without the
strain: two steps against the FP64 oracle with the mixed mode's bounds (1e-6
on the vorticity over the points active in both, at most 0.2% of the grid
different)."""

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


@pytest.mark.parametrize("n0,J", [(16, 2), (16, 5), (16, 6)])
@pytest.mark.parametrize("sgs", [dict(), dict(sgs=W.SGS_DYNAMIC, cs=0.17, re=2000.0)], ids=["uv", "strain"])
def test_mixed_steps(n0, J, sgs):
    prm = small_params(n0=n0, J=J, eps=1e-3, m=12, prec=W.PREC_MIXED, **sgs)
    cfg = oracle_config(prm)
    v = W.fujiwhara_small().vortices
    st = O.initial_state(cfg, v.xc, v.yc, v.gamma, v.s)
    with B.Run(prm) as run:
        run.set_grid(st.active, st.omega)
        for _ in range(2):
            st, _ = O.step(cfg, st)
            run.step(1)
        run.sync()
        idx, om = run.active()
    ref_idx = np.flatnonzero(st.active.ravel())
    common, ia, ib = np.intersect1d(idx, ref_idx, return_indices=True)
    assert idx.size + ref_idx.size - 2 * common.size <= 0.002 * ref_idx.size
    assert rel_l2(om[ia], st.omega.ravel()[ref_idx][ib]) <= 1e-6
