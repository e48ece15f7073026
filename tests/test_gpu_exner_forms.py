"""One step of the velocity-Exner form in every form of its Krylov kernel
against the FP64 oracle, both schemes: the table of basis digits in shared
memory at few and at many entries per block, of 64-bit integers, with and
without ghosts, orders 2p = 4 and 8, the largest dimension, and a problem too
large for either (the kernel with the basis in global memory).  The bounds
are those of the form's other parity tests: 1e-10 on the fields, 1e-12 on
beta, the Krylov dimension equal."""

import numpy as np
import pytest

from oracle import exner as E
from oracle import wrc_oracle as O
from paper_1604_08159_gb300 import binding as B
from paper_1604_08159_gb300 import workloads as W

from helpers import oracle_config, rel_l2, small_params

pytestmark = pytest.mark.gpu

VORT = dict(xc=[-0.7, 0.6], yc=[0.1, -0.2], gamma=[2.0, 1.2], s=[0.45, 0.5])


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_08159_gb300 import build
    build.build()
    B.load()


@pytest.mark.parametrize("n0,J,eps,m,p,scheme", [
    (16, 1, 0.0, 10, 2, W.SCHEME_FROZEN),        # 3072 entries, no ghosts
    (32, 2, 0.0, 31, 2, W.SCHEME_ROSENBROCK),    # 49152 entries, 324 a block
    (16, 4, 1e-6, 31, 4, W.SCHEME_FROZEN),       # 25K entries with ghosts
    (16, 4, 3e-6, 30, 2, W.SCHEME_ROSENBROCK),   # about 75K entries: integers
    (32, 3, 0.0, 12, 2, W.SCHEME_FROZEN),        # 196608 entries: do not fit
])
def test_exner_step_every_form(n0, J, eps, m, p, scheme):
    prm = small_params(model=W.MODEL_EXNER, cpt=4.0, coriolis=0.5, re=1000.0, dt=0.005, n0=n0, J=J, eps=eps, m=m, p=p,
                       scheme=scheme, gx=0.2, gy=-0.1, rayleigh_r=0.05)
    cfg = oracle_config(prm)
    st = E.exner_vortex_state(cfg, VORT["xc"], VORT["yc"], VORT["gamma"], VORT["s"], 1.0)
    om = O.vortex_field(cfg.NJ, VORT["xc"], VORT["yc"], VORT["gamma"], VORT["s"])
    psi = O.streamfunction(om, cfg.h, cfg.p)
    u0, v0 = O.velocity(psi, cfg.h, cfg.p)
    with B.Run(prm) as run:
        run.exner_init(u0, v0, np.ones_like(u0))
        st, info = E.exner_step(cfg, st)
        run.step(1)
        run.sync()
        kr = run.krylov()
        assert kr["k"] == info.k
        assert abs(kr["beta"] - info.beta) <= 1e-12 * info.beta
        idx, u, v, pi = run.exner()
        act, _, _ = run.masks()
        assert np.array_equal(act, st.active)
        a = st.active
        err = rel_l2(np.concatenate([u, v, pi]), np.concatenate([st.u[a], st.v[a], st.pi[a]]))
        assert err <= 1e-10, err
