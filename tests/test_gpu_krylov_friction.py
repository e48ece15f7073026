"""Krylov steps whose operator is near a multiple of the identity, where the
rounding of the ghost values may grow by |q_j . A q_j| / h_{j+1} a step and
leave the range of their fixed point: strong Rayleigh friction, and viscous
flows near an eigenvector.  One step against the FP64 oracle with the bounds
of the step parity tests (omega 1e-10, mixed 1e-6 over the common grid; beta
1e-12; k equal)."""

import numpy as np
import pytest

from oracle import exner as E
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


def one_step(prm, st):
    """The oracle's step and the library's from the same state."""
    cfg = oracle_config(prm)
    if prm.prec == W.PREC_MIXED:
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
        want = st2.omega.ravel()
        if prm.prec == W.PREC_FP64:
            assert abs(kr["beta"] - info.beta) <= 1e-12 * info.beta
            assert np.array_equal(idx, ref)
            assert rel_l2(om, want[ref]) <= 1e-10
        else:
            common, ia, ib = np.intersect1d(idx, ref, assume_unique=True, return_indices=True)
            assert idx.size + ref.size - 2 * common.size <= max(2, 0.002 * ref.size)
            assert rel_l2(om[ia], want[ref][ib]) <= 1e-6


@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_MIXED])
@pytest.mark.parametrize("r", [50.0, 1e4])
@pytest.mark.parametrize("kw", [dict(n0=16, J=3, eps=1e-3), dict(n0=16, J=4, eps=1e-4, p=4), dict(n0=32, J=4, eps=1e-9)],
                         ids=["narrow", "order 8", "streaming"])
def test_strong_friction(kw, r, prec):
    prm = small_params(m=31, re=2000.0, rayleigh_r=r, dt=min(1e-2, 1.0 / r), prec=prec, **kw)
    v = W.random_field_params(11, 5)
    one_step(prm, O.initial_state(oracle_config(prm), v.xc, v.yc, v.gamma, v.s))


@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_MIXED])
@pytest.mark.parametrize("kw,k", [(dict(n0=16, J=3, eps=1e-3), 3), (dict(n0=32, J=4, eps=4e-8), 3)],
                         ids=["table", "streaming"])
def test_near_eigenvector(kw, k, prec):
    prm = small_params(m=31, re=1.0, dt=1e-3, prec=prec, **kw)
    cfg = oracle_config(prm)
    x = 2 * np.pi * np.arange(cfg.NJ) / cfg.NJ
    one_step(prm, O.state_from_field(cfg, np.outer(np.sin(k * x), np.sin(k * x))))


@pytest.mark.parametrize("scheme", [W.SCHEME_FROZEN, W.SCHEME_ROSENBROCK])
def test_exner_friction(scheme):
    prm = small_params(model=W.MODEL_EXNER, cpt=25.0, coriolis=0.5, re=2000.0, dt=1e-4, m=31, rayleigh_r=1e4,
                       scheme=scheme)
    cfg = oracle_config(prm)
    v = W.fujiwhara_small().vortices
    st = E.exner_vortex_state(cfg, v.xc, v.yc, v.gamma, v.s, 1.0)
    om = O.vortex_field(cfg.NJ, v.xc, v.yc, v.gamma, v.s)
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
        _, u, vv, pi = run.exner()
        a = st.active
        assert rel_l2(np.concatenate([u, vv, pi]), np.concatenate([st.u[a], st.v[a], st.pi[a]])) <= 1e-10
