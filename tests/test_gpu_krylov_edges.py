"""The Krylov launch's tables at the edges of their forms, on a device of 152
SMs.  A grid of 152000 points (the 256^2 sublattice of 512^2 and a band of
whole rows) gives blocks of 1008 points, next to the most a table takes: at
m = 5 digits as halves (six rows of ~1040 columns, each product warp in eight
turns, its f32 sums nearest to 2^24), at m = 10 64-bit integers.  And the
launch of each form whose grid barriers run out (a limit of 100 ns) reports
it, leaves the device usable, and a new initial condition steps as if nothing
had happened."""

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


def band_state(cfg):
    """Every second point of every second row, and whole rows up to 152000 points."""
    act = np.zeros((cfg.NJ, cfg.NJ), dtype=bool)
    act[::2, ::2] = True
    row = 100
    while act.sum() <= 152000 - 512:
        act[row] = True
        row += 1
    v = W.random_field_params(11, 5)
    om = O.vortex_field(cfg.NJ, v.xc, v.yc, v.gamma, v.s)
    return act, np.where(act, om, 0.0)


@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_MIXED])
@pytest.mark.parametrize("m", [5, 10])
def test_largest_blocks(m, prec):
    prm = small_params(n0=32, J=4, eps=1e-7, m=m, re=2000.0, prec=prec)
    cfg = oracle_config(prm)
    act, om = band_state(cfg)
    if prec == W.PREC_MIXED:
        om = om.astype(np.float32).astype(np.float64)
    v = W.random_field_params(11, 5)
    st = O.initial_state(cfg, v.xc, v.yc, v.gamma, v.s)
    st.active, st.omega = act, om
    with B.Run(prm) as run:
        run.set_grid(act, om)
        assert 151000 < run.counts()[0] <= 152 * 1008
        st2, info = O.step(cfg, st)
        run.step(1)
        run.sync()
        kr = run.krylov()
        assert kr["k"] == info.k
        idx, got = run.active()
        ref = np.flatnonzero(st2.active.ravel())
        want = st2.omega.ravel()
        if prec == W.PREC_FP64:
            assert abs(kr["beta"] - info.beta) <= 1e-12 * info.beta
            assert np.array_equal(idx, ref) and rel_l2(got, want[ref]) <= 1e-10
        else:
            common, ia, ib = np.intersect1d(idx, ref, assume_unique=True, return_indices=True)
            assert idx.size + ref.size - 2 * common.size <= 0.002 * ref.size
            assert rel_l2(got[ia], want[ref][ib]) <= 1e-6


@pytest.mark.parametrize("kw", [dict(n0=32, J=2, m=31), dict(n0=32, J=3, m=31), dict(n0=32, J=4, m=18)],
                         ids=["halves", "words", "streaming"])
def test_wait_limit_runs_out(kw):
    prm = small_params(eps=0.0, **kw)
    v = W.fujiwhara_small().vortices
    with B.Run(prm) as run:
        run.init_vortices(v)
        run.step(1)
        ref = run.active()
        run.init_vortices(v)
        run.set_wait_limit(1e-7)
        with pytest.raises(B.WrcError) as e:
            run.step(1)
        assert e.value.status == -5
        run.set_wait_limit(2.0)
        run.init_vortices(v)
        run.step(1)
        for got, want in zip(run.active(), ref):
            assert np.array_equal(got, want)


def test_exner_wait_limit_runs_out():
    prm = small_params(model=W.MODEL_EXNER, cpt=4.0, coriolis=0.5, re=1000.0, dt=0.005, n0=16, J=2, eps=0.0, m=20)
    v = W.fujiwhara_small().vortices
    with B.Run(prm) as run:
        run.exner_init_vortices(v)
        run.step(1)
        ref = run.exner()
        run.exner_init_vortices(v)
        run.set_wait_limit(1e-7)
        with pytest.raises(B.WrcError) as e:
            run.step(1)
        assert e.value.status == -5
        run.set_wait_limit(2.0)
        run.exner_init_vortices(v)
        run.step(1)
        for got, want in zip(run.exner(), ref):
            assert np.array_equal(got, want)
