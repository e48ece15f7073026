"""A grid whose arrays cannot grow (the allocation refused on the host by a
test switch, at the size of the basis): WRC_ERR_OOM, no step from that run
until a new initial condition, and from there the results of a run that never
met the failure, bit for bit -- in batched launches and for the Rosenbrock
step, whose basis is kept in global memory."""

import numpy as np
import pytest

from paper_1604_08159_gb300 import binding as B
from paper_1604_08159_gb300 import workloads as W

from helpers import small_params

pytestmark = pytest.mark.gpu

VORT = W.fujiwhara_small().vortices


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_08159_gb300 import build
    build.build()
    B.load()


def grow_until_refused(run, monkeypatch):
    """Thresholds towards zero widen the grid by its adjacent zones."""
    monkeypatch.setenv("WRC_ALLOC_TEST_LIMIT", str(1 << 20))
    try:
        for q in range(8):
            run.threshold(1e-30)
    except B.WrcError as e:
        assert e.status == -2, e
        return
    finally:
        monkeypatch.delenv("WRC_ALLOC_TEST_LIMIT")
    raise AssertionError("no growth was refused")


def test_batched_member(monkeypatch):
    prm, low = small_params(m=30), small_params(m=30, eps=1e-30)   # threshold's eps becomes the run's
    with B.Ensemble([low, prm]) as ens:
        for mem in ens.members:
            mem.init_vortices(VORT)
        ens.step(1)
        ref = [mem.active() for mem in ens.members]
    with B.Ensemble([prm, prm]) as ens:
        for mem in ens.members:
            mem.init_vortices(VORT)
        ens.step(1)
        grow_until_refused(ens.members[0], monkeypatch)
        with pytest.raises(B.WrcError, match="no initial condition"):
            ens.step(1)
        for mem in ens.members:
            mem.init_vortices(VORT)
        ens.step(1)
        for mem, r in zip(ens.members, ref):
            for got, want in zip(mem.active(), r):
                assert np.array_equal(got, want)


def test_rosenbrock_run(monkeypatch):
    prm = dict(m=30, scheme=W.SCHEME_ROSENBROCK)
    with B.Run(small_params(eps=1e-30, **prm)) as run:
        run.init_vortices(VORT)
        run.step(1)
        ref = run.active()
    with B.Run(small_params(**prm)) as run:
        run.init_vortices(VORT)
        run.step(1)
        grow_until_refused(run, monkeypatch)
        with pytest.raises(B.WrcError, match="no initial condition"):
            run.step(1)
        run.init_vortices(VORT)
        run.step(1)
        for got, want in zip(run.active(), ref):
            assert np.array_equal(got, want)


def test_tables_of_the_solve(monkeypatch):
    """The FP64 solve's table, the largest of a run's tables: a failed
    allocation of it is out of memory (a server waits and tries again), and
    leaves nothing pending."""
    prm = small_params(n0=32, J=4)   # (n / 2 + 1) n doubles: 1.05 MB
    monkeypatch.setenv("WRC_ALLOC_TEST_LIMIT", str(1 << 20))
    with pytest.raises(B.WrcError) as e:
        B.Run(prm)
    assert e.value.status == -2
    monkeypatch.delenv("WRC_ALLOC_TEST_LIMIT")
    with B.Run(prm) as run:
        run.init_vortices(VORT)
        run.step(1)
        run.sync()


def test_tables_of_a_batched_launch(monkeypatch):
    """The launch's block table refused at the first step: an error, and after a
    new initial condition a step as if nothing had happened."""
    prm = small_params()
    ref = None
    for refuse in (False, True):
        with B.Ensemble([prm, prm]) as ens:
            for mem in ens.members:
                mem.init_vortices(VORT)
            if refuse:
                monkeypatch.setenv("WRC_ALLOC_TEST_LIMIT", "1000")
                with pytest.raises(B.WrcError):
                    ens.step(1)
                monkeypatch.delenv("WRC_ALLOC_TEST_LIMIT")
                for mem in ens.members:
                    mem.init_vortices(VORT)
            ens.step(1)
            got = ens.members[1].active()
            ref = ref or got
            for x, y in zip(got, ref):
                assert np.array_equal(x, y)
