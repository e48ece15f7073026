"""A velocity-Exner flow in other units -- velocities times c, C = c_p theta_0
times c^2, f and the viscosity times c, the time step over c, pi as it is --
is the same flow: c = 2^9 (as SI units would be) and c so large that the pi
part of a Krylov vector is up to 2^-122 of its velocity part.  One step
converged in the Krylov dimension must give the velocity times c and the same
pi: 1e-12 and 1e-13 relative, the roundings of steps in different norms."""

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


def step(c, scheme):
    prm = small_params(model=W.MODEL_EXNER, cpt=25.0 * c * c, coriolis=0.5 * c, re=2000.0 / c, dt=2e-3 / c, m=31,
                       eps=0.0, n0=16, J=2, scheme=scheme)
    v = W.Vortices(np.array([-0.6, 0.6]), np.zeros(2), np.array([1.0, 0.8]) * c, np.full(2, 0.5))
    with B.Run(prm) as run:
        run.exner_init_vortices(v, 1.0)
        run.step(1)
        run.sync()
        _, a, b, pi = run.exner()
        return np.concatenate([a, b]) / c, pi


@pytest.mark.parametrize("scheme", [W.SCHEME_FROZEN, W.SCHEME_ROSENBROCK])
@pytest.mark.parametrize("e", [9, 20, 60, 120])
def test_step_in_other_units(e, scheme):
    uv, pi = step(1.0, scheme)
    uv2, pi2 = step(2.0 ** e, scheme)
    assert rel_l2(uv2, uv) <= 1e-12
    assert rel_l2(pi2, pi) <= 1e-13
