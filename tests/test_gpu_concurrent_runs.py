"""Independent runs stepped by a thread and on a stream each: the results of a
run alone, bit for bit, and small runs share the device -- eight at once have
at least 2.2 times the throughput of one (with launches over most of the SMs
they had 1.6 times, with blocks of 48 points 3)."""

import threading
import time

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


@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_MIXED])
def test_eight_small_runs(prec):
    import torch
    prm = small_params(prec=prec)
    streams = [torch.cuda.Stream() for _ in range(8)]
    runs = [B.Run(prm, s.cuda_stream) for s in streams]

    def seconds(some, steps=40):
        def work(r):
            r.step(steps)
            r.sync()
        best = 1e9
        for _ in range(3):
            for r in runs:
                r.init_vortices(VORT)
                r.step(2)
                r.sync()
            threads = [threading.Thread(target=work, args=(r,)) for r in some]
            t = time.perf_counter()
            for x in threads:
                x.start()
            for x in threads:
                x.join()
            best = min(best, time.perf_counter() - t)
        return best

    try:
        one = seconds(runs[:1])
        alone = runs[0].active()
        all8 = seconds(runs)
        for r in runs:
            for got, want in zip(r.active(), alone):
                assert np.array_equal(got, want)
        assert 8 * one / all8 >= 2.2, (one, all8)
    finally:
        for r in runs:
            r.close()
