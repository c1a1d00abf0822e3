"""Changing the wind of a long line costs no more than its length.

The factor tables of a line are one elimination from its first row on; a thread that owns a chunk far down must not run
it row by row, or the work grows with the square of the line.  16 times the rows may take 16 times the time (the
best of several calls each; row by row, they took 30 to 40 times).
"""
import time

import pytest

from gpu_helpers import need_gpu
from scenarios.generate import H_ELEMENT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_mean_wind_time_against_line_length(prec, p):
    wf = need_gpu()
    best = {}
    for n in (1024, 16384):
        prm = wf.wf_params_default(Lx=n * H_ELEMENT, Ly=4 * H_ELEMENT, wind_x=0.3, wind_y=0.2,
                                   precision=wf.WF_FP32 if prec == "fp32" else wf.WF_FP64)
        sim = wf.Simulation(n, 4, p, 1e-3, prm)
        times = []
        for k in range(6):
            t0 = time.perf_counter()
            wf.wf_set_mean_wind(sim.h, 0.3 + 1e-3 * (k + 1), 0.2)
            times.append(time.perf_counter() - t0)
        sim.close()
        best[n] = min(times)
    assert best[16384] <= 16.0 * best[1024], best
