"""Overlapping the launches of a step costs nothing: against the same kernels one at a time.

wf_step replays graphs whose kernels begin beside the end of the one before; with profiling on, an event before and after
each kernel keeps them apart, and their times add up to a step without overlap or launch latency.  A step may
take that sum and a quarter (what an event adds to a kernel of some microseconds makes the sum larger, never smaller).
FP64, where the quadrature is few long CTAs and their places decide its time.
"""
import time

import numpy as np
import pytest

from gpu_helpers import need_gpu
from scenarios.generate import H_ELEMENT, greville

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,p,slots,scheme", [(256, 256, 2, 8, "pr"), (40, 40, 2, 64, "strang"), (400, 400, 2, 1, "pr"),
                                                  (400, 400, 3, 1, "strang"), (60, 33, 3, 9, "pr"), (40, 40, 1, 64, "explicit")])
def test_step_against_its_kernels(nx, ny, p, slots, scheme):
    wf = need_gpu()
    Lx, Ly = nx * H_ELEMENT, ny * H_ELEMENT
    x, y = greville(nx, p, Lx), greville(ny, p, Ly)
    T0 = 300.0 + 700.0 * np.exp(-((x[None, :] - 0.6 * Lx) ** 2 + (y[:, None] - 0.4 * Ly) ** 2) / 18.0)
    f0 = np.random.RandomState(7).uniform(0.0, 1.0, T0.shape)
    prm = wf.wf_params_default(Lx=Lx, Ly=Ly, wind_x=1.7, wind_y=-0.9, precision=wf.WF_FP64,
                               scheme={"pr": wf.WF_PR, "strang": wf.WF_STRANG_CN, "explicit": wf.WF_EXPLICIT}[scheme])
    steps = 16
    with wf.Batch(nx, ny, p, 1e-3, prm, capacity=slots) as b:
        def load():
            for s in range(slots):
                b.set_slot(s, T0, f0, (1.7, -0.9))
                b.activate(s)
            b.status()

        load()
        b.step(steps)  # captures
        b.status()
        times = []
        for _ in range(4):
            load()
            t0 = time.perf_counter()
            b.step(steps)
            b.status()
            times.append((time.perf_counter() - t0) / steps)
        load()
        wf.wf_set_profiling(b.h, True)
        b.step(steps)
        alone = sum(ms for ms, _ in wf.wf_kernel_times(b.h).values()) / steps * 1e-3
    assert min(times) <= 1.25 * alone, (min(times) * 1e6, alone * 1e6)
