"""Handles of several host threads: each one's steps are those it takes alone.

A kernel's limit of dynamic shared memory belongs to the process, and the sizes that handles ask for differ (grids,
segment heights, wind ranks): a thread that sets the limit must not take it below what another just raised it to.
The threads create, step and destroy handles of one kernel at sizes of their own, at the same time.
"""
import threading

import numpy as np
import pytest

from gpu_helpers import need_gpu
from scenarios import make_scenario

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_handles_of_several_threads(prec):
    wf = need_gpu()
    P = wf.WF_FP32 if prec == "fp32" else wf.WF_FP64
    sizes = [24, 48, 90, 130, 200, 260, 400, 600]
    scs = [make_scenario(f"t{n}", n, 2, 1e-3, 1, n, wind=(1.0, -0.6), fuel_sigma=3.0, wind_perturbation=0.1) for n in sizes]

    def run(sc, seg):
        with wf.simulation_from_scenario(sc, precision=P) as sim:
            wf.wf_set_tuning(sim.h, (0, 0, seg, 0, 0, 0, 0, 0))
            sim.step(3)
            assert sim.sync() == wf.WF_OK
            return sim.state()

    alone = [run(sc, 0) for sc in scs]
    failed, start = [], threading.Barrier(len(scs))

    def work(i):
        try:
            start.wait()
            for k in range(12):
                T, phi = run(scs[(i + k) % len(scs)], (0, 5, 17, 40)[(i + k) % 4])
                if not (np.array_equal(T, alone[(i + k) % len(scs)][0]) and np.array_equal(phi, alone[(i + k) % len(scs)][1])):
                    failed.append((i, k, "bits"))
        except Exception as e:  # noqa: BLE001  a thread's failure has to reach the test
            failed.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(scs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
