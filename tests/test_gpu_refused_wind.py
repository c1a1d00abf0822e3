"""A wind that a slot refuses leaves the slot as it was, however often it is asked for.

The refused operators (their inverse decays far more slowly than that of the handle's own winds) have overwritten the
slot's tables by the time they are refused: the slot has to get its own ones back, the same request has to be
refused again, and the slot's next steps have to be those of a domain that never heard of it.
"""
import numpy as np
import pytest

from gpu_helpers import need_gpu
from scenarios.generate import H_ELEMENT, greville

pytestmark = pytest.mark.gpu

NX, NY, P, WIND, FAR = 400, 60, 3, (1.7, -0.9), (1e5, -1e5)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("scheme", ["pr", "strang"])
@pytest.mark.parametrize("call", ["set_slot", "set_mean_wind"])
def test_refused_wind_leaves_the_slot(prec, scheme, call):
    wf = need_gpu()
    Lx, Ly = NX * H_ELEMENT, NY * H_ELEMENT
    x, y = greville(NX, P, Lx), greville(NY, P, Ly)
    T0 = 300.0 + 700.0 * np.exp(-((x[None, :] - 0.4 * Lx) ** 2 + (y[:, None] - 0.5 * Ly) ** 2) / 18.0)
    f0 = np.random.RandomState(5).uniform(0.0, 1.0, T0.shape)
    prm = wf.wf_params_default(Lx=Lx, Ly=Ly, wind_x=0.3, wind_y=0.4, precision=wf.WF_FP32 if prec == "fp32" else wf.WF_FP64,
                               scheme=wf.WF_PR if scheme == "pr" else wf.WF_STRANG_CN)
    out = []
    for refuse in (False, True):
        with wf.Batch(NX, NY, P, 1e-3, prm, capacity=2) as b:
            b.set_slot(0, T0, f0, WIND)
            b.activate(0)
            b.step(2)
            for _ in range(2 if refuse else 0):
                with pytest.raises(wf.WFError) as e:
                    if call == "set_slot":
                        b.set_slot(0, np.full_like(T0, 310.0), f0, FAR)
                    else:
                        wf.wf_set_mean_wind(b.h, *FAR, slot=0)
                assert e.value.code == wf.WF_ETRUNC
            b.step(3)
            assert not b.status().any()
            out.append(b.state(0))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
