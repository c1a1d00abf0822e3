"""Which launches a step form runs, and that every form gives the bits of form 0.

Form 0: one launch each for the quadrature, the x and the y passes.  Form 3 asks for two groups of slots; where there are
no two (one slot, manufactured forcing, the allocation-free step) the launches of form 0 run, and so they do where
the persistent form 2 cannot take a handle's lines.  The count of launches of the first unprofiled step is that of
its captures, of one step and of eight.
"""
import numpy as np
import pytest

from gpu_helpers import need_gpu
from scenarios import make_scenario

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wf():
    return need_gpu()


def _captured(wf, nx, ny, p, form, mms=False):
    prm = wf.wf_params_default(Lx=1.5 * nx, Ly=1.5 * ny, precision=wf.WF_FP32, heat_scale=0.0 if mms else 1e4)
    with wf.Simulation(nx, ny, p, 1e-3, prm) as sim:
        sim.set_state(np.full((ny + p, nx + p), 300.0), np.full((ny + p, nx + p), 0.5))
        if mms:
            wf.wf_set_mms(sim.h, [(10.0, 1, 1, 1.0)])
        wf.wf_set_tuning(sim.h, (0, 0, 0, 0, 0, 0, form, 0))
        n0 = wf.wf_launch_count()
        sim.step(1)
        assert sim.sync() == wf.WF_OK
        return wf.wf_launch_count() - n0, wf.wf_get_tuning(sim.h)[6]


def test_launches_of_one_slot(wf):
    assert _captured(wf, 200, 150, 2, 0) == (9 * 3, 0)
    assert _captured(wf, 200, 150, 2, 3) == (9 * 3, 3)
    assert _captured(wf, 200, 150, 2, 1) == (9 * 7, 1)
    # the forcing and its clock: two launches more
    assert _captured(wf, 200, 150, 2, 0, mms=True) == (9 * 5, 0)
    assert _captured(wf, 200, 150, 2, 3, mms=True) == (9 * 5, 3)


def test_lines_too_long_for_the_persistent_form(wf):
    assert _captured(wf, 17000, 2, 2, 2) == (9 * 3, 0)


@pytest.mark.parametrize("form,per_step", [(0, 3), (1, 7), (2, 3), (3, 3)])
def test_launches_of_the_allocation_free_step(wf, form, per_step):
    import torch

    sc = make_scenario("forms", 200, 2, 1e-3, 1, 5)
    sim = wf.simulation_from_scenario(sc, precision=wf.WF_FP32)
    wf.wf_set_tuning(sim.h, (0, 0, 0, 0, 0, 0, form, 0))
    a = [torch.tensor(x, dtype=torch.float32, device="cuda") for x in (sc.T0, sc.fuel0)]
    torch.cuda.synchronize()
    n0 = wf.wf_launch_count()
    assert wf.wf_step_noalloc(sim.h, a[0].data_ptr(), a[1].data_ptr(), sc.Nx, 2) == wf.WF_OK
    n1 = wf.wf_launch_count()
    assert sim.sync() == wf.WF_OK
    sim.close()
    assert n1 - n0 == 2 * per_step


@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("slots", [1, 3])
def test_forms_give_the_bits_of_form_0(wf, p, prec, slots):
    winds = [(1.0, 0.5), (-2.0, 1.5), (0.3, -2.7)]
    scs = [make_scenario(f"f{i}", 70, p, 1e-3, 1, 60 + i, wind=winds[i], fuel_sigma=3.0, wind_perturbation=0.1) for i in range(slots)]
    out = []
    for form in range(4):
        prm = wf.wf_params_default(Lx=scs[0].Lx, Ly=scs[0].Ly, precision=wf.WF_FP32 if prec == "fp32" else wf.WF_FP64)
        with wf.Batch(scs[0].nx, scs[0].ny, p, 1e-3, prm, capacity=slots) as b:
            for i, sc in enumerate(scs):
                b.load_scenario(i, sc)
            wf.wf_set_tuning(b.h, (0, 0, 0, 0, 0, 0, form, 0))
            b.step(10)
            assert not b.status().any()
            out.append([b.state(i) for i in range(slots)])
    for form in (1, 2, 3):
        for (T, f), (T0, f0) in zip(out[form], out[0]):
            assert np.array_equal(T, T0) and np.array_equal(f, f0), form
