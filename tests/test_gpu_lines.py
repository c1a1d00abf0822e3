"""The line passes at the sizes where they can go wrong, against the FP64 oracle.

Lines around a chunk and its multiples, around the lengths where the chunk length changes (144 values; 1600 in
FP32, 1088 in FP64), lines too short for uniform factors (4p values) and one longer, lines cut into several
tiles with few lines beside them (one, and one more than a CTA takes), lines of more than 512 chunks, rows that
do not fit the shared memory, and rows whose length is no multiple of 16 bytes, in every scheme.  Operators whose
states decay slowly (a large diffusivity) take the tables of every row's factors, in the domain and beside others in
a batch.  Bars: those of the parity tests, FP64 1e-10; FP32, two steps, 1e-5 relative and 1e-4 of the fire's
departure from ambient.  The slowly decaying operator (theta C_d / h^2 = 475) runs in FP64, without fire: the
explicit terms are about 2e3 times T, so 2e3 * 2.2e-16 relative at most, well below 1e-10.
"""
import numpy as np
import pytest

from gpu_helpers import assert_parity, need_gpu
from oracle.physics import Params
from oracle.step import Problem
from scenarios.generate import H_ELEMENT, greville

pytestmark = pytest.mark.gpu

# values per line (Nx, Ny): degrees are subtracted below
SIZES = [(8, 13), (12, 9), (18, 27), (27, 28), (33, 144), (144, 35), (145, 33), (34, 145), (289, 153), (256, 290), (9, 1600),
         (1601, 9), (40, 1090), (1100, 33), (5, 2200), (2200, 6)]


@pytest.fixture(scope="module")
def wf():
    return need_gpu()


def _state(nx, ny, p, hot):
    Lx, Ly = nx * H_ELEMENT, ny * H_ELEMENT
    x, y = greville(nx, p, Lx), greville(ny, p, Ly)
    T = 300.0 + hot * np.exp(-((x[None, :] - 0.6 * Lx) ** 2 + (y[:, None] - 0.5 * Ly) ** 2) / 40.0)
    T = np.maximum(T, 300.0 + 0.7 * hot * np.exp(-((x[None, :]) ** 2 + (y[:, None] - Ly) ** 2) / 30.0))
    return Lx, Ly, T, np.random.RandomState(nx + 7 * ny + p).uniform(0.0, 1.0, T.shape)


def _check(wf, Nx, Ny, p, prec, scheme, wind=(1.7, -0.9), kappa=0.3, hot=900.0, steps=2):
    nx, ny = Nx - p, Ny - p
    Lx, Ly, T0, f0 = _state(nx, ny, p, hot)
    prm = wf.wf_params_default(Lx=Lx, Ly=Ly, wind_x=wind[0], wind_y=wind[1], kappa=kappa,
                               precision=wf.WF_FP32 if prec == "fp32" else wf.WF_FP64,
                               scheme={"pr": wf.WF_PR, "strang": wf.WF_STRANG_CN, "explicit": wf.WF_EXPLICIT}[scheme])
    sim = wf.Simulation(nx, ny, p, 1e-3, prm)
    sim.set_state(T0, f0)
    sim.step(steps)
    assert sim.sync() == wf.WF_OK
    T, phi = sim.state()
    sim.close()
    To, po = Problem(nx, ny, p, Lx, Ly, 1e-3, wind, None, Params(kappa=kappa), scheme, "ads").run(T0, f0, steps)
    assert_parity(T, phi, To, po, prec, rel_bar=1e-10 if prec == "fp64" else 1e-5)


@pytest.mark.parametrize("Nx,Ny", SIZES)
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_line_lengths_against_oracle(wf, Nx, Ny, p, prec):
    _check(wf, Nx, Ny, p, prec, ("pr", "strang", "explicit")[(SIZES.index((Nx, Ny)) + p) % 3])


@pytest.mark.parametrize("Nx,Ny,prec", [(17003, 4, "fp32"), (4, 17003, "fp32"), (30001, 4, "fp64"), (4, 17003, "fp64")])
@pytest.mark.parametrize("scheme", ["pr", "strang"])
def test_longest_lines_against_oracle(wf, Nx, Ny, prec, scheme):
    _check(wf, Nx, Ny, 2, prec, scheme, steps=1)


@pytest.mark.parametrize("Nx,Ny", [(70, 300), (610, 37)])
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("scheme", ["pr", "strang"])
def test_slow_decay_against_oracle(wf, Nx, Ny, p, scheme):
    _check(wf, Nx, Ny, p, "fp64", scheme, wind=(0.0, 0.0), kappa=3e6, hot=400.0, steps=1)


@pytest.mark.parametrize("Nx,Ny", [(4, 17003), (17003, 4)])
@pytest.mark.parametrize("scheme", ["pr", "strang"])
def test_slow_decay_on_longest_lines_against_oracle(wf, Nx, Ny, scheme):
    """More than 512 chunks whose states reach over several tiles."""
    _check(wf, Nx, Ny, 2, "fp64", scheme, wind=(0.0, 0.0), kappa=3e6, hot=400.0, steps=1)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("scheme", ["pr", "strang"])
def test_slow_decay_beside_other_slots(wf, prec, scheme):
    """Slot 1's wind has no uniform factors on these short lines; slot 0 keeps the bits of a run by itself."""
    p, nx, ny = 2, 50, 44
    Lx, Ly, T0, f0 = _state(nx, ny, p, 900.0)
    prm = wf.wf_params_default(Lx=Lx, Ly=Ly, wind_x=1.7, wind_y=-0.9, precision=wf.WF_FP32 if prec == "fp32" else wf.WF_FP64,
                               scheme=wf.WF_PR if scheme == "pr" else wf.WF_STRANG_CN)
    with wf.Batch(nx, ny, p, 1e-3, prm, capacity=2) as b:
        b.set_slot(0, T0, f0, (1.7, -0.9))
        b.set_slot(1, np.full_like(T0, 300.0), f0, (1e5, -1e5))
        b.activate(0)
        b.activate(1)
        b.step(3)
        b.status()
        T, phi = b.state(0)
    sim = wf.Simulation(nx, ny, p, 1e-3, prm)
    sim.set_state(T0, f0)
    sim.step(3)
    assert sim.sync() == wf.WF_OK
    Ts, ps = sim.state()
    sim.close()
    assert np.array_equal(T, Ts) and np.array_equal(phi, ps)


@pytest.mark.parametrize("n", [60, 300])
def test_captured_steps_follow_a_new_wind(wf, n):
    """A caller's graph of allocation-free steps addresses the factors: replayed after a change to a wind whose
    operators reach further, it gives the bits of steps launched then."""
    torch = pytest.importorskip("torch")
    Lx, Ly, T0, f0 = _state(n, n, 2, 900.0)
    prm = wf.wf_params_default(Lx=Lx, Ly=Ly, wind_x=0.5, wind_y=-0.5, precision=wf.WF_FP32)
    sim = wf.Simulation(n, n, 2, 1e-3, prm)
    st = torch.cuda.Stream()
    wf.wf_set_stream(sim.h, st.cuda_stream)
    a = [torch.tensor(x, dtype=torch.float32, device="cuda") for x in (T0, f0)]
    step = lambda: wf.wf_step_noalloc(sim.h, a[0].data_ptr(), a[1].data_ptr(), n + 2, 2)  # noqa: E731
    with torch.cuda.stream(st):
        assert step() == wf.WF_OK  # looks the scratch address up before the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        assert step() == wf.WF_OK
    wf.wf_set_mean_wind(sim.h, 1500.0, -1200.0)
    out = []
    for run in (g.replay, step):
        for x, x0 in zip(a, (T0, f0)):
            x.copy_(torch.tensor(x0, dtype=torch.float32))
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            run()
        torch.cuda.synchronize()
        out.append([x.cpu().numpy().copy() for x in a])
    sim.close()
    assert np.isfinite(out[1][0]).all()
    assert all(np.array_equal(x, y) for x, y in zip(*out))
