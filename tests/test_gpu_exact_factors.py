"""FP32 lines whose operators have no uniform factors: every row's own, states from many chunks.

Uniform factors need states that die out within 128 rows (to 1e-8).  A large diffusivity carries them further, and so
does a strong mean wind; that the operators here do is checked on their inverses.  Lines of several chunks of 17 and of
33 values, columns of whole CTAs, against the FP64 oracle at the bars of the FP32 line tests (two of them: 1e-5
relative, 1e-4 of the largest departure from ambient); in a batch, beside a slot with uniform factors, against a
domain of its own, bit for bit.
"""
import numpy as np
import pytest

from gpu_helpers import assert_parity, need_gpu
from oracle.physics import Params
from oracle.step import Problem
from scenarios.generate import H_ELEMENT, greville

pytestmark = pytest.mark.gpu

DT = 1e-3


@pytest.fixture(scope="module")
def wf():
    return need_gpu()


def _state(nx, ny, p, hot):
    Lx, Ly = nx * H_ELEMENT, ny * H_ELEMENT
    x, y = greville(nx, p, Lx), greville(ny, p, Ly)
    T = 300.0 + hot * np.exp(-((x[None, :] - 0.6 * Lx) ** 2 + (y[:, None] - 0.5 * Ly) ** 2) / 40.0)
    T = np.maximum(T, 300.0 + 0.7 * hot * np.exp(-((x[None, :]) ** 2 + (y[:, None] - Ly) ** 2) / 30.0))
    return Lx, Ly, T, np.random.RandomState(nx + 7 * ny + p).uniform(0.0, 1.0, T.shape)


def _reaches(p, theta, wind, kappa, rows=128):
    """What is left of the inverse of the x operator `rows` rows from the diagonal, of a line of 400 elements."""
    pr = Problem(400, 4, p, 400 * H_ELEMENT, 4 * H_ELEMENT, DT, wind, None, Params(kappa=kappa), "pr", "ads")
    col = np.abs(np.linalg.inv(pr.x_op(theta, 1.0).toarray())[:, 200])
    return max(col[200 - rows:200 - rows + p].max(), col[200 + rows:200 + rows + p].max()) / col[200]


def _prm(wf, Lx, Ly, scheme, wind, kappa):
    return wf.wf_params_default(Lx=Lx, Ly=Ly, wind_x=wind[0], wind_y=wind[1], kappa=kappa, precision=wf.WF_FP32,
                                scheme=wf.WF_PR if scheme == "pr" else wf.WF_STRANG_CN)


@pytest.mark.parametrize("Nx,Ny", [(70, 300), (610, 37), (25, 2000), (1700, 20), (9, 130)])
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("scheme", ["pr", "strang"])
def test_slow_decay_against_oracle(wf, Nx, Ny, p, scheme):
    kappa, nx, ny = 3e6, Nx - p, Ny - p
    assert _reaches(p, (0.5 if scheme == "pr" else 0.25) * DT, (0.0, 0.0), kappa) > 1e-6
    Lx, Ly, T0, f0 = _state(nx, ny, p, 400.0)
    with wf.Simulation(nx, ny, p, DT, _prm(wf, Lx, Ly, scheme, (0.0, 0.0), kappa)) as sim:
        sim.set_state(T0, f0)
        sim.step(1)
        assert sim.sync() == wf.WF_OK
        T, phi = sim.state()
    To, po = Problem(nx, ny, p, Lx, Ly, DT, (0.0, 0.0), None, Params(kappa=kappa), scheme, "ads").run(T0, f0, 1)
    assert_parity(T, phi, To, po, "fp32", rel_bar=1e-5)


@pytest.mark.parametrize("nx,ny", [(50, 44), (200, 30)])
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("scheme", ["pr", "strang"])
def test_strong_wind_beside_another_slot(wf, nx, ny, p, scheme):
    # (one step: such winds are far past what the explicit terms stand)
    w = {1: 2e4, 2: 2e4, 3: 1e4}[p]
    kappa, winds = 0.3, ((1.7, -0.9), (w if scheme == "pr" else 2.0 * w, -w))
    assert _reaches(p, (0.5 if scheme == "pr" else 0.25) * DT, winds[1], kappa) > 1e-6
    Lx, Ly, T0, f0 = _state(nx, ny, p, 100.0)
    with wf.Batch(nx, ny, p, DT, _prm(wf, Lx, Ly, scheme, winds[1], kappa), capacity=2) as b:
        for s in range(2):
            b.set_slot(s, T0, f0, winds[s])
            b.activate(s)
        b.step(1)
        assert not b.status().any()
        got = [b.state(s) for s in range(2)]
    for s in range(2):
        with wf.Simulation(nx, ny, p, DT, _prm(wf, Lx, Ly, scheme, winds[s], kappa)) as sim:
            sim.set_state(T0, f0)
            sim.step(1)
            assert sim.sync() == wf.WF_OK
            T, phi = sim.state()
        assert np.array_equal(got[s][0], T) and np.array_equal(got[s][1], phi), s
        assert not np.array_equal(T, T0.astype(np.float32))
