"""The quadrature kernel at the sizes where it can go wrong, against the FP64 oracle.

Domains of one element (both boundaries meet in it), of two and three (elements with two boundaries in
reach), around the 32 - p columns of a strip and around the rows of a segment, with a fire in a corner (the
reaction and the fuel sums in elements next to two boundaries), a wind variation of every rank, every scheme
and order.  The bars are those of the parity tests: FP64 1e-10; FP32, a few steps, 1e-5 relative and 1e-4 of
the fire's departure from ambient.
"""
import numpy as np
import pytest

from gpu_helpers import assert_parity, need_gpu
from oracle.physics import Params
from oracle.step import Problem
from scenarios.generate import H_ELEMENT, greville

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (1, 40), (2, 3), (3, 2), (5, 31), (28, 9), (29, 30), (31, 17), (60, 5), (64, 33), (91, 8)]


@pytest.fixture(scope="module")
def wf():
    return need_gpu()


def _case(nx, ny, p, seed, rank):
    rng = np.random.RandomState(seed)
    Lx, Ly = nx * H_ELEMENT, ny * H_ELEMENT
    x, y = greville(nx, p, Lx), greville(ny, p, Ly)
    T = 300.0 + 900.0 * np.exp(-((x[None, :] - Lx) ** 2 + y[:, None] ** 2) / 18.0)
    T = np.maximum(T, 300.0 + 600.0 * np.exp(-((x[None, :] - 0.3 * Lx) ** 2 + (y[:, None] - Ly) ** 2) / 30.0))
    fuel = rng.uniform(0.0, 1.0, T.shape)
    fac = [rng.uniform(-0.2, 0.2, (rank, n)) for n in (nx + p, ny + p, nx + p, ny + p)] if rank else None
    return Lx, Ly, T, fuel, tuple(rng.uniform(-2.0, 2.0, 2)), fac


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_quadrature_sizes_against_oracle(wf, nx, ny, p, prec):
    k = SIZES.index((nx, ny))
    scheme = ("pr", "strang", "explicit")[k % 3]
    rank = (k + p) % 5
    Lx, Ly, T0, f0, wind, fac = _case(nx, ny, p, 100 * k + p, rank)
    prm = wf.wf_params_default(Lx=Lx, Ly=Ly, wind_x=wind[0], wind_y=wind[1],
                               precision=wf.WF_FP32 if prec == "fp32" else wf.WF_FP64,
                               scheme={"pr": wf.WF_PR, "strang": wf.WF_STRANG_CN, "explicit": wf.WF_EXPLICIT}[scheme],
                               scale_heat_by_fuel=k % 2)
    sim = wf.Simulation(nx, ny, p, 1e-3, prm)
    sim.set_state(T0, f0)
    if rank:
        sim.set_wind(rank, np.concatenate([a.ravel() for a in fac]))
    sim.step(2)
    assert sim.sync() == wf.WF_OK
    T, phi = sim.state()
    sim.close()
    P = Problem(nx, ny, p, Lx, Ly, 1e-3, wind, fac, Params(scale_heat_by_fuel=bool(k % 2)), scheme, "ads")
    To, po = P.run(T0, f0, 2)
    assert_parity(T, phi, To, po, prec, rel_bar=1e-10 if prec == "fp64" else 1e-5)


@pytest.mark.parametrize("nx,ny", [(5, 31), (29, 30), (64, 33), (91, 8)])
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("scheme", ["pr", "strang"])
def test_serial_and_row_parallel_quadrature_agree(wf, nx, ny, p, scheme):
    """FP32: a batch of more than 128 element rows per SM takes the serial form, one domain the row-parallel one;
    a slot's bits are those of the domain alone."""
    Lx, Ly, T0, f0, wind, fac = _case(nx, ny, p, 900 + nx + p, 2)
    factors = np.concatenate([a.ravel() for a in fac])
    prm = wf.wf_params_default(Lx=Lx, Ly=Ly, wind_x=wind[0], wind_y=wind[1], precision=wf.WF_FP32,
                               scheme=wf.WF_PR if scheme == "pr" else wf.WF_STRANG_CN)
    strips = -(-(nx + p) // (32 - p))
    S = 130 * 152 // (strips * (ny + p)) + 1
    with wf.Batch(nx, ny, p, 1e-3, prm, capacity=S) as b:
        b.set_slot(S - 1, T0, f0, wind, 2, factors)
        b.activate(S - 1)
        b.step(2)
        assert not b.status().any()
        T, phi = b.state(S - 1)
    sim = wf.Simulation(nx, ny, p, 1e-3, prm)
    sim.set_state(T0, f0)
    sim.set_wind(2, factors)
    sim.step(2)
    assert sim.sync() == wf.WF_OK
    Ts, ps = sim.state()
    sim.close()
    assert np.array_equal(T, Ts) and np.array_equal(phi, ps)
