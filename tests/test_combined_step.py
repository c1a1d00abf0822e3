"""The combined Peaceman-Rachford step the GPU path solves, against the two substeps of the oracle.

With one F per step the two systems of Eq. matrixPR are equivalent to one,
    (X_+ (x) Y_+) (T^{n+1} - T^n) = tau F - tau (A_x (x) M^y) T^n - tau (M^x (x) A_y) T^n,
for every order, rectangular grid and wind (theta = tau / 2, X_+ = M^x + theta A_x, Y_+ = M^y + theta A_y).
Both sides are solved here in FP64 by the oracle's banded solves.  The two forms differ by the rounding
of a few operators of condition number below 1e3 applied to |T| <= 1e3 K: 1e3 * 1e3 * 2.2e-16 K, a few
1e-10 K, is the bar on the increment's error.
"""
import numpy as np
import pytest

from oracle.step import Problem
from scenarios import make_scenario


@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("nx,ny", [(19, 33), (30, 12)])
def test_combined_step_equals_two_substeps(p, nx, ny):
    sc = make_scenario("cmb", max(nx, ny), p, 1e-3, 1, 40 + p, wind=(2.1, -1.3), fuel_sigma=3.0)
    T, phi = sc.T0[:ny + p, :nx + p].copy(), sc.fuel0[:ny + p, :nx + p].copy()
    h = sc.Lx / sc.nx
    P = Problem(nx, ny, p, nx * h, ny * h, 5e-3, sc.wind, None, None, "pr", "ads")
    Tn, _ = P.pr_step(T, phi)
    F, _ = P.load(T, phi)
    tau, th = P.dt, 0.5 * P.dt
    # -tau (A_x (x) M^y) T - tau (M^x (x) A_y) T from the explicit sides at theta = tau
    m = P.apply(("m",), T)
    R = tau * F + (P.apply(("x", tau, -1.0), T) - m) + (P.apply(("y", tau, -1.0), T) - m)
    P.factors = lambda key: (P.x_op(th, 1.0), P.y_op(th, 1.0))
    d = P.solve(("xy",), R)
    assert np.abs(T + d - Tn).max() <= 5e-10
