"""FP64 1d1v deposit (integer weights, 64-bit denominator window) where its
units, rows and windows can go wrong: thousands of markers per cell, sparse
sets, markers thousands of velocity rows from their chunk's reference (beyond
the fixed-point range of a row), values over 12 decades and
of either sign, odd nx; grids and diagnostics against the FP64 oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1804_03901_gb300 import inputs

pytestmark = pytest.mark.gpu

# the suite's FP64 tolerance: in the sparse sets a cell may be reached by
# weights near 1e-4, which carry the 1e-14 rounding of x / dx
TOL = 1e-10


@pytest.mark.parametrize("nx,nv,n,values", [(8, 4, 30000, "decades"), (64, 300, 600, "decades"),
                                            (33, 50, 4001, "signed"), (16, 7000, 9000, "smooth"),
                                            (256, 64, 640, "smooth"), (5, 2, 65, "signed")])
def test_integer_weights(nx, nv, n, values):
    import torch
    assert torch.cuda.is_available()
    from paper_1804_03901_gb300 import avl as A
    L, dt, vmin, vmax = 0.3 * nx, 0.1, -4.0, 5.0
    sim = A.Simulation(A.make_domain(1, nx, L, dt, precision=A.AVL_FP64),
                       [A.make_species(-1.0, 1.0, (nv,), (vmin,), (vmax,))])
    orc = O.OracleSim(1, nx, L, dt, [O.Species(-1.0, 1.0, (nv,), (vmin,), (vmax,))])
    x, v, f = inputs.random_markers(3 * nx + n, n, L, vmin, vmax, v_overhang=0.4 if nv == 7000 else 0.05)
    rng = np.random.default_rng(n)
    if values == "signed":
        f = np.where(rng.uniform(size=n) < 0.1, 0.0, rng.normal(1.0, 0.5, n))
    elif values == "smooth":
        f = np.exp(-0.5 * v * v) * (1.0 + 0.3 * np.cos(2 * np.pi * x / L))
    sim.set_markers(0, x, v, f)
    for step in range(4):
        xs, vs, fs = sim.get_markers(0)
        orc.set_markers(0, xs, vs[0], fs)
        orc.refresh()
        if step:
            sim.step(1)
            orc.step(1)
        got, den = sim.get_f(0, with_n=True)
        for a, b in ((got, orc.f[0]), (den, orc.den[0]), (sim.get_diag()[3:], orc.diag()[3:])):
            err = np.linalg.norm(a - b) / np.linalg.norm(b)
            assert err < TOL, (step, err)
    sim.close()
