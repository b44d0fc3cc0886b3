"""FP64 1d3v deposit (64-bit integer sums) where its sums, units and chunks can
go wrong: hundreds of markers per column (sums flushed inside a chunk, several
chunks per segment), values over 12 decades, of either sign and zero, one and
two columns per thread; grids against the FP64 oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1804_03901_gb300 import inputs

pytestmark = pytest.mark.gpu

# weights carry the rounding of x / dx and of the v_x row, some 1e-14 of a
# cell, and enter f through the spread of the values in a cell; n directly
TOL = 1e-12


@pytest.mark.parametrize("B", [None, (0.3, -0.9, 1.4)], ids=["kick", "boris"])
@pytest.mark.parametrize("nx,nv,n,values", [(4, (2, 2, 2), 20000, "decades"), (33, (3, 2, 2), 9000, "signed"),
                                            (256, (3, 2, 2), 60000, "smooth"), (257, (2, 3, 2), 5000, "decades"),
                                            (512, (2, 2, 3), 30000, "signed")])
def test_fixed_point_sums(nx, nv, n, values, B):
    import torch
    assert torch.cuda.is_available()
    from paper_1804_03901_gb300 import avl as A
    L, dt, vmin, vmax = 0.4 * nx, 0.07, (-3.0, -2.0, -2.5), (3.0, 2.0, 1.5)
    sim = A.Simulation(A.make_domain(3, nx, L, dt, precision=A.AVL_FP64),
                       [A.make_species(-1.0, 1.0, nv, vmin, vmax)])
    orc = O.OracleSim(3, nx, L, dt, [O.Species(-1.0, 1.0, nv, vmin, vmax)])
    x, v, f = inputs.random_markers3(17 * nx + n, n, L, vmin, vmax)
    rng = np.random.default_rng(n)
    if values == "signed":
        f = np.where(rng.uniform(size=n) < 0.1, 0.0, rng.normal(1.0, 0.5, n))
    elif values == "smooth":
        f = np.exp(-0.5 * (v ** 2).sum(0)) * (1.0 + 0.3 * np.cos(2 * np.pi * x / L))
    sim.set_markers(0, x, v, f)
    if B:
        sim.set_bfield(B)
        orc.B = np.array(B)
    for step in range(3):
        xs, vs, fs = sim.get_markers(0)
        orc.set_markers(0, xs, vs, fs)
        orc.refresh()
        if step == 0:
            assert abs(np.sort(fs) - np.sort(f)).max() == 0.0
        else:
            sim.step(1)
            orc.step(1)
        got, den = sim.get_f(0, with_n=True)
        # W_kin, N and the entropy (table logarithm, units of 2^-53)
        for a, b in ((got, orc.f[0]), (den, orc.den[0]), (sim.get_diag()[3:], orc.diag()[3:])):
            assert np.linalg.norm(a - b) < TOL * np.linalg.norm(b), (step, np.linalg.norm(a - b) / np.linalg.norm(b))
    sim.close()
