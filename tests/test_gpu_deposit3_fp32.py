"""FP32 1d3v push and deposit at the edges of its chunks: segments of many
chunks, one to four columns per thread with columns left over, and steps in
which more markers leave their row than a chunk keeps in shared memory; grids
against the oracle from the library's own markers."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1804_03901_gb300 import inputs

pytestmark = pytest.mark.gpu

# positions and rows are rounded to 2^-24 of a cell, which enters f through
# the spread of the values in a cell and its smallest weight sums: 1e-5 as for
# the other FP32 grids
TOL = 1e-5


@pytest.mark.parametrize("nx,nv,n,dt", [(4, (3, 2, 2), 20000, 0.07), (33, (8, 2, 2), 30000, 0.6),
                                        (256, (3, 2, 2), 60000, 0.07), (256, (8, 2, 3), 90000, 0.6),
                                        (300, (4, 2, 2), 40000, 0.3), (700, (4, 2, 2), 60000, 0.3)])
def test_deposit3_fp32(nx, nv, n, dt):
    import torch
    assert torch.cuda.is_available()
    from paper_1804_03901_gb300 import avl as A
    L, vmin, vmax = 0.4 * nx, (-3.0, -2.0, -2.5), (3.0, 2.0, 1.5)
    sim = A.Simulation(A.make_domain(3, nx, L, dt, precision=A.AVL_FP32), [A.make_species(-1.0, 1.0, nv, vmin, vmax)])
    orc = O.OracleSim(3, nx, L, dt, [O.Species(-1.0, 1.0, nv, vmin, vmax)])
    x, v, _ = inputs.random_markers3(17 * nx + n, n, L, vmin, vmax)
    f = np.exp(-0.5 * (v ** 2).sum(0)) * (1.0 + 0.3 * np.cos(2 * np.pi * x / L))
    sim.set_markers(0, x, v, f)
    for step in range(3):
        orc.set_markers(0, *sim.get_markers(0))
        orc.refresh()
        if step:
            sim.step(1)
            orc.step(1)
        got, den = sim.get_f(0, with_n=True)
        for a, b in ((got, orc.f[0]), (den, orc.den[0])):
            assert np.linalg.norm(a - b) < TOL * np.linalg.norm(b), (step, np.linalg.norm(a - b) / np.linalg.norm(b))
    sim.close()
