"""FP32 charge and marker number as sums of f: the blocks of a finalize add in
FP64, so sums that FP64 holds exactly (f in 24 bits at two scales, cells of
size 1, one marker at every cell centre) come out exactly."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nv", [(16, (8,)), (40, (24,)), (32, (8, 2, 2)), (33, (6, 3, 4))])
def test_sums_are_exact(nx, nv):
    import torch
    assert torch.cuda.is_available()
    from paper_1804_03901_gb300 import avl as A
    vmin = tuple(-(n // 2) * 1.0 for n in nv)
    vmax = tuple(a + n for a, n in zip(vmin, nv))
    sim = A.Simulation(A.make_domain(len(nv), nx, float(nx), 0.01, precision=A.AVL_FP32),
                       [A.make_species(-1.0, 1.0, nv, vmin, vmax)])
    at = np.meshgrid(np.arange(nx) + 0.5, *[a + np.arange(n) + 0.5 for a, n in zip(vmin, nv)], indexing="ij")
    n = at[0].size
    rng = np.random.default_rng(n)
    # 24 bits below 2 in one of 16 cells, below 2^-20 in the others: multiples of
    # 2^-44, sums below 2^9
    f = rng.integers(1 << 23, 1 << 24, n) * np.where(np.arange(n) % 16 == 5, 2.0 ** -23, 2.0 ** -44)
    sim.set_markers(0, at[0].ravel(), np.array([a.ravel() for a in at[1:]]), f)
    got = sim.get_f(0)
    assert np.array_equal(got.ravel(), f)
    assert sim.get_diag()[4] == math.fsum(f)
    rho = [-math.fsum(c) for c in got.reshape(nx, -1)]
    assert np.array_equal(sim.get_rho(), rho)
    sim.close()
