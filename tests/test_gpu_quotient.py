"""Integer logarithm of the FP64 finalize: the entropy sum f log f where log f is
small."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def simulation(nx, nv):
    import torch
    assert torch.cuda.is_available()
    from paper_1804_03901_gb300 import avl as A
    vmin = tuple(-(n // 2) * 1.0 for n in nv)
    vmax = tuple(a + n for a, n in zip(vmin, nv))
    return vmin, A.Simulation(A.make_domain(len(nv), nx, float(nx), 0.01, precision=A.AVL_FP64),
                              [A.make_species(-1.0, 1.0, nv, vmin, vmax)])


@pytest.mark.parametrize("nv", [(24,), (8, 3, 2)])
@pytest.mark.parametrize("lo,hi", [(1e-9, 1e-8), (1e-6, 2e-6), (-2e-3, -1e-3), (0.01, 0.1), (-0.1249, 0.1249),
                                   (0.12, 0.13), (-0.13, -0.12), (-0.9, 3.0), (1e3, 1e9)])
def test_entropy(nv, lo, hi):
    nx = 32
    vmin, sim = simulation(nx, nv)
    at = np.meshgrid(np.arange(nx) + 0.5, *[a + np.arange(n) + 0.5 for a, n in zip(vmin, nv)], indexing="ij")
    f = 1.0 + np.random.default_rng(1).uniform(lo, hi, at[0].size)
    sim.set_markers(0, at[0].ravel(), np.array([a.ravel() for a in at[1:]]), f)
    s = [v * math.log1p(v - 1.0) if 0.5 < v < 2.0 else v * math.log(v) for v in f]   # (v - 1: exact)
    # log f within 2^-51 of itself or, outside 1 -+ 1/8, within 2^-52; sums of 8e2
    # or 1.5e3 terms in trees and groups of at most 64
    tol = 2.0 ** -47 * math.fsum(abs(v) for v in s)
    assert abs(sim.get_diag()[5] - math.fsum(s)) < tol
    sim.close()
