"""Integer quotient and logarithm of the FP64 finalize: f = num / den rounded
to nearest where num and den are exact (dyadic weights and values), and the
entropy sum f log f where log f is small."""
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


@pytest.mark.parametrize("nx,nv,n", [(256, (128,), 150000), (61, (7,), 3000)])
def test_quotient_to_nearest(nx, nv, n):
    vmin, sim = simulation(nx, nv)
    rng = np.random.default_rng(n)
    # weights in x of 20 bits, none in v; values of 18 bits: sums of fewer than 2^14
    # products are exact
    i, w = rng.integers(0, nx - 1, n), rng.integers(1, 1 << 20, n) / 2.0 ** 20
    row = rng.integers(0, nv[0], n)
    f = rng.integers(1 << 17, 1 << 18, n) / 2.0 ** 17
    sim.set_markers(0, i + 0.5 + w, vmin[0] + row + 0.5, f)
    num, den = np.zeros((nx, nv[0])), np.zeros((nx, nv[0]))
    for k, a in ((i, 1.0 - w), (i + 1, w)):
        np.add.at(num, (k, row), a * f)
        np.add.at(den, (k, row), a)
    got, d = sim.get_f(0, with_n=True)
    assert np.array_equal(d, den)
    assert np.array_equal(got, np.divide(num, den, out=np.zeros_like(num), where=den > 0))
    sim.close()


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
