"""GPU adjoint against the oracle's discrete adjoint at the edges of its
kernels: columns fewer than a warp's patch, rows beyond the fixed-point range
of a marker's row, marker counts that are no multiple of a warp, warps whose
markers scatter over more cells than a patch holds, and fields larger than
the FP32 push stages or than the adjoint deposit copies 32 times.

Tolerances as for the adjoint elsewhere: FP64 J within 1e-10 and the gradient
within 1e-8 of its largest component (2^-53 with some 1e3 roundings a value
and the division by the smallest weight sums, about 1e-4 of a marker), FP32
within 2e-3 (2^-24 likewise).
"""
import numpy as np
import pytest

from oracle import adjoint as AD
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1804_03901_gb300 import build
    build.build()
    from paper_1804_03901_gb300 import avl
    return avl


@pytest.mark.parametrize("nx,nv,lat,nsteps,dt,prec", [
    (4, 24, (1, 1), 6, 0.1, 0),
    (4, 24, (1, 1), 6, 0.1, 1),
    (5, 1100, (1, 2), 4, 0.1, 0),      # rows beyond 1023
    (33, 37, (3, 3), 8, 0.1, 0),       # 10989 markers
    (33, 37, (3, 3), 8, 0.1, 1),
    (16, 24, (2, 1), 6, 1.0, 0),       # a warp spans the grid
    (1100, 24, (1, 1), 2, 0.1, 0),     # four copies of e
    (2100, 24, (1, 1), 2, 0.1, 1),     # field read from global memory, four copies of e
])
def test_adjoint_edges(A, nx, nv, lat, nsteps, dt, prec):
    L, seed = 10.0, 11
    species = [dict(q=-1.0, m=1.0, nv=(nv,), vmin=(-5.0,), vmax=(5.0,), mobile=True),
               dict(q=1.0, m=100.0, nv=(8,), vmin=(-0.5,), vmax=(0.5,), mobile=False)]
    f0s = [dict(beams=[(0.5, (1.5,), (0.6,)), (0.5, (-1.5,), (0.6,))], modes=[(1, 0.02, 0.3), (2, 0.01, 1.1)]),
           dict(beams=[(1.0, (0.0,), (0.1,))], modes=[(1, 0.005, 0.0)])]
    lattices = [lat + (1, 1), (1, 1, 1, 1)]
    sim = A.Simulation(A.make_domain(1, nx, L, dt, 1.0, True, prec), [A.make_species(**sp) for sp in species])
    for s in range(2):
        sim.init_markers(s, lattices[s], A.make_f0(**f0s[s]), seed, 1.0)
    J, ga, gu = sim.adjoint(0, A.make_f0(**f0s[0]), nsteps, 3)
    sim.close()
    Jo, goa, gou, _ = AD.field_energy_gradient(nx, L, dt, [O.Species(**sp) for sp in species],
                                               [O.F0(**f) for f in f0s], lattices, seed, 1.0, 0, nsteps)
    g, go = np.concatenate([ga, gu]), np.concatenate([goa, gou])
    tolJ, tolg = (1e-10, 1e-8) if prec == 0 else (2e-3, 2e-3)
    assert J == pytest.approx(Jo, rel=tolJ)
    assert np.max(np.abs(g - go)) < tolg * np.max(np.abs(go)), (g, go)
