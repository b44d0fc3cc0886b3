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


@pytest.mark.parametrize("w", [1e-3, 1e-4])
def test_adjoint_cell_of_small_weights(A, w):
    """After the step a cell of the last velocity row is reached by one marker
    with weight w alone; there the gradient has terms (f - F) / w.  The mode
    amplitude that puts the marker there comes from the oracle; a short step
    and a strong field keep the markers of the row (v near 0) in their columns."""
    nx, nv, L, seed, jitter, dt, cP = 8, 64, 10.0, 11, 1e-9, 1e-6, 4e5
    dx, dv = L / nx, 0.125
    sp = dict(q=-1.0, m=1.0, nv=(nv,), vmin=((1 - nv) * dv,), vmax=(dv,), mobile=True)
    f0 = lambda amp: dict(beams=[(1.0, (-1.0,), (1.5,))], modes=[(1, amp, 0.3), (2, 0.01, 1.1)])

    def weight(amp):   # of the last row, least over its markers after the push
        x, v, f = O.init_markers(1, nx, L, O.Species(**sp), (1, 1, 1, 1), O.F0(**f0(amp)), 0, seed, jitter)
        orc = O.OracleSim(1, nx, L, dt, [O.Species(**sp)], cP, True)
        orc.set_markers(0, x, v, f)
        orc.refresh()
        E, v = orc.E, np.asarray(v).reshape(-1)
        i0 = np.floor(x / dx - 0.5).astype(int)
        u = x / dx - 0.5 - i0
        t = (v - dt * ((1.0 - u) * E[i0 % nx] + u * E[(i0 + 1) % nx]) - sp["vmin"][0]) / dv - 0.5
        return np.min(t[v > 0.0]) - (nv - 2)

    lo, hi = 0.0, 0.9
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if weight(mid) > w else (lo, mid)
    amp = 0.5 * (lo + hi)
    assert 0.9 * w < weight(amp) < 1.1 * w
    sim = A.Simulation(A.make_domain(1, nx, L, dt, cP, True, 0), [A.make_species(**sp)])
    sim.init_markers(0, (1, 1, 1, 1), A.make_f0(**f0(amp)), seed, jitter)
    J, ga, gu = sim.adjoint(0, A.make_f0(**f0(amp)), 1, 1)
    sim.close()
    Jo, goa, gou, _ = AD.field_energy_gradient(nx, L, dt, [O.Species(**sp)], [O.F0(**f0(amp))], [(1, 1, 1, 1)], seed,
                                               jitter, 0, 1, cP, True)
    g, go = np.concatenate([ga, gu]), np.concatenate([goa, gou])
    # the cell's share of the gradient is about w; its F keeps 2^-52 and w itself
    # 2^-52 / w, whatever w is, and the sums have some 1e2 roundings
    assert J == pytest.approx(Jo, rel=1e-13)
    assert np.max(np.abs(g - go)) < 1e-13 * np.max(np.abs(go)), (g - go, go)
