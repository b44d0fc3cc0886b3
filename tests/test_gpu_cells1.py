"""FP64 1d1v deposit cell by cell: f and n of every reached cell relative to
the oracle's, where norms over the grid would not see them -- sparse cells
that only small weights reach beside a dense core, in chunks of any size,
dense cells whose counts carry out of a word, and the counter of out-of-window
runs."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu

NX, NV, VMIN, VMAX = 64, 64, -32.0, 32.0   # cells of size 1: positions and weights are exact counts


def simulation(dt=0.001, nx=NX):
    from paper_1804_03901_gb300 import avl as A
    sim = A.Simulation(A.make_domain(1, nx, float(nx), dt, precision=A.AVL_FP64),
                       [A.make_species(-1.0, 1.0, (NV,), (VMIN,), (VMAX,))])
    return sim, O.OracleSim(1, nx, float(nx), dt, [O.Species(-1.0, 1.0, (NV,), (VMIN,), (VMAX,))])


def dyadic(w):
    return np.round(np.asarray(w) * 2.0 ** 30) / 2.0 ** 30


def compare(sim, orc, tol_f, tol_n):
    got, n = sim.get_f(0, with_n=True)
    ref, den = orc.f[0], orc.den[0]
    reached = den > 0
    assert np.array_equal(n > 0, reached)
    err_f = np.max(np.abs(got - ref)[reached] / np.abs(ref)[reached])
    err_n = np.max(np.abs(n - den)[reached] / den[reached])
    assert err_f < tol_f and err_n < tol_n, (err_f, err_n)


@pytest.mark.parametrize("chunk", [0, 64, 1 << 17])
def test_sparse_cells(chunk, monkeypatch):
    import torch
    assert torch.cuda.is_available()
    if chunk:
        monkeypatch.setenv("AVL_CHUNK_M", str(chunk))
    rng = np.random.default_rng(11)
    n = 100000 if chunk != 64 else 3000
    # the core: rows 8 to 39; beyond it lone markers, three cells apart
    x, v = [dyadic(rng.uniform(0.0, NX, n))], [dyadic(rng.uniform(-24.0, 8.0, n))]
    k = 0
    for w in (1e-2, 1e-3, 1e-4, 1e-5, 1e-6):
        for a, b in ((w, 0.37), (0.37, w), (w, w)):
            for side in (14.5, 20.5, 26.5):
                x.append([3 * (k % 20) + 0.5 + dyadic(a)])
                v.append([side + 3 * (k // 20 % 2) + dyadic(b)])
                k += 1
    x, v = np.concatenate(x), np.concatenate(v)
    f = rng.uniform(0.5, 2.0, x.size)
    sim, orc = simulation()
    sim.set_markers(0, x, v, f)
    orc.set_markers(0, x, v, f)
    orc.refresh()
    # integer weights of at least 2^-24 are within 3/4 2^-57 (smaller ones are FP64
    # products); f takes the same weights above and below
    compare(sim, orc, 1e-11, 1e-10)
    for _ in range(2):
        xs, vs, fs = sim.get_markers(0)
        orc.set_markers(0, xs, vs[0], fs)
        orc.refresh()
        sim.step(1)
        orc.step(1)
        # weights of 1e-6 carry the rounding of x and of the rows, some 2^-47
        compare(sim, orc, 1e-7, 1e-7)
    sim.close()


def test_dense_cells(monkeypatch):
    """Thousands of markers of a chunk per cell: sums of weights far beyond 64-bit counts of 2^-57."""
    monkeypatch.setenv("AVL_CHUNK_M", "16384")
    rng = np.random.default_rng(12)
    n = 60000
    x, v = dyadic(rng.uniform(0.0, 4.0, n)), dyadic(rng.uniform(-1.0, 1.0, n))
    f = rng.uniform(0.5, 2.0, n)
    sim, orc = simulation(nx=4)
    sim.set_markers(0, x, v, f)
    orc.set_markers(0, x, v, f)
    orc.refresh()
    compare(sim, orc, 1e-11, 1e-11)   # sums of 2e4 terms in any order
    sim.step(1)
    xs, vs, fs = sim.get_markers(0)
    orc.set_markers(0, xs, vs[0], fs)
    orc.refresh()
    compare(sim, orc, 1e-9, 1e-9)
    sim.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kinds,runs", [((0, 0, 0, 0), 1), ((0, 0, 1, 1), 2), ((0, 1, 0, 1), 4)])
def test_out_of_window_runs(kinds, runs, precision, monkeypatch):
    """The counter of avl_get_stats: runs of consecutive markers with the same
    cells that miss their chunk's window, in either precision."""
    from paper_1804_03901_gb300 import avl as A
    monkeypatch.setenv("AVL_WMAX", "6")
    prec = A.AVL_FP64 if precision == "fp64" else A.AVL_FP32
    sim = A.Simulation(A.make_domain(1, NX, float(NX), 1e-4, precision=prec),
                       [A.make_species(-1.0, 1.0, (NV,), (VMIN,), (VMAX,))])
    x = np.concatenate([np.arange(60) + 0.75, 10.75 + 20.0 * np.array(kinds)])
    v = np.concatenate([np.full(60, VMIN + 20.75), np.full(4, VMIN + 50.75)])
    sim.set_markers(0, x, v, np.ones(64))
    sim.step(1)
    assert sim.get_stats()[0][0] == runs
    sim.close()
