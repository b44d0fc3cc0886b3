"""FP64 1d3v deposit cell by cell: f and n of every reached cell relative to
the oracle's, where norms over the grid would not see them -- markers alone in
their cells with weights from 1e-2 to 1e-6 in one to four directions."""
import itertools

import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu

NX, NV, VMIN, VMAX = 64, (48, 4, 4), (-24.0, -2.0, -2.0), (24.0, 2.0, 2.0)   # cells of size 1: positions
                                                                            # and weights are exact counts


def simulation(dt=0.001, softening=True):
    from paper_1804_03901_gb300 import avl as A
    sim = A.Simulation(A.make_domain(3, NX, float(NX), dt, 1.0, softening, A.AVL_FP64),
                       [A.make_species(-1.0, 1.0, NV, VMIN, VMAX)])
    return sim, O.OracleSim(3, NX, float(NX), dt, [O.Species(-1.0, 1.0, NV, VMIN, VMAX)])


def dyadic(w):
    return np.round(np.asarray(w) * 2.0 ** 30) / 2.0 ** 30


def lone_markers():
    """One marker for each set of directions (weight w of the next cell there, 0.37
    elsewhere) and each w, three cells apart in x and v_x."""
    x, v, k = [], [], 0
    for w in (1e-2, 1e-3, 1e-4, 1e-5, 1e-6):
        for dirs in itertools.product((0, 1), repeat=4):
            if not any(dirs):
                continue
            c = [dyadic(w if d else 0.37) for d in dirs]
            x.append(3 * (k % 20) + 0.5 + c[0])
            v.append([-22.5 + 3 * (k // 20) + c[1], -0.5 + c[2], -0.5 + c[3]])
            k += 1
    f = np.random.default_rng(3).uniform(0.5, 2.0, k)
    return np.array(x), np.array(v).T.copy(), f


def compare(sim, orc, tol_f, tol_n):
    got, n = sim.get_f(0, with_n=True)
    ref, den = orc.f[0], orc.den[0]
    reached = den > 0
    assert np.array_equal(n > 0, reached)
    err_f = np.max(np.abs(got - ref)[reached] / np.abs(ref)[reached])
    err_n = np.max(np.abs(n - den)[reached] / den[reached])
    assert err_f < tol_f and err_n < tol_n, (err_f, err_n)


@pytest.mark.parametrize("B", [None, (0.3, -0.9, 1.4)], ids=["kick", "boris"])
def test_lone_markers(B):
    import torch
    assert torch.cuda.is_available()
    sim, orc = simulation()
    x, v, f = lone_markers()
    sim.set_markers(0, x, v, f)
    if B:
        sim.set_bfield(B)
        orc.B = np.array(B)
    orc.set_markers(0, x, v, f)
    orc.refresh()
    # a sum of integer weights of at least 2^-20 has an error of a few 2^-57
    # (smaller weights are FP64 products), and f carries that of both sums
    compare(sim, orc, 1e-10, 1e-10)
    for _ in range(3):
        xs, vs, fs = sim.get_markers(0)
        orc.set_markers(0, xs, vs, fs)
        orc.refresh()
        sim.step(1)
        orc.step(1)
        # n carries the rounding of x and of the rows, some 2^-48 of a cell here,
        # over weights of 1e-6
        compare(sim, orc, 1e-10, 1e-7)
    sim.close()


@pytest.mark.parametrize("where", ["vx up", "vx down", "x"])
@pytest.mark.parametrize("fall", [1e6, 1e18])
def test_steep_values(where, fall):
    """f falls by `fall` from one v_x row or one x column to the next."""
    sim, orc = simulation()
    rng = np.random.default_rng(5)
    n = 30000
    x = dyadic(rng.uniform(0.0, 16.0, n))
    v = dyadic(np.array([rng.uniform(-8.0, 4.0, n), rng.uniform(-2.0, 2.0, n), rng.uniform(-2.0, 2.0, n)]))
    at = np.floor(x) if where == "x" else np.floor(v[0]) if where == "vx up" else -np.floor(v[0])
    f = fall ** (at / 1.0 - at.max()) * rng.uniform(0.5, 2.0, n)
    sim.set_markers(0, x, v, f)
    orc.set_markers(0, x, v, f)
    orc.refresh()
    # the unit of a column's sums is 2^-56 of the largest value, which reaches the
    # cell with a weight of at least 2^-20: some 20 markers of 1.5 x 2^-36
    compare(sim, orc, 1e-9, 1e-10)
    sim.close()


def test_value_range():
    sim, orc = simulation()
    k = np.arange(8)
    x, v = 3 * k + 0.5 + dyadic(0.3), np.array([-20.5 + 3 * k + dyadic(0.4), 0 * k + dyadic(0.3) - 0.5, 0 * k - 0.75])
    f = np.array([1.0, 1e-305, -3e-300, 1e-290, 1e140, -1e130, 0.0, 1e-60])
    sim.set_markers(0, x, v, f)
    orc.set_markers(0, x, v, f)
    orc.refresh()
    got, ref, den = sim.get_f(0), orc.f[0], orc.den[0]
    assert np.all(np.abs(got - ref)[den > 0] <= 1e-12 * np.abs(ref)[den > 0])
    sim.close()


def test_overflow_is_reported():
    """Five markers whose weighted values add up beyond the range: f is infinite
    and the call says so."""
    from paper_1804_03901_gb300 import avl as A
    sim, _ = simulation()
    with pytest.raises(A.AvlError) as e:
        sim.set_markers(0, np.full(5, 4.5), np.full((3, 5), -0.5), np.full(5, 1.7e308))
        sim.synchronize()
    assert e.value.status == A.AVL_ENUMERIC
    sim.close()
