"""Field solve of a step on grids that are no power of two: the circulant
product over the cluster (up to 1024 cells) and the direct transforms beyond,
E against the oracle's solve of the same rho."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("softening", [True, False], ids=["softened", "plain"])
@pytest.mark.parametrize("nx", [5, 6, 7, 33, 100, 500, 1000, 1023, 1025])
def test_field_of_step(nx, softening):
    import torch
    assert torch.cuda.is_available()
    from paper_1804_03901_gb300 import avl as A
    L = 0.4 * nx
    sim = A.Simulation(A.make_domain(1, nx, L, 0.05, 1.0, softening, A.AVL_FP64),
                       [A.make_species(-1.0, 1.0, (12,), (-4.0,), (4.0,))])
    # a large mean charge (removed by the solve) and two modes
    sim.init_markers(0, (2, 2, 1, 1), A.make_f0([(1.0, (0.0,), (1.0,))], [(1, 0.2, 0.3), (2, 1e-3, 1.0)]), nx)
    for _ in range(2):
        rho, E = sim.get_rho(), sim.get_E()
        ref = O.poisson(nx, L, 1.0, softening, rho)
        # nx products, each rounded to 2^-53 of max |G| max |rho - rho_0|
        assert np.linalg.norm(E - ref) < 1e-12 * np.linalg.norm(ref)
        sim.step(1)
    sim.close()
