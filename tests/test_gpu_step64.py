"""The FP64 step's boundary nodes in a grid of several waves, launched as a
programmatic dependent of the step before it (node-based walls, more than about
389,000 cells), against the oracle."""
import numpy as np
import pytest

import lbm_cases as lc
import oracle

pytestmark = pytest.mark.gpu
FP64_TOL = 1e-12  # relative max-norm, as on the smaller lattices


@pytest.mark.parametrize("model", ["mrt", "bgk", "q9"])
def test_boundary_nodes_of_a_large_lattice(model):
    import paper_1510_08224_gb300 as P
    case = lc.cavity_nee(n=640, Ra=1e5, noise=1e-3)
    case = {"mrt": lambda c: c, "bgk": lc.with_bgk, "q9": lc.with_d2q9_temperature}[model](case)
    f0, g0 = lc.random_state(case, seed=13, amp_f=0.002, amp_g=0.005)
    a, o = P.Lattice(case, storage="f64"), oracle.OracleLattice(case)
    for lat in (a, o):
        lat.set_populations(f0, g0)
    for n in (1, 2, 41):  # launched directly, then replayed as graphs too
        a.step(n)
        o.step(n)
        for u, v in zip(a.populations(), o.populations()):
            assert np.abs(u - v).max() <= FP64_TOL * np.abs(v).max(), n
