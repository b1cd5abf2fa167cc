"""Which runs take several steps per launch, where that depends on more than
the kind of lattice; the bits are those of single steps either way."""
import numpy as np
import pytest

import lbm_cases as lc

pytestmark = pytest.mark.gpu


def _same_as_single_steps(case, storage, runs, prepare=lambda lat: None):
    import paper_1510_08224_gb300 as P
    f0, g0 = lc.random_state(case, seed=7)
    a, b = P.Lattice(case, storage=storage), P.Lattice(case, storage=storage)
    b.set_step_kernel("scalar")
    prepare(a)
    for n in runs:
        for lat in (a, b):
            lat.set_populations(f0, g0)
            lat.step(n)
        for u, v in zip(a.populations(), b.populations()):
            assert np.array_equal(u, v), n
    per = a.steps_per_launch()
    a.close(), b.close()
    return per


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("model", ["mrt", "q9"])
def test_wide_lattices_of_few_rows_take_single_steps(model, storage):
    """A tile of many rows is mostly idle on a wide lattice of one to a few,
    also as a member of a batch; short ones of as few rows, and tall ones of
    few columns, take the tiles."""
    import paper_1510_08224_gb300 as P
    q9 = lc.with_d2q9_temperature if model == "q9" else (lambda c: c)
    kin = dict(s_e=1.3, s_q=1.1, s_eps=1.5, zeta_e=1.2, zeta_nu=0.9)
    wide = [q9(lc.rayleigh_benard(nx=150000, H=2, Ra=1e4, sigma=1e-2)),
            q9(lc.periodic_box(300001, 1, nu=0.03, alpha=0.04, kinetic=kin))]
    for case in wide:
        assert _same_as_single_steps(case, storage, (2, 9)) == 1
    for case in (q9(lc.rayleigh_benard(nx=1000, H=2, Ra=1e4, sigma=1e-2)),
                 q9(lc.rayleigh_benard(nx=4, H=5000, Ra=1e4, sigma=1e-2))):
        assert _same_as_single_steps(case, storage, (2, 9)) > 1
    if model == "mrt":
        b = P.Batch()
        lats = [P.Lattice(c, storage=storage) for c in (wide[0], lc.cavity(n=40, Ra=1e4, noise=1e-3))]
        for lat in lats:
            b.add(lat)
        assert b.steps_per_launch() == 1
        b.remove(lats[0])
        assert b.steps_per_launch() > 1
        b.close()


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("side", [60, 700])
def test_two_steps_that_end_on_their_first_buffer(side, storage):
    """A batch's run of two steps, and a lattice's once a run was recorded: two
    launches of one step on small lattices, single steps on large ones."""
    import torch
    import paper_1510_08224_gb300 as P
    case = lc.cavity(n=side, n_y=side - 9, Ra=1e4, noise=1e-3)
    f0, g0 = lc.random_state(case, seed=9)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        a, b, c = (P.Lattice(case, storage=storage, stream=stream) for _ in range(3))
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            a.step(2)
        batch = P.Batch(stream=stream)
        c.set_step_kernel("scalar")
        for lat in (a, b, c):
            lat.set_populations(f0, g0)
        batch.add(b)
        for n in (2, 2, 3, 1, 2):  # ends on the buffer the recorded run began on
            a.step(n), batch.step(n), c.step(n)
        graph.replay(), c.step(2), batch.step(2)
    stream.synchronize()
    want = c.populations()
    for lat in (a, b):
        for u, v in zip(lat.populations(), want):
            assert np.array_equal(u, v)
    batch.close()


def test_two_steps_of_a_large_half_precision_lattice():
    """Single steps for a run of two, the tiles for longer ones."""
    case = lc.with_d2q9_temperature(lc.cavity(n=1001, n_y=990, Ra=1e5, noise=1e-3))
    assert _same_as_single_steps(case, "f16", (2, 3, 8)) > 1
