"""A region's copy that does not arrive in time (launches of several steps): the
test hook makes every block record that; the kernel returns normally, the next
synchronising call reports LBM_ETIMEOUT once, and the lattice works again. In a batch both the batch and the member report."""
import numpy as np
import pytest

import lbm_cases as lc

pytestmark = pytest.mark.gpu
ETIMEOUT = 5


def _timed_out(P, call):
    with pytest.raises(P.LBMError) as e:
        call()
    assert e.value.status == ETIMEOUT


def _case(name):
    if name == "box":  # no walls: no barrier between the wait and the last step of a one-step launch
        return lc.periodic_box(97, 200, nu=0.03, alpha=0.04)
    return lc.cavity(n=65, Ra=1e4, n_y=64, noise=1e-3)


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("name", ["box", "cavity"])
@pytest.mark.parametrize("steps", [2, 3, 8])
def test_late_copy_is_reported_once(name, storage, steps):
    import torch
    import paper_1510_08224_gb300 as P
    case = _case(name)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        a, b = P.Lattice(case, storage=storage, stream=side), P.Lattice(case, storage=storage, stream=side)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):  # from here on a run of an even length ends on its first buffer
            a.step(2)
        assert a.steps_per_launch() > 1
        a.debug_late_copies(True)
        a.step(2 * steps)
        _timed_out(P, lambda: P.lbm._check(P.load().lbm_sync(a.handle), a.handle))
        a.step(2 * steps)
        _timed_out(P, a.macro)
        a.debug_late_copies(False)
        f0, g0 = lc.random_state(case, seed=3)
        for lat in (a, b):
            lat.set_populations(f0, g0)
            lat.step(steps)
    side.synchronize()
    for u, v in zip(a.populations(), b.populations()):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("first", ["member", "batch"])
def test_late_copy_of_a_member_is_reported_by_member_and_batch(first, storage):
    import paper_1510_08224_gb300 as P
    cases = [_case("cavity"), _case("box"), lc.cavity(n=40, Ra=1e4, noise=1e-3)]
    lats = [P.Lattice(c, storage=storage) for c in cases]
    lats[1].debug_late_copies(True)
    b = P.Batch()
    for lat in lats:
        b.add(lat)
    with pytest.raises(P.LBMError):  # a member's hook is set before it joins
        lats[1].debug_late_copies(False)
    b.step(8)
    lats[0].macro(), lats[2].residual()
    if first == "member":
        for read in (lats[1].macro, b.sync):
            _timed_out(P, read)
    else:
        _timed_out(P, b.residuals)
    b.sync()
    for lat in lats:  # reported once
        lat.macro()
    b.remove(lats[1])
    lats[1].debug_late_copies(False)
    b.add(lats[1])
    states = [lc.random_state(c, seed=20 + i) for i, c in enumerate(cases)]
    for lat, s in zip(lats, states):
        lat.set_populations(*s)
    b.step(8)
    b.sync()
    for lat, c, s in zip(lats, cases, states):
        ref = P.Lattice(c, storage=storage)
        ref.set_populations(*s)
        ref.step(8)
        for u, v in zip(lat.populations(), ref.populations()):
            assert np.array_equal(u, v)
    b.close()
