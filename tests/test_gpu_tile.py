"""The several-steps-per-launch kernels (AUTO, runs of two steps or more)
against the one-cell kernel stepped one launch at a time: the same bits, on
lattices whose sizes sit at the edges of tiles and of their 16-byte copies,
periodic along x, y or both (narrower than a tile too), with fixed, moving and
insulated walls, scattered solids and many walls, for both temperature
lattices, both collisions and both storages, and for every number of steps per
launch and remainder."""
import numpy as np
import pytest

import lbm_cases as lc

pytestmark = pytest.mark.gpu


def _many_walls(count):
    """A cavity whose left wall is cut into pieces of `count` different temperatures."""
    case = lc.cavity(n=40, Ra=1e4, n_y=33, noise=1e-3)
    walls = list(case.walls) + [lc.Wall(0.0, 0.01 * (k % 3), lc.DIRICHLET, k / count) for k in range(count)]
    flags = case.flags.copy()
    for k in range(count):
        flags[1 + k % 33, 0] = 5 + k
    return case.with_(walls=walls, flags=flags)


def _cases():
    kin = dict(s_e=1.3, s_q=1.1, s_eps=1.5, zeta_e=1.2, zeta_nu=0.9)
    return {
        "cavity_20x13": lc.cavity(n=20, Ra=1e4, n_y=13, noise=1e-3),
        "cavity_65x64": lc.cavity(n=65, Ra=1e4, n_y=64, noise=1e-3),
        "rb_133x7": lc.rayleigh_benard(nx=133, H=7, Ra=1e5, sigma=1e-2),
        "rb_30x50": lc.rayleigh_benard(nx=30, H=50, Ra=1e5, sigma=1e-2),
        "rb_3x40": lc.rayleigh_benard(nx=3, H=40, Ra=1e4, sigma=1e-2),
        "couette_5x9": lc.couette(H=9, nx=5, U0=0.05),
        "porous_8x64": lc.porous_couette(H=64),
        "solids_261x19": lc.obstacle_channel(nx=261, H=19, frac=0.15, seed=4),
        "box_7x5": lc.periodic_box(7, 5, nu=0.03, alpha=0.04, g_beta=2e-3, T0=0.5, kinetic=kin, ax=1e-5),
        "box_1x1": lc.periodic_box(1, 1, nu=0.03, alpha=0.04),
        "box_97x41": lc.periodic_box(97, 41, nu=0.02, alpha=0.03, T0=0.2, kinetic=kin, ay=2e-5),
        "walls_15": _many_walls(11),
        "walls_16": _many_walls(12),  # one more than a block keeps: steps one launch at a time
        "cavity_200x150": lc.cavity(n=200, Ra=1e5, n_y=150, noise=1e-3),
    }


CASES = _cases()
MODELS = {"mrt": lambda c: c, "bgk": lc.with_bgk, "q9": lc.with_d2q9_temperature,
          "q9_bgk": lambda c: lc.with_bgk(lc.with_d2q9_temperature(c))}


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("model", list(MODELS))
@pytest.mark.parametrize("name", list(CASES))
def test_runs_equal_single_steps(name, model, storage):
    import paper_1510_08224_gb300 as P
    case = MODELS[model](CASES[name])
    f0, g0 = lc.random_state(case, seed=11)
    a, b = P.Lattice(case, storage=storage), P.Lattice(case, storage=storage)
    b.set_step_kernel("scalar")
    for lat in (a, b):
        lat.set_populations(f0, g0)
    done = 0
    for n in (2, 3, 1, 7, 8, 9, 17):  # every launch size up to 8, odd and even, both starting buffers
        a.step(n)
        for _ in range(n):
            b.step(1)
        done += n
        assert a.info()["steps"] == done
        for u, v in zip(a.populations(), b.populations()):
            assert np.array_equal(u, v), (n, float(np.abs(u - v).max()))
    for u, v in zip(a.macro(), b.macro()):
        assert np.array_equal(u, v)


def test_runs_inside_a_callers_capture():
    """An even run recorded into a caller's CUDA graph and replayed, other even
    runs between the replays."""
    import torch
    import paper_1510_08224_gb300 as P
    case = CASES["cavity_65x64"]
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        a, b = P.Lattice(case, storage="f32", stream=side), P.Lattice(case, storage="f32", stream=side)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            a.step(8)
        for n in (2, 20, 8):
            graph.replay()
            a.step(n)
            b.step(8 + n)
    side.synchronize()
    for u, v in zip(a.populations(), b.populations()):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("model", ["mrt", "q9"])
@pytest.mark.parametrize("name", ["cavity", "box"])
def test_lattices_of_several_waves_of_tiles(name, model, storage):
    """Sizes that take the shapes for many tiles, the last ones ragged."""
    import paper_1510_08224_gb300 as P
    case = MODELS[model](lc.cavity(n=1031, Ra=1e6, n_y=909, noise=1e-3) if name == "cavity" else
                         lc.periodic_box(1021, 903, nu=0.03, alpha=0.04, g_beta=1e-4, T0=0.5, ax=1e-5))
    f0, g0 = lc.random_state(case, seed=5)
    a, b = P.Lattice(case, storage=storage), P.Lattice(case, storage=storage)
    b.set_step_kernel("scalar")
    for lat in (a, b):
        lat.set_populations(f0, g0)
        lat.step(11)
    for u, v in zip(a.populations(), b.populations()):
        assert np.array_equal(u, v), float(np.abs(u - v).max())


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_batch_runs_equal_single_steps_alone(storage):
    """Members whose tiles are ragged, wrap, or have moving and many walls, more
    than one launch takes, joined at odd and even steps."""
    import paper_1510_08224_gb300 as P
    names = ["cavity_20x13", "rb_3x40", "couette_5x9", "solids_261x19", "box_1x1", "rb_133x7", "walls_15"]
    cases = [CASES[names[i % len(names)]] for i in range(69)] + [lc.cavity(n=301, Ra=1e5, n_y=203, noise=1e-3)]
    a = [P.Lattice(c, storage=storage) for c in cases]
    b = [P.Lattice(c, storage=storage) for c in cases]
    batch = P.Batch()
    for i, (case, u, v) in enumerate(zip(cases, a, b)):
        f0, g0 = lc.random_state(case, seed=i)
        v.set_step_kernel("scalar")
        for lat in (u, v):
            lat.set_populations(f0, g0)
            lat.step(i % 3)
        batch.add(u)
    for n in (2, 3, 16):
        batch.step(n)
        for lat in b:
            lat.step(n)
        for u, v in zip(a, b):
            for x, y in zip(u.populations(), v.populations()):
                assert np.array_equal(x, y), n
    batch.close()
