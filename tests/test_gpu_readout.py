"""Where lbm_read_macro may write: outputs of different kinds of memory in one
call, and outputs on any byte, give the values of a plain read; and lbm_create
takes its initial temperature from any byte."""
import ctypes as C
import threading
import time

import numpy as np
import pytest

import lbm_cases as lc

pytestmark = pytest.mark.gpu


def _lattice(storage="f32", nx=301, H=68):
    import paper_1510_08224_gb300 as P
    case = lc.rayleigh_benard(nx=nx, H=H, Ra=1e5, sigma=1e-2)
    lat = P.Lattice(case, storage=storage)
    lat.step(40)
    return P, lat


def _output(kind, ny, nx):
    """(the object that owns ny x nx doubles of memory of a kind, their address)."""
    import torch
    if kind == "pageable":
        a = np.full((ny, nx), -1.1)
        return a, a.ctypes.data
    t = torch.full((ny, nx), -1.1, dtype=torch.float64)
    t = t.cuda() if kind == "device" else t.pin_memory()
    return t, t.data_ptr()


def _values(owner):
    return owner if isinstance(owner, np.ndarray) else owner.cpu().numpy()


@pytest.mark.parametrize("kinds", [("pageable", "device", "page-locked", None), ("device", None, "pageable", "pageable"),
                                   ("page-locked", "pageable", None, "device")])
def test_outputs_of_several_kinds_in_one_call(kinds):
    """A pageable output beside a device or a page-locked one: the host handles
    the pages of the pageable one alone."""
    P, lat = _lattice()
    ref = lat.macro()
    outs = [None if k is None else _output(k, lat.ny, lat.nx) for k in kinds]
    ptr = [None if o is None else C.cast(o[1], C.POINTER(C.c_double)) for o in outs]
    assert P.load().lbm_read_macro(lat.handle, *ptr) == 0
    for o, r in zip(outs, ref):
        assert o is None or np.array_equal(_values(o[0]), r)
    lat.close()


@pytest.mark.parametrize("kinds", [("pageable",) * 4, ("page-locked",) * 4, ("device",) * 4,
                                   ("pageable", None, "device", "page-locked")])
@pytest.mark.parametrize("shift", [1, 4])
def test_outputs_on_any_byte(kinds, shift):
    """Outputs that are not on a double's boundary (views into packed buffers)
    take the staging area, whatever memory they lie in."""
    import torch
    P, lat = _lattice()
    ref = lat.macro()
    n = 8 * lat.ny * lat.nx
    outs = []
    for kind in kinds:
        t = torch.full((n + 8,), 7, dtype=torch.uint8, pin_memory=kind == "page-locked")
        outs.append(None if kind is None else t.cuda() if kind == "device" else t)
    ptr = [None if t is None else C.cast(t.data_ptr() + shift, C.POINTER(C.c_double)) for t in outs]
    assert P.load().lbm_read_macro(lat.handle, *ptr) == 0
    for t, r in zip(outs, ref):
        if t is not None:
            b = t.cpu().numpy()
            assert np.array_equal(b[shift:shift + n].copy().view(np.float64).reshape(r.shape), r)
            assert (b[:shift] == 7).all() and (b[shift + n:] == 7).all()
    lat.close()


@pytest.mark.parametrize("kind", ["pageable", "page-locked", "device"])
def test_initial_temperature_on_any_byte(kind):
    """A T_init that is not on a double's boundary is staged, not read in place."""
    import torch
    P, lat = _lattice()
    case = lat.case
    n = 8 * case.ny * case.nx
    t = torch.zeros(n + 8, dtype=torch.uint8, pin_memory=kind == "page-locked")
    t.numpy()[3:3 + n] = np.ascontiguousarray(case.T_init, dtype=np.float64).reshape(-1).view(np.uint8)
    t = t.cuda() if kind == "device" else t
    p, keep = P.make_params(case, "f32")
    p.T_init = t.data_ptr() + 3
    h = C.c_void_p()
    L = P.load()
    assert L.lbm_create(C.byref(p), None, None, C.c_size_t(0), C.byref(h)) == 0
    T = np.zeros((case.ny, case.nx))
    assert L.lbm_read_macro(h, None, None, None, C.cast(T.ctypes.data, C.POINTER(C.c_double))) == 0
    assert np.array_equal(T, P.Lattice(case, storage="f32").macro()[3])
    L.lbm_destroy(h)
    lat.close()
    del keep


@pytest.mark.parametrize("nx,H", [(61, 30), (301, 398)])
def test_pageable_outputs_are_written_in_stream_order(nx, H):
    """Work queued before the read still finds what the outputs held, of a few
    pages or of many."""
    import torch
    P, lat = _lattice(nx=nx, H=H)
    ref = lat.macro()
    outs = [_output("pageable", lat.ny, lat.nx) for _ in range(4)]
    ptr = [C.cast(o[1], C.POINTER(C.c_double)) for o in outs]
    status = []
    torch.cuda._sleep(int(1e9))  # about half a second on the lattice's stream
    reader = threading.Thread(target=lambda: status.append(P.load().lbm_read_macro(lat.handle, *ptr)))
    reader.start()
    time.sleep(0.1)
    seen = [o[0].copy() for o in outs]
    assert reader.is_alive()
    reader.join()
    assert status == [0]
    for s, o, r in zip(seen, outs, ref):
        assert (s == -1.1).all() and np.array_equal(o[0], r)
    lat.close()
