"""The engine's host side without a GPU: creating it, queueing and cancelling jobs make no call that
needs a device (what runs on the GPU is set up when the first job runs)."""
import ctypes as C

import pytest

from paper_1804_01184_gb300 import engine, fwi


@pytest.fixture
def L(monkeypatch):
    from paper_1804_01184_gb300 import build
    try:
        path = build.build()
    except RuntimeError as e:   # no nvcc on this machine
        pytest.skip(str(e))
    monkeypatch.setattr(fwi, "_lib", fwi._open(path))
    monkeypatch.setattr(engine, "_bound", False)
    return engine._lib()


def test_create_submit_cancel(L):
    h, t = C.c_void_p(), C.c_longlong()
    assert L.fwi_engine_create(C.byref(h), C.c_void_p(1 << 20), 1 << 30, None) == 0, L.fwi_last_error()
    J = engine._Job()
    J.kind, J.grid, J.pz = engine.JOB_MODEL, fwi.make_grid(64, 48, 5.0, 5e-4, 100, sponge=8), 0
    J.xi_a = J.xi_b = J.traces = 1 << 21                     # never read: the job does not run
    J.src, J.rec = fwi._Sources(1, 1 << 21, 1 << 21), fwi._Receivers(2, 1 << 21)
    assert L.fwi_engine_submit(h, C.byref(J), C.byref(t)) == 0, L.fwi_last_error()
    q, r, p, u = C.c_int(), C.c_int(), C.c_int(), C.c_size_t()
    assert L.fwi_engine_info(h, C.byref(q), C.byref(r), C.byref(p), C.byref(u)) == 0
    assert (q.value, r.value, p.value, u.value) == (1, 0, 0, 0)
    assert L.fwi_engine_cancel(h, t) == 0
    assert L.fwi_engine_cancel(h, t) != 0
    L.fwi_engine_destroy(h)
