"""The bounds-checked debug build on both kinds of time step: on chip (mailbox words, rows of shared
memory, fields) and streaming.  Nothing is reported, and the results are bitwise the default build's."""
import ctypes

import numpy as np
import pytest

from paper_1804_01184_gb300 import inputs as I
from tests._common import gpu_grid
from tests.test_gpu_resident import GRIDS, case, kernels

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_01184_gb300 import build, fwi
    build.build(checked=True)
    return fwi


def calls(F, nx, nz, order, sponge):
    w = case(nx, nz, order, sponge, nt=40)
    hi = np.array([(nx - 1) * w.dx, (nz - 1) * w.dx])
    more = (hi * np.random.default_rng(3).random((90, 2))).astype(np.float32)   # more than a tile lists
    w.rec_xy = np.concatenate([w.rec_xy, more, more[::5]]).astype(np.float32)
    g, nr = gpu_grid(w), len(w.rec_xy)
    ar, tail = (g, w.pz, w.xi_a, w.xi_b), (w.src_xy, w.wavelet, w.rec_xy)
    d = [I.random_like(w.xi_a.shape, s, 0.05) for s in (1, 2)]
    res = I.random_like((w.ns, nr, w.nt), 11, 1.0)
    return lambda: (F.fwi_model(*ar, *tail), F.fwi_born(*ar, *d, *tail), F.fwi_adjoint(*ar, *tail, res),
                    *F.fwi_gradient(*ar, *tail, res))


@pytest.mark.parametrize("tz", [0, 40])     # on chip; a fixed strip height asks for the streaming kernels
@pytest.mark.parametrize("nx,nz,order,sponge", GRIDS + [(240, 150, 8, 6)])
def test_single_calls(F, nx, nz, order, sponge, tz):
    from paper_1804_01184_gb300 import build
    call = calls(F, nx, nz, order, sponge)
    ref = call()
    with F.library(build.LIB_CHECKED):
        F.fwi_set_tile(tz, 0)               # the debug build's own setting
        try:
            got, used = kernels(F, call)    # every call checks its status: a caught access raises
        finally:
            F.fwi_set_tile(0, 0)
    want = {"k_res_fwd", "k_res_born", "k_res_adj"} if tz == 0 else set()
    assert {k.split("::")[-1].split("<")[0] for k in used if "k_res_" in k} == want, used
    assert all(torch.equal(x, y) for x, y in zip(got, ref))


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("op", ["model", "born", "gradient"])
def test_engine(F, op, order):
    """The engine's kernels and its mailboxes cut to the tiles; its one job has the arena's first block,
    which begins with the job's status word."""
    from paper_1804_01184_gb300 import build, engine
    w = case(170, 110, order, 10, ns=3, nr=20, nt=60)
    g = gpu_grid(w)
    ar, tail = (g, w.pz, w.xi_a, w.xi_b), (w.src_xy, w.wavelet, w.rec_xy)
    d = [I.random_like(w.xi_a.shape, s, 0.05) for s in (1, 2)]
    data = I.random_like((w.ns, w.nr, w.nt), 3, 1.0)
    ref = {"model": lambda: (F.fwi_model(*ar, *tail),), "born": lambda: (F.fwi_born(*ar, *d, *tail),),
           "gradient": lambda: F.fwi_gradient(*ar, *tail, data)}[op]()
    with F.library(build.LIB_CHECKED):
        engine._bound = False               # bind the engine's entry points in this library
        try:
            E = engine.Engine(1 << 30)
            if op == "model":
                E.submit_model(*ar, *tail, work_budget=1 << 28)
            elif op == "born":
                E.submit_born(*ar, *d, *tail, work_budget=1 << 28)
            else:
                E.submit_gradient(*ar, *tail, data, work_budget=1 << 28)
            (out,), used = kernels(F, lambda: E.drain(256))
            status = ctypes.c_int.from_buffer_copy(E.arena[:4].cpu().numpy().tobytes()).value
            E.close()
        finally:
            engine._bound = False
    assert any("k_res_" in k for k in used), used
    assert status == 0
    got = (out.traces,) if out.traces is not None else (out.misfit, out.grads)
    assert all(torch.equal(x, y) for x, y in zip(got, ref))
