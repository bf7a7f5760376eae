"""Streams that hold part of the GPU's SMs (green contexts): launches that need more at once, the
on-chip steps' cooperative ones and the misfit's cluster, have another way.  Results as on the whole
GPU.  (Waits are kept short, so that blocks that did not run together would end by themselves.)"""
import ctypes as C

import numpy as np
import pytest

from paper_1804_01184_gb300 import inputs as I
from tests._common import gpu_grid

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_01184_gb300 import build, fwi
    build.build()
    torch.zeros(1, device="cuda")
    return fwi


@pytest.fixture(params=[8, 32])
def part(F, request):
    """A stream of request.param SMs (opaque driver structures in buffers larger than they are)."""
    L = C.CDLL("libcuda.so.1")
    if not hasattr(L, "cuGreenCtxStreamCreate"):
        pytest.skip("no green contexts")
    full, some, rest = (C.create_string_buffer(4096) for _ in range(3))
    dev, n, desc, ctx, st = C.c_int(), C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()
    ok = L.cuDeviceGet(C.byref(dev), torch.cuda.current_device()) == 0 and L.cuDeviceGetDevResource(dev, full, 1) == 0
    ok = ok and L.cuDevSmResourceSplitByCount(some, C.byref(n), full, rest, C.c_uint(0), C.c_uint(request.param)) == 0
    ok = ok and L.cuDevResourceGenerateDesc(C.byref(desc), some, C.c_uint(1)) == 0
    ok = ok and L.cuGreenCtxCreate(C.byref(ctx), desc, dev, C.c_uint(1)) == 0
    if not ok or L.cuGreenCtxStreamCreate(C.byref(st), ctx, C.c_uint(1), C.c_int(0)) != 0:
        pytest.skip("no stream of part of the GPU here")
    F.fwi_set_wait_limit(2000)
    stream = torch.cuda.ExternalStream(st.value)
    yield stream
    F.fwi_set_wait_limit(-1)
    torch.cuda.synchronize()
    L.cuStreamDestroy_v2(st)
    L.cuGreenCtxDestroy(ctx)


def test_calls_and_engine(F, part):
    from paper_1804_01184_gb300 import engine
    w = I.small_case(seed=41, nx=161, nz=140, nt=50, order=8, sponge=20, ns=6, nr=9)
    g = gpu_grid(w)
    ar, tail = (g, w.pz, w.xi_a, w.xi_b), (w.src_xy, w.wavelet, w.rec_xy)
    d = [I.random_like(w.xi_a.shape, s, 0.05) for s in (1, 2)]
    data = I.random_like((w.ns, w.nr, w.nt), 3, 1.0)
    calls = lambda: (F.fwi_model(*ar, *tail), F.fwi_born(*ar, *d, *tail), *F.fwi_gradient(*ar, *tail, data))
    ref = calls()
    torch.cuda.synchronize()
    with torch.cuda.stream(part):
        got = calls()
    assert all(torch.equal(x, y) for x, y in zip(got, ref))
    E = engine.Engine(1 << 30, stream=part)
    E.submit_model(*ar, *tail, work_budget=1 << 28)
    (res,) = E.drain(256)
    E.close()
    assert torch.equal(res.traces, ref[0])


def test_misfit(F, part):
    """FP64 sums of n positive terms in other orders: n 2^-53 of the sum, with room."""
    rng = np.random.default_rng(7)
    a, b = (rng.standard_normal(200000).astype(np.float32) for _ in range(2))
    t, d = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    torch.cuda.synchronize()
    with torch.cuda.stream(part):
        J = F.fwi_misfit(t, d)
    part.synchronize()
    ref = 0.5 * ((a.astype(np.float64) - b) ** 2).sum()
    assert abs(J.item() - ref) <= 200000 * 2.0 ** -52 * ref
