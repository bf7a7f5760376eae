"""On-chip launches that are refused (a stream that cannot hold them; here a bound on their blocks gives
the same refusal): the steps stream, and the results are the same bits.  Bounds of 0 and of one less
than a launch takes; a bound that lets forward launches pass and refuses the adjoint's, and the other
way round."""
import pytest

from paper_1804_01184_gb300 import inputs as I
from tests._common import gpu_grid
from tests.test_gpu_resident import kernels

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_01184_gb300 import build, fwi
    build.build()
    return fwi


def calls(F, w, every=0):
    g = gpu_grid(w)
    ar, tail = (g, w.pz, w.xi_a, w.xi_b), (w.src_xy, w.wavelet, w.rec_xy)
    d = [I.random_like(w.xi_a.shape, s, 0.05) for s in (1, 2)]
    data = I.random_like((w.ns, w.nr, w.nt), 3, 1.0)
    return {"model": lambda: (F.fwi_model(*ar, *tail),), "born": lambda: (F.fwi_born(*ar, *d, *tail),),
            "adjoint": lambda: (F.fwi_adjoint(*ar, *tail, data),), "gradient": lambda: F.fwi_gradient(*ar, *tail, data)}


@pytest.mark.parametrize("blocks", [0, 1, 5, 20, 40, 60, 80, 120])
@pytest.mark.parametrize("op,every", [("model", 0), ("born", 0), ("adjoint", 0), ("gradient", 0), ("gradient", 23)])
def test_single_calls(F, op, every, blocks):
    w = I.small_case(seed=31, nx=140, nz=120, nt=70, order=8, sponge=9, ns=5, nr=9)
    call = calls(F, w)[op]
    F.fwi_set_checkpoint(every)
    try:
        ref = call()
        F.fwi_set_chip_blocks(blocks)
        try:
            got, used = kernels(F, call)
        finally:
            F.fwi_set_chip_blocks(-1)
    finally:
        F.fwi_set_checkpoint(0)
    if blocks == 0:
        assert not any("k_res_" in k for k in used), used
        assert any("_warp<4," in k for k in used), used
    assert all(torch.equal(x, y) for x, y in zip(got, ref))


@pytest.mark.parametrize("blocks", [0, 40])
def test_engine(F, blocks):
    from paper_1804_01184_gb300 import engine
    w = I.small_case(seed=32, nx=140, nz=120, nt=70, order=8, sponge=9, ns=3, nr=9)
    g = gpu_grid(w)
    ar, tail = (g, w.pz, w.xi_a, w.xi_b), (w.src_xy, w.wavelet, w.rec_xy)
    data = I.random_like((w.ns, w.nr, w.nt), 3, 1.0)
    c = calls(F, w)
    ref = (*c["model"](), *c["gradient"]())
    F.fwi_set_chip_blocks(blocks)
    try:
        E = engine.Engine(1 << 30)
        t = [E.submit_model(*ar, *tail, work_budget=1 << 28), E.submit_gradient(*ar, *tail, data, work_budget=1 << 28)]
        out, used = kernels(F, lambda: {r.ticket: r for r in E.drain(256)})
        E.close()
    finally:
        F.fwi_set_chip_blocks(-1)
    assert not any("k_res_" in k for k in used), used
    got = (out[t[0]].traces, out[t[1]].misfit, out[t[1]].grads)
    assert all(torch.equal(x, y) for x, y in zip(got, ref))


def test_engine_follows_the_bound_between_calls(F):
    """The bound holds for the calls that follow it, also in an engine that has stepped on chip before."""
    from paper_1804_01184_gb300 import engine
    w = I.small_case(seed=33, nx=140, nz=120, nt=70, order=8, sponge=9, ns=3, nr=9)
    g = gpu_grid(w)
    ar, tail = (g, w.pz, w.xi_a, w.xi_b), (w.src_xy, w.wavelet, w.rec_xy)
    E = engine.Engine(1 << 30)
    out = []
    try:
        for blocks, on in ((-1, True), (0, False), (60, False), (-1, True)):
            F.fwi_set_chip_blocks(blocks)
            E.submit_model(*ar, *tail, work_budget=1 << 28)
            (res,), used = kernels(F, lambda: E.drain(256))
            assert any("k_res_" in k for k in used) == on, used
            out.append(res.traces)
    finally:
        F.fwi_set_chip_blocks(-1)
        E.close()
    assert all(torch.equal(x, out[0]) for x in out[1:])
