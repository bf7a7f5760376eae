"""Expired waits between the blocks of an on-chip launch: with a limit of no polls every wait expires at
its first look, whatever the neighbour has sent.  The launch ends, the call (or the engine) reports
FWI_ETIMEOUT, and the next call is sound."""
import threading

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


@pytest.fixture
def no_polls(F):
    F.fwi_set_wait_limit(0)
    yield
    F.fwi_set_wait_limit(-1)


def workload(order):
    return I.small_case(seed=21, nx=180, nz=130, nt=60, order=order, sponge=12, ns=2, nr=9)


def calls(F, w):
    g = gpu_grid(w)
    ar, tail = (g, w.pz, w.xi_a, w.xi_b), (w.src_xy, w.wavelet, w.rec_xy)
    d = [I.random_like(w.xi_a.shape, s, 0.05) for s in (1, 2)]
    data = I.random_like((w.ns, w.nr, w.nt), 3, 1.0)
    return {"model": ("k_res_fwd", lambda: (F.fwi_model(*ar, *tail),)),
            "born": ("k_res_born", lambda: (F.fwi_born(*ar, *d, *tail),)),
            "gradient": ("k_res_adj", lambda: F.fwi_gradient(*ar, *tail, data))}


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("op", ["model", "born", "gradient"])
def test_single_call_reports_and_the_next_is_sound(F, op, order):
    name, call = calls(F, workload(order))[op]
    ref = call()
    F.fwi_set_wait_limit(0)
    try:
        def attempt():
            with pytest.raises(F.FwiError) as e:
                call()
            return e.value

        err, used = kernels(F, attempt)
    finally:
        F.fwi_set_wait_limit(-1)
    assert err.code == -4, err
    assert any(name in k for k in used), used
    assert all(torch.equal(x, y) for x, y in zip(call(), ref))


def test_a_shot_of_one_block_does_not_wait(F, no_polls):
    w = I.small_case(seed=22, nx=20, nz=9, nt=40, order=8, sponge=2, ns=2, nr=5)   # too small to cut
    got, used = kernels(F, lambda: F.fwi_model(gpu_grid(w), w.pz, w.xi_a, w.xi_b, w.src_xy, w.wavelet, w.rec_xy))
    assert any("k_res_fwd" in k for k in used), used
    assert torch.isfinite(got).all() and got.abs().max().item() > 0


def test_the_limit_is_the_calling_threads(F, no_polls):
    _, call = calls(F, workload(8))["model"]
    out, errors = [], []

    def other():
        try:
            out.append(call())
        except Exception as e:   # noqa: BLE001 -- shown by the assertion below
            errors.append(e)

    t = threading.Thread(target=other)
    t.start()
    t.join()
    assert out and not errors


@pytest.mark.parametrize("op", ["model", "born", "gradient"])
def test_engine_reports(F, op):
    from paper_1804_01184_gb300 import engine
    w = workload(8)
    g = gpu_grid(w)
    ar, tail = (g, w.pz, w.xi_a, w.xi_b), (w.src_xy, w.wavelet, w.rec_xy)
    d = [I.random_like(w.xi_a.shape, s, 0.05) for s in (1, 2)]
    data = I.random_like((w.ns, w.nr, w.nt), 3, 1.0)

    def submit(E):
        if op == "model":
            return E.submit_model(*ar, *tail, work_budget=1 << 28)
        if op == "born":
            return E.submit_born(*ar, *d, *tail, work_budget=1 << 28)
        return E.submit_gradient(*ar, *tail, data, work_budget=1 << 28)

    F.fwi_set_wait_limit(0)
    try:
        E = engine.Engine(1 << 30)
        submit(E)
        with pytest.raises(F.FwiError) as e:
            E.drain(256)
        assert e.value.code == -4, e.value
        with pytest.raises(F.FwiError):     # and no ticket comes back afterwards
            E.run(8)
        E.close()
    finally:
        F.fwi_set_wait_limit(-1)
    E = engine.Engine(1 << 30)              # a new engine is sound, also with the old one's status word
    submit(E)
    (res,) = E.drain(256)
    E.close()
    one = calls(F, w)[op][1]()
    got = (res.traces,) if res.traces is not None else (res.misfit, res.grads)
    assert all(torch.equal(x, y) for x, y in zip(got, one))
