"""When a single call steps on chip: the rule counts the launches of a call's shots, whose cost short
runs (accumulation chunks or checkpoints of a step) do not spread over many steps, and what the
streaming steps of the same shots take."""
import numpy as np
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


def chip(used):
    return {k.split("::")[-1].split("<")[0] for k in used if "k_res_" in k}


def gradient(F, order, ns):
    w = I.small_case(seed=51, nx=185, nz=185, nt=48, order=order, sponge=8, ns=ns, nr=9)
    data = I.random_like((w.ns, w.nr, w.nt), 3, 1.0)
    return lambda: F.fwi_gradient(gpu_grid(w), w.pz, w.xi_a, w.xi_b, w.src_xy, w.wavelet, w.rec_xy, data)


@pytest.mark.parametrize("order", [4, 8])
def test_runs_of_one_step_over_many_launches_stream(F, order):
    call = gradient(F, order, 40)            # several launches of shots
    _, used = kernels(F, call)
    assert chip(used) == {"k_res_fwd", "k_res_adj"}, used
    F.fwi_set_accumulation(1)
    try:
        got, used = kernels(F, call)
        assert chip(used) == {"k_res_fwd"}, used
        F.fwi_set_chip_blocks(0)
        ref = call()
    finally:
        F.fwi_set_chip_blocks(-1)
        F.fwi_set_accumulation(0)
    assert all(torch.equal(x, y) for x, y in zip(got, ref))
    F.fwi_set_checkpoint(1)
    try:
        got, used = kernels(F, call)
        assert not chip(used), used
        F.fwi_set_chip_blocks(0)
        ref = call()
    finally:
        F.fwi_set_chip_blocks(-1)
        F.fwi_set_checkpoint(0)
    assert all(torch.equal(x, y) for x, y in zip(got, ref))


@pytest.mark.parametrize("order", [4, 8])
def test_runs_of_one_step_in_one_launch_stay(F, order):
    call = gradient(F, order, 2)
    F.fwi_set_accumulation(1)
    try:
        _, used = kernels(F, call)
    finally:
        F.fwi_set_accumulation(0)
    assert chip(used) == {"k_res_fwd", "k_res_adj"}, used


@pytest.mark.parametrize("order,n,ns,nt,on", [(8, 681, 1, 64, True), (8, 681, 16, 64, False), (8, 720, 16, 32, False),
                                              (4, 800, 16, 32, False), (8, 320, 16, 64, True), (4, 512, 8, 64, True)])
def test_forward_calls(F, order, n, ns, nt, on):
    """Calls that streaming made 15 to 18 % faster than on chip, and calls far on the other side."""
    w = I.small_case(seed=52, nx=64, nz=64, nt=nt, order=order, sponge=0, ns=ns, nr=4)
    w.nx = w.nz = n
    w.xi_a, w.xi_b = (np.zeros((n, n), np.float32) for _ in range(2))
    _, used = kernels(F, lambda: F.fwi_model(gpu_grid(w), w.pz, w.xi_a, w.xi_b, w.src_xy, w.wavelet, w.rec_xy))
    assert chip(used) == ({"k_res_fwd"} if on else set()), used
