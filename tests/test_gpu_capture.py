"""Whole operations under stream capture, with the time steps on chip (cooperative launches) and
streaming (launches that may begin before the previous one ends): a replayed graph gives the
call's own results, bitwise."""
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
    return fwi


@pytest.mark.parametrize("op", ["born", "gradient"])
@pytest.mark.parametrize("tz", [0, 24])     # a fixed strip height asks for the streaming kernels
def test_replay_is_the_call(F, op, tz):
    w = I.small_case(seed=11, nx=130, nz=75, nt=45, order=8, sponge=9, ns=3, nr=12)
    g = gpu_grid(w)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    model, acq = (d(w.xi_a), d(w.xi_b)), (d(w.src_xy), d(w.wavelet), d(w.rec_xy))
    F.fwi_set_tile(tz, 0)
    try:
        if op == "born":
            work, out = F.workspace(g, w.ns, w.nr, F.OP_BORN), torch.zeros((w.ns, w.nr, w.nt), device="cuda")
            pert = (d(0.5 * w.xi_b), d(-0.5 * w.xi_a))
            call = lambda: F.fwi_born(g, w.pz, *model, *pert, *acq, dtraces=out, work=work, check=False)
        else:
            work = F.workspace(g, w.ns, w.nr, F.OP_GRADIENT)
            data, J = d(I.random_like((w.ns, w.nr, w.nt), 5, 1.0)), torch.zeros((), dtype=torch.float64, device="cuda")
            out = torch.zeros((5, 2, w.nz, w.nx), dtype=torch.float64, device="cuda")
            call = lambda: F.fwi_gradient(g, w.pz, *model, *acq, data, misfit=J, grads=out, work=work, check=False)
        call()
        torch.cuda.synchronize()
        ref = out.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            call()
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
    finally:
        F.fwi_set_tile(0, 0)
    assert ref.abs().max().item() > 0
    assert torch.equal(out, ref)
