"""fwi_misfit's cluster reduction: sizes on either side of a block's share and of the unrolled
loop, aligned or not, weighted or not, against numpy in 64 bits (FP64 sums of n positive terms in
other orders: n 2^-53, with room)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,nt", [(0, 1), (1, 1), (511, 7), (2048, 16), (2049, 3), (8192, 64), (40000, 125), (1400000, 1400)])
@pytest.mark.parametrize("off", [0, 1])
def test_misfit(n, nt, off):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_01184_gb300 import fwi as F
    rng = np.random.default_rng(n + off)
    a, b = ((rng.standard_normal(n + off) * 10.0 ** rng.uniform(-30, 15)).astype(np.float32) for _ in range(2))
    t, d = torch.from_numpy(a).cuda()[off:], torch.from_numpy(b).cuda()[off:]
    r2 = (a[off:].astype(np.float64) - b[off:]) ** 2
    J = F.fwi_misfit(t, d).item()
    assert abs(J - 0.5 * r2.sum()) <= max(n, 8) * 2.0 ** -52 * 0.5 * r2.sum()
    if n and n % nt == 0:
        w = rng.random(n // nt).astype(np.float32)
        Jw, ref = F.fwi_misfit(t, d, weights=w, nt=nt).item(), 0.5 * (np.repeat(w.astype(np.float64), nt) * r2).sum()
        assert abs(Jw - ref) <= max(n, 8) * 2.0 ** -52 * ref
    assert F.fwi_misfit(t, d).item() == J
