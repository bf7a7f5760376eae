"""Green tables of the frequency-domain Born path: built through radial polynomials where they
pay, by Bessel functions near a point and where they do not."""
import numpy as np
import pytest

from paper_1804_01184_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def FB():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_01184_gb300 import build, fborn
    build.build()
    return fborn


@pytest.mark.parametrize("nx,nz,ns,nr,nf,df,dx,ring", [
    (121, 121, 10, 100, 60, 0.25, 5.0, 490.0),       # the paper's acquisition: every node tabulated
    (60, 41, 4, 20, 33, 0.4, 5.0, 195.0),            # near and tabulated nodes, a ragged frequency block
    (61, 33, 3, 9, 5, 3.0, 5.0, 190.0),              # few frequencies
    (40, 40, 2, 6, 2, 0.01, 5.0, 160.0),             # every node near: no table
    (200, 3, 1, 2, 32, 0.5, 2.0, 230.0)])
def test_green_tables_against_bessel(FB, nx, nz, ns, nr, nf, df, dx, ring):
    """Data of a single-node scatterer, which is one node's table values: those of sampled nodes
    against the oracle's Hankel functions.  Values are rounded to FP32 once (2^-24); a datum is
    three products and sums of such values with FP32 splits of 22 bits: bound 2e-6."""
    from scipy.special import hankel1
    half = [(nx - 1) / 2.0 * dx, (nz - 1) / 2.0 * dx]
    freqs = df * np.arange(1, nf + 1)
    src, rec = I.circle(ns, ring, (0.0, 0.0)), I.circle(nr, ring, (0.0, 0.0), 0.5)
    spec = np.ones(nf, np.complex64)
    acq = FB.Acquisition(FB.make_fgrid(nx, nz, nf, dx, -half[0], -half[1]), freqs, spec, src, rec)
    rng = np.random.default_rng(nx)
    for _ in range(6):
        ix, iz = int(rng.integers(nx)), int(rng.integers(nz))
        xa, xb = np.zeros((nz, nx), np.float32), np.zeros((nz, nx), np.float32)
        xa[iz, ix] = 0.5                              # a contrast in 1/K alone
        got = acq.model(4, xa, xb, scheme=FB.LINEAR, incident=False).cpu().numpy().astype(np.complex128)
        X = np.array([ix * dx - half[0], iz * dx - half[1]])
        k = 2 * np.pi * freqs / 2000.0
        G = [500j * hankel1(0, k[:, None] * np.hypot(*(np.asarray(p, np.float64) - X).T)[None, :]) for p in (src, rec)]
        w2 = (2 * np.pi * freqs) ** 2 / (2000.0 * 2000.0 ** 2) * dx * dx * 0.5
        ref = w2[:, None, None] * G[0][:, :, None] * G[1][:, None, :]
        assert np.abs(got - ref).max() <= 2e-6 * np.abs(ref).max()
        assert np.linalg.norm(got - ref) <= 2e-6 * np.linalg.norm(ref)
