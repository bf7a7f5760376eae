"""The Green tables themselves (G_o and dG_o/dr of every point, node and frequency), read from an
acquisition's workspace: each component against double-precision Bessel functions, wherever the value
comes from (radial polynomials, Bessel functions near a point), and which kernels made them."""
import ctypes

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


def ring(n, radius, phase=0.0):
    return np.asarray(I.circle(n, radius, (0.0, 0.0), phase), np.float32)


def tables(acq):
    """(G, dG/dr) as complex64 [nf][P][Ns] and the row exponents [nf][P], by the workspace's layout."""
    nf, N, P, ns, nr = acq.fg.nf, acq.fg.nx * acq.fg.nz, acq.ns + acq.nr, acq.ns, acq.nr
    up = lambda v, a: (v + a - 1) // a * a
    Ns, M, nchunk = up(N, 128), nf * ns * nr, (N + 255) // 256
    sizes = dict(status=4, spec=8 * nf, fr=8 * nf, pts=8 * P, Tg=8 * nf * P * Ns, Td=8 * nf * P * Ns, inc=8 * M,
                 part=8 * nchunk * M, data=8 * M, res=8 * M, fpart=48 * nf * N, mpart=8 * ((M + 31) // 32),
                 xc=8 * Ns, xmax=8, rsx=4 * nf * P)
    at, off = {}, 0
    for k, b in sizes.items():
        at[k] = off
        off = up(off + b, 256)
    assert off == acq.work.numel()
    w = acq.work.cpu().numpy()
    cut = lambda k, t: w[at[k]:at[k] + sizes[k]].view(t)
    return cut("Tg", np.complex64).reshape(nf, P, Ns), cut("Td", np.complex64).reshape(nf, P, Ns), \
        cut("rsx", np.int32).reshape(nf, P)


# grid (centred unless x0 is given), points, frequencies, the kernels expected
CASES = {
    "paper": dict(nx=121, nz=121, dx=5.0, src=ring(10, 490.0), rec=ring(100, 490.0, 0.5), f=0.25 * np.arange(1, 61), radial=1, near=0),
    "near and far nodes": dict(nx=60, nz=41, dx=5.0, src=ring(4, 195.0), rec=ring(20, 195.0, 0.5), f=0.4 * np.arange(1, 34), radial=1, near=1),
    "few frequencies": dict(nx=61, nz=33, dx=5.0, src=ring(3, 190.0), rec=ring(9, 190.0, 0.5), f=3.0 * np.arange(1, 6), radial=1, near=1),
    "few frequencies, more points": dict(nx=61, nz=33, dx=5.0, src=ring(6, 190.0), rec=ring(19, 200.0, 0.5), f=3.0 * np.arange(1, 6), radial=1, near=1),
    "the highest wavenumber of an interval": dict(nx=80, nz=60, dx=0.8, src=ring(5, 54.0), rec=ring(14, 55.0, 0.5), f=np.linspace(0.7, 19.89, 40), radial=1, near=1),
    "four decades of frequency": dict(nx=90, nz=64, dx=4.0, src=ring(5, 235.0), rec=ring(30, 240.0, 0.5), f=np.geomspace(0.002, 14.0, 37), radial=1, near=1),
    # the table of all frequencies does not fit the scratch: two frequency blocks
    "frequency blocks": dict(nx=9, nz=121, dx=5.0, src=ring(3, 360.0), rec=ring(7, 370.0, 0.5), f=0.25 * np.arange(1, 61), radial=2, near=0),
    # distances that are whole intervals (h = 1): both sides of an interval's edge and of the first one
    "interval edges": dict(nx=200, nz=40, dx=1.0, x0=0.0, z0=0.0, src=np.array([[-3.0, 0.0], [-40.0, 5.0]], np.float32),
                           rec=np.array([[203.0, 0.0], [-64.0, 3.0], [-63.0, 7.0], [230.0, 39.0], [-32.0, 1.0], [-31.0, 9.0]], np.float32),
                           f=0.5 * np.arange(1, 31), radial=1, near=1),
    # wavenumbers whose pairs FP32 does not hold
    "seven decades of frequency": dict(nx=60, nz=41, dx=5.0, src=ring(2, 195.0), rec=ring(8, 195.0, 0.5), f=np.geomspace(1e-6, 13.0, 33), radial=0, near=1),
    "every node near": dict(nx=40, nz=40, dx=5.0, src=ring(2, 160.0), rec=ring(6, 160.0, 0.5), f=0.01 * np.arange(1, 3), radial=0, near=1),
    "too small to pay": dict(nx=200, nz=3, dx=2.0, src=ring(1, 230.0), rec=ring(2, 230.0, 0.5), f=0.5 * np.arange(1, 33), radial=0, near=1),
}


@pytest.mark.parametrize("name", CASES)
def test_tables_are_rounded_bessel_values(FB, name):
    """FP64 values rounded to FP32 once: half an ulp (2^-24 of the component, also where it is near
    zero), and the FP64 evaluations' own error, here and in the reference: the argument's rounding, some
    units of 2^-52 of it, moves a component by that much of the amplitude (arguments up to 60, and
    polynomial sums kept to 2^-47), within 2^-43 of the amplitude."""
    from scipy.special import j0, j1, y0, y1

    c = CASES[name]
    x0, z0 = c.get("x0", -(c["nx"] - 1) / 2.0 * c["dx"]), c.get("z0", -(c["nz"] - 1) / 2.0 * c["dx"])
    L, buf = FB.lib(), ctypes.create_string_buffer(1 << 16)
    L.fwi_profile_report(buf, len(buf))
    L.fwi_profile(1)
    nf = len(c["f"])
    acq = FB.Acquisition(FB.make_fgrid(c["nx"], c["nz"], nf, c["dx"], x0, z0), c["f"], np.ones(nf, np.complex64), c["src"], c["rec"])
    torch.cuda.synchronize()
    L.fwi_profile(0)
    L.fwi_profile_report(buf, len(buf))
    used = {f[0].split("::")[-1]: int(f[1]) for f in map(str.split, buf.value.decode().splitlines())}
    assert (used.get("k_fb_green_radial", 0), used.get("k_fb_green", 0)) == (c["radial"], c["near"]), used
    G, D, rsx = tables(acq)
    N, P = c["nx"] * c["nz"], acq.ns + acq.nr
    assert not G[..., N:].any() and not D[..., N:].any()
    mx = np.max([np.abs(t.view(np.float32)).max(-1) for t in (G, D)], 0).astype(np.float64)
    assert (rsx == np.clip(13 - np.floor(np.log2(mx)), -126, 126)).all()
    pts = np.concatenate([acq.src, acq.rec]).astype(np.float64)
    n = np.arange(N) if nf * P * N <= 3000000 else np.sort(np.random.default_rng(5).choice(N, 3000000 // (nf * P), replace=False))
    r = np.hypot(x0 + (n % c["nx"]) * c["dx"] - pts[:, :1], z0 + (n // c["nx"]) * c["dx"] - pts[:, 1:])
    k = (2.0 * np.pi * np.asarray(c["f"], np.float64) / 2000.0)[:, None, None]
    x = k * r
    for got, scale, re, im in ((G[..., n], 500.0 + 0 * k, -y0(x), j0(x)), (D[..., n], 500.0 * k, y1(x), -j1(x))):
        amp = np.hypot(re, im)
        for g, ref in ((got.real, re), (got.imag, im)):
            excess = np.abs(g.astype(np.float64) / scale - ref) - 2.0 ** -24 * np.abs(ref)
            assert (excess <= 2.0 ** -43 * amp).all(), float((excess / amp).max())
