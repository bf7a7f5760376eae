"""The work a user of this framework has it do, as cases for timing.

Each case is one call (or one step of a user's loop) through the public entry points: forward
shots, Born modelling, misfit gradients, differentiation through autograd, line searches and
mixed request batches on the engine, and the frequency-domain Born path of Schemes I/II.
``prepare`` makes what the program holds before the call, ``run`` is one pass, ``exact`` the same
outputs in 64 bits from plain torch.  Outputs keep the types the entry points return.
"""
import math

import numpy as np
import torch

DEV = "cuda"


# ----------------------------------------------------------------------------- cases

def _fd(name, op, nx, nz, nt, ns, nr, order=8, sponge=40, dx=5.0, dt=5e-4, f_peak=15.0, pz=0, sigma=20.0, **more):
    return dict(name=name, op=op, nx=nx, nz=nz, nt=nt, ns=ns, nr=nr, order=order, sponge=sponge, dx=dx, dt=dt,
                f_peak=f_peak, pz=pz, sigma=sigma, **more)


def listed():
    return [
        # The smallest calls: a couple of shots on a small heterogeneous model (the sizes of the
        # smoke check and of the parity tests); launch latency is everything.
        _fd("model-small", "model", 70, 54, 200, 2, 6, sponge=8, f_peak=25.0),
        # The point-scatterer workload, whole record: 4th order, K-rho contrasts.
        _fd("model-point", "model", 201, 201, 800, 8, 64, order=4, pz=3, sigma=10.0),
        # One shot on the large grid: interactive modelling, the plain per-shot path.
        _fd("model-shot", "model", 601, 601, 500, 1, 256),
        # The benchmark's acquisition (64 shots, 256 receivers), a stretch of its record.
        _fd("model-gaussian", "model", 601, 601, 200, 64, 256),
        # Born modelling on the same acquisition.
        _fd("born-gaussian", "born", 601, 601, 150, 64, 256),
        # Misfit and gradient on the same acquisition, the whole history kept; all five
        # parameterizations, as fwi_gradient returns them.
        _fd("gradient-gaussian", "gradient", 601, 601, 200, 64, 256, budget_gb=32),
        # The gradient of one descent iteration with unknown fields on the paper's own acquisition
        # (10 sources, 100 receivers, 5 Hz), whole record, through Inversion.
        _fd("gradient-paper", "inversion", 121, 121, 1400, 10, 100, dx=10.0, dt=1e-3, f_peak=5.0, sigma=50.0),
        # That iteration's line search: 8 trial models as engine jobs, their misfits reduced.
        _fd("linesearch-paper", "linesearch", 121, 121, 1400, 10, 100, dx=10.0, dt=1e-3, f_peak=5.0, sigma=50.0,
            trials=8),
        # Differentiation on the fine smooth model: forward, torch misfit, backward with
        # checkpointing (the budget stands in for a record whose history does not fit).
        _fd("autograd-smooth", "autograd", 1201, 1201, 160, 16, 256, dx=2.5, dt=2.5e-4, sigma=25.0, budget_gb=6),
        # A batch of light mixed requests (forward, Born, gradient) running together in the engine.
        dict(name="engine-light", op="engine", mix=11, jobs=12, side_lo=128, side_hi=256, nt_lo=500, nt_hi=1000,
             ns_hi=4, nr=64, order=8, sponge=40, dx=5.0, dt=5e-4, f_peak=15.0, pz=0, sigma=20.0),
        # One descent iteration's gradient in the frequency domain (Scheme I), the paper's acquisition:
        # 60 frequencies, 10 sources, 100 receivers, 121 x 121 nodes.
        dict(name="fborn-gradient", op="fgradient", nx=121, nz=121, nf=60, ns=10, nr=100, dx=5.0, df=0.25, f_peak=5.0,
             pz=0, scheme=1),
        # A new acquisition (its Green tables) and its Born data under the exact map (Scheme II).
        dict(name="fborn-survey", op="fsurvey", nx=121, nz=121, nf=60, ns=10, nr=100, dx=5.0, df=0.25, f_peak=5.0,
             pz=0, scheme=2),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["model", "model", "born", "gradient", "inversion", "linesearch", "autograd", "engine", "fgradient",
                     "fsurvey"])
    if op in ("fgradient", "fsurvey"):
        while True:
            nx, nz = _logint(rng, 9, 121), _logint(rng, 9, 121)
            nf, ns, nr = _logint(rng, 2, 60), _logint(rng, 1, 32), _logint(rng, 3, 200)
            if nf * nx * nz * (ns + nr) <= 60 * 121 * 121 * 110 and nf * nx * nz * ns * nr <= 60 * 121 * 121 * 1000:
                break
        return dict(op=op, nx=nx, nz=nz, nf=nf, ns=ns, nr=nr, dx=5.0, df=15.0 / nf, f_peak=5.0, pz=rng.randrange(5),
                    scheme=rng.choice([1, 2]))
    if op == "engine":
        lo = _logint(rng, 32, 160)
        return dict(op=op, mix=rng.randrange(1 << 20), jobs=rng.randint(3, 12), side_lo=lo, side_hi=int(lo * 1.6),
                    nt_lo=200, nt_hi=800, ns_hi=rng.randint(1, 4), nr=rng.randint(5, 64), order=rng.choice([4, 8]),
                    sponge=rng.choice([8, 20, 40]), dx=5.0, dt=5e-4, f_peak=15.0, pz=0, sigma=20.0)
    cost = {"model": 1, "born": 2, "gradient": 3, "inversion": 3, "linesearch": 8, "autograd": 4}[op]
    big = {"inversion": 200, "linesearch": 200}.get(op, 700)
    while True:
        nx = _logint(rng, 24, big)
        nz = max(20, int(nx * rng.uniform(0.6, 1.5)))
        ns, nt = _logint(rng, 1, 64), _logint(rng, 60, 1400)
        sponge = rng.choice([0, 8, 20, 40])
        if cost * (nx + 2 * sponge) * (nz + 2 * sponge) * ns * nt <= 5e9:
            break
    more = {"trials": 8} if op == "linesearch" else {}
    if op in ("gradient", "autograd"):
        more["budget_gb"] = rng.choice([1, 4, 24])
    return dict(op=op, nx=nx, nz=nz, nt=nt, ns=ns, nr=_logint(rng, 3, 256), order=rng.choice([4, 8, 8]), sponge=sponge,
                dx=5.0, dt=5e-4, f_peak=15.0, pz=0 if op in ("inversion", "linesearch") else rng.randrange(5),
                sigma=20.0, **more)


# ---------------------------------------------------------------------------- inputs

def _ricker(t, f):
    a = (math.pi * f * (t - 1.0 / f)) ** 2
    return (1.0 - 2.0 * a) * torch.exp(-a)


def _ring(n, radius, centre, phase):
    th = 2.0 * math.pi * (np.arange(n) + phase) / n
    return np.stack([centre[0] + radius * np.cos(th), centre[1] + radius * np.sin(th)], 1).astype(np.float32)


def _field(gen, nx, nz, dx, sigma, amp):
    """A smooth random background (a few percent) and one Gaussian scatterer of contrast amp."""
    k = torch.randn((1, 1, 9, 9), generator=gen)
    bg = torch.nn.functional.interpolate(k, size=(nz, nx), mode="bicubic", align_corners=True)[0, 0]
    bg = 0.05 * bg / bg.abs().max()
    cx, cz = [(0.35 + 0.3 * float(v)) * (m - 1) * dx for v, m in zip(torch.rand(2, generator=gen), (nx, nz))]
    x, z = torch.arange(nx) * dx - cx, torch.arange(nz) * dx - cz
    g = torch.exp(-(x[None, :] ** 2 + z[:, None] ** 2) / (2.0 * sigma * sigma))
    return (bg + amp * g).float()


def _fd_inputs(c, seed):
    """Contrasts of the current model, acquisition, wavelet (all float32, on the GPU)."""
    gen = torch.Generator().manual_seed(seed)
    nx, nz, dx = c["nx"], c["nz"], c["dx"]
    amp = (torch.rand(4, generator=gen) - 0.5).tolist()          # contrasts in [-0.5, 0.5]
    centre = ((nx - 1) * dx / 2.0, (nz - 1) * dx / 2.0)
    radius = 0.4 * (min(nx, nz) - 1) * dx
    ph = torch.rand(2, generator=gen).tolist()
    t = (torch.arange(c["nt"], dtype=torch.float64) + 0.5) * c["dt"]
    u = dict(a=_field(gen, nx, nz, dx, c["sigma"], 0.8 * amp[0]), b=_field(gen, nx, nz, dx, c["sigma"], 0.8 * amp[1]),
             src=torch.from_numpy(_ring(c["ns"], radius, centre, ph[0])),
             rec=torch.from_numpy(_ring(c["nr"], radius, centre, ph[1])), wav=_ricker(t, c["f_peak"]).float())
    if c["op"] in ("born", "mixed-born"):
        u["da"] = _field(gen, nx, nz, dx, c["sigma"], 0.2 * amp[2])
        u["db"] = _field(gen, nx, nz, dx, c["sigma"], 0.2 * amp[3])
    u = {k: v.to(DEV) for k, v in u.items()}
    if c["op"] not in ("model", "born", "mixed-born"):
        # observed traces: the direct arrival of every source-receiver pair and recording noise
        w = 2.0 * math.pi * c["f_peak"]
        r = torch.cdist(u["src"].double(), u["rec"].double()).clamp_min(dx)
        a = 0.25 * w * 2000.0 * torch.sqrt(2.0 / (math.pi * (w / 2000.0) * r))
        d = a[..., None] * _ricker(t.to(DEV) - (r / 2000.0)[..., None], c["f_peak"])
        g2 = torch.Generator(DEV).manual_seed(seed + 1)
        u["data"] = (d + 0.05 * a.mean() * torch.randn(d.shape, generator=g2, device=DEV)).float()
    if c["op"] == "linesearch":   # trial models along a descent direction
        s = _field(gen, nx, nz, dx, c["sigma"], 0.5).to(DEV)
        u["trials"] = [(u["a"] + 0.01 * 2.0 ** (k - 3) * s, u["b"] - 0.005 * 2.0 ** (k - 3) * s)
                       for k in range(c["trials"])]
    return u


def _mix(c):
    """The jobs of an engine case (kind and sizes fixed by the case, not by the seed)."""
    rng = np.random.default_rng(c["mix"])
    out = []
    for k in range(c["jobs"]):
        n = int(rng.integers(c["side_lo"], c["side_hi"] + 1))
        out.append(dict(c, op=("model", "mixed-born", "gradient")[k % 3], nx=n, nz=n,
                        nt=int(rng.integers(c["nt_lo"], c["nt_hi"] + 1)), ns=int(rng.integers(1, c["ns_hi"] + 1))))
    return out


def _freq_inputs(c, seed):
    gen = torch.Generator().manual_seed(seed)
    nx, nz, dx = c["nx"], c["nz"], c["dx"]
    amp = (0.4 * (torch.rand(2, generator=gen) - 0.5)).tolist()
    a, b = (_field(gen, nx, nz, dx, 0.08 * max(nx, nz) * dx, v).to(DEV) for v in amp)
    half = 0.5 * dx * math.hypot(nx - 1, nz - 1)
    ph = torch.rand(2, generator=gen).tolist()
    src, rec = _ring(c["ns"], 1.16 * half + dx, (0.0, 0.0), ph[0]), _ring(c["nr"], 1.2 * half + 2 * dx, (0.0, 0.0), ph[1])
    f = c["df"] * np.arange(1, c["nf"] + 1, dtype=np.float64)
    S = (2.0 / math.sqrt(math.pi) * f * f / c["f_peak"] ** 3 * np.exp(-(f / c["f_peak"]) ** 2)
         * np.exp(2j * math.pi * f / c["f_peak"])).astype(np.complex64)
    u = dict(a=a, b=b, src=src, rec=rec, freqs=f, spectrum=S, x0=-(nx - 1) / 2.0 * dx, z0=-(nz - 1) / 2.0 * dx)
    if c["op"] == "fgradient":    # observed data: the direct field with 20 % of scattered field
        G = _green(torch.from_numpy(f).to(DEV)[:, None, None],
                   torch.cdist(torch.from_numpy(src).double(), torch.from_numpy(rec).double()).to(DEV))[0]
        g2 = torch.Generator(DEV).manual_seed(seed + 1)
        n = torch.randn(G.shape + (2,), generator=g2, device=DEV, dtype=torch.float64)
        q = torch.from_numpy(S).to(DEV)[:, None, None] * G * (1.0 + 0.2 * torch.view_as_complex(n))
        u["data"] = q.to(torch.complex64)
    return u


# -------------------------------------------------------------------- prepare and run

def _grid(c):
    from paper_1804_01184_gb300 import fwi
    return fwi.make_grid(nx=c["nx"], nz=c["nz"], dx=c["dx"], dt=c["dt"], nt=c["nt"], order=c["order"],
                         sponge=c["sponge"])


def prepare(case, seed):
    from paper_1804_01184_gb300 import engine, fborn, fwi, inputs, invert
    c, op = case, case["op"]
    s = dict(case=c, op=op)
    if op in ("fgradient", "fsurvey"):
        u = s["u"] = _freq_inputs(c, seed)
        s["grid"] = fborn.make_fgrid(c["nx"], c["nz"], c["nf"], c["dx"], u["x0"], u["z0"])
        if op == "fgradient":
            acq = fborn.Acquisition(s["grid"], u["freqs"], u["spectrum"], u["src"], u["rec"])
            s["inv"] = invert.BornInversion(acq, c["pz"], u["data"], c["scheme"])
        return s
    if op == "engine":
        s["jobs"] = [(j, _fd_inputs(j, seed + 17 * k)) for k, j in enumerate(_mix(c))]
        s["engine"] = engine.Engine(6 << 30)
        return s
    u = s["u"] = _fd_inputs(c, seed)
    g = s["grid"] = _grid(c)
    ns, nr = c["ns"], c["nr"]
    if op in ("model", "born"):
        s["work"] = fwi.workspace(g, ns, nr, fwi.OP_MODEL if op == "model" else fwi.OP_BORN)
        s["out"] = torch.empty((ns, nr, c["nt"]), device=DEV)
    elif op == "gradient":
        s["work"] = fwi.workspace(g, ns, nr, fwi.OP_GRADIENT, int(c["budget_gb"] * (1 << 30)))
    elif op in ("inversion", "linesearch"):
        w = inputs.Workload("paper", c["nx"], c["nz"], c["dx"], c["dt"], c["nt"], c["order"], c["sponge"], 2000.0,
                            2000.0, c["pz"], u["a"].cpu().numpy(), u["b"].cpu().numpy(), u["src"].cpu().numpy(),
                            u["rec"].cpu().numpy(), u["wav"].cpu().numpy())
        s["inv"] = invert.Inversion(w, c["pz"], u["data"], arena_bytes=4 << 30)
    return s


def run(state):
    from paper_1804_01184_gb300 import autograd, fborn, fwi
    op, c = state["op"], state["case"]
    u, g = state.get("u"), state.get("grid")
    if op == "model":
        return fwi.fwi_model(g, c["pz"], u["a"], u["b"], u["src"], u["wav"], u["rec"], traces=state["out"],
                             work=state["work"], check=False)
    if op == "born":
        return fwi.fwi_born(g, c["pz"], u["a"], u["b"], u["da"], u["db"], u["src"], u["wav"], u["rec"],
                            dtraces=state["out"], work=state["work"], check=False)
    if op == "gradient":
        return fwi.fwi_gradient(g, c["pz"], u["a"], u["b"], u["src"], u["wav"], u["rec"], u["data"],
                                work=state["work"], check=False)
    if op == "inversion":
        return state["inv"].gradient((u["a"], u["b"]))
    if op == "linesearch":
        return state["inv"].misfits(u["trials"])
    if op == "autograd":
        a, b = u["a"].requires_grad_(True), u["b"].requires_grad_(True)
        tr = autograd.model(a, b, g, c["pz"], u["src"], u["wav"], u["rec"], budget_bytes=int(c["budget_gb"] * (1 << 30)))
        ga, gb = torch.autograd.grad(0.5 * (tr - u["data"]).square().sum(), (a, b))
        return tr.detach(), ga, gb
    if op == "engine":
        e, order = state["engine"], []
        for j, v in state["jobs"]:
            head = (_grid(j), j["pz"], v["a"], v["b"])
            tail = (v["src"], v["wav"], v["rec"])
            if j["op"] == "model":
                order.append(e.submit_model(*head, *tail, work_budget=1 << 28))
            elif j["op"] == "mixed-born":
                order.append(e.submit_born(*head, v["da"], v["db"], *tail, work_budget=1 << 28))
            else:
                order.append(e.submit_gradient(*head, *tail, v["data"], work_budget=1 << 28))
        got = {r.ticket: r for r in e.drain()}
        return [got[t].traces if got[t].traces is not None else (got[t].misfit, got[t].grads) for t in order]
    if op == "fgradient":
        return state["inv"].gradient((u["a"], u["b"]))
    acq = fborn.Acquisition(g, u["freqs"], u["spectrum"], u["src"], u["rec"])
    return acq.model(c["pz"], u["a"], u["b"], scheme=c["scheme"])


# --------------------------------------------------------------------------- the work

def _cells(c):
    return (c["nx"] + 2 * c["sponge"]) * (c["nz"] + 2 * c["sponge"])


def work(case):
    """Inputs and outputs once; the scheme's operations: a derivative of order 2M takes M
    subtractions and M multiply-adds, a step four of them and its updates."""
    c, op = case, case["op"]
    if op in ("fgradient", "fsurvey"):
        N, M, P = c["nx"] * c["nz"], c["nf"] * c["ns"] * c["nr"], c["nf"] * (c["ns"] + c["nr"])
        table = 16.0 * P * N                        # G_o and dG_o/dr of every point and node
        if op == "fsurvey":                         # write the tables, contract them once
            return dict(bytes=table + 8.0 * N + 8.0 * M, flops=24.0 * M * N + 60.0 * P * N)
        return dict(bytes=table + 16.0 * N + 16.0 * M, flops=2 * 24.0 * M * N)
    if op == "engine":
        w = [work(j) for j in _mix(c)]
        return dict(bytes=sum(x["bytes"] for x in w), flops=sum(x["flops"] for x in w))
    cells, traces = _cells(c), 4.0 * c["ns"] * c["nr"] * c["nt"]
    step = 4 * 3 * (c["order"] // 2) + 12
    per = {"model": 1, "born": 2, "mixed-born": 2, "gradient": 3, "inversion": 3, "autograd": 4, "linesearch": 1}[op]
    steps = float(cells) * c["ns"] * c["nt"] * c.get("trials", 1)
    fields = 4.0 * c["nx"] * c["nz"]
    io = {"model": 2 * fields + traces, "born": 4 * fields + traces, "mixed-born": 4 * fields + traces,
          "gradient": 22 * fields + traces, "inversion": 4 * fields + traces, "autograd": 4 * fields + 2 * traces,
          "linesearch": 2 * fields * c.get("trials", 1) + traces}[op]
    return dict(bytes=io, flops=per * step * steps)


# ------------------------------------------------------------------ the same in 64 bits

class _Scheme:
    """The staggered-grid scheme on [shots][Nz][Nx] float64 tensors (zero outside the grid)."""

    def __init__(self, c, u):
        self.c = c
        S, nx, nz, self.dt, self.dx = c["sponge"], c["nx"], c["nz"], c["dt"], c["dx"]
        self.S, self.Nx, self.Nz, self.M = S, nx + 2 * S, nz + 2 * S, c["order"] // 2
        self.coef = ([9 / 8, -1 / 24] if self.M == 2 else [1225 / 1024, -245 / 3072, 49 / 5120, -5 / 7168])
        self.vo = self.ro = 2000.0
        pad = lambda n: (torch.arange(n + 2 * S, device=DEV) - S).clamp(0, n - 1)
        self.ix, self.iz = pad(nx), pad(nz)
        self.K0, self.rho0 = self.maps(c["pz"], u["a"].double(), u["b"].double())
        self.K, self.rho = self.spread(self.K0), self.spread(self.rho0)
        self.bx, self.bz = 2.0 / (self.rho + self.right(self.rho)), 2.0 / (self.rho + self.down(self.rho))
        ax, axh, az, azh = (self.profile(n, h) for n in (nx, nz) for h in (0.0, 0.5))
        self.dp, self.dvx, self.dvz = az[:, None] * ax, az[:, None] * axh, azh[:, None] * ax
        self.wav = u["wav"].double().tolist()
        self.src, self.rec = self.footprint(u["src"]), self.footprint(u["rec"])

    def spread(self, f):
        return f[self.iz][:, self.ix]

    def right(self, f):
        return torch.cat([f[..., 1:], f[..., -1:]], -1)

    def down(self, f):
        return torch.cat([f[..., 1:, :], f[..., -1:, :]], -2)

    def maps(self, pz, a, b):
        A, B, vo, ro = 1 + a, 1 + b, self.vo, self.ro
        Ko = ro * vo * vo
        return {0: lambda: (Ko * B * A * A, ro * B), 1: lambda: (Ko * A * A / B, ro * B),
                2: lambda: (Ko * A * B, ro * B / A), 3: lambda: (Ko * A, ro * B), 4: lambda: (Ko / A, ro / B)}[pz]()

    def profile(self, n, half):
        S, v = self.S, torch.arange(n + 2 * self.S, device=DEV, dtype=torch.float64) + half
        if S == 0:
            return torch.ones_like(v)
        d = torch.maximum((S - v).clamp_min(0), (v - (S + n - 1)).clamp_min(0)) / S
        return torch.exp(-3.0 * self.vo * math.log(1e3) / (2.0 * S * self.dx) * d * d * self.dt)

    def footprint(self, xy):
        f = xy.double() / self.dx + self.S
        i = torch.minimum(f[:, 0].floor().long(), torch.tensor(self.Nx - 2, device=DEV))
        j = torch.minimum(f[:, 1].floor().long(), torch.tensor(self.Nz - 2, device=DEV))
        tx, tz = f[:, 0] - i, f[:, 1] - j
        at = torch.stack([j * self.Nx + i, j * self.Nx + i + 1, (j + 1) * self.Nx + i, (j + 1) * self.Nx + i + 1], 1)
        return at, torch.stack([(1 - tx) * (1 - tz), tx * (1 - tz), (1 - tx) * tz, tx * tz], 1)

    def diff(self, f, axis, plus):
        """dt D+ f (plus) or dt D- f along x (axis -1) or z (axis -2)."""
        M, n = self.M, f.shape[axis]
        w = torch.nn.functional.pad(f, (M, M, 0, 0) if axis == -1 else (0, 0, M, M))
        out = 0
        for k in range(1, M + 1):
            hi, lo = (M + k, M - k + 1) if plus else (M + k - 1, M - k)
            out = out + self.coef[k - 1] * self.dt / self.dx * (w.narrow(axis, hi, n) - w.narrow(axis, lo, n))
        return out

    def source(self, n, s0, s1):
        at, w = self.src
        return at[s0:s1], self.wav[n] * self.dt / self.dx ** 2 * w[s0:s1]

    def sample(self, p):
        at, w = self.rec
        return (p.flatten(1)[:, at] * w).sum(-1)

    def forward(self, s0, s1, keep=False):
        """Traces of shots s0 .. s1 and, with keep, p^0 .. p^nt."""
        z = lambda: torch.zeros((s1 - s0, self.Nz, self.Nx), device=DEV, dtype=torch.float64)
        p, vx, vz = z(), z(), z()
        tr = torch.empty((s1 - s0, self.rec[0].shape[0], self.c["nt"]), device=DEV, dtype=torch.float64)
        hist = [p] if keep else None
        for n in range(self.c["nt"]):
            vx = self.dvx * (vx - self.bx * self.diff(p, -1, True))
            vz = self.dvz * (vz - self.bz * self.diff(p, -2, True))
            p = self.dp * (p - self.K * (self.diff(vx, -1, False) + self.diff(vz, -2, False)))
            at, w = self.source(n, s0, s1)
            p.flatten(1).scatter_add_(1, at, w * self.K.flatten()[at])
            tr[:, :, n] = self.sample(p)
            if keep:
                hist.append(p)
        return tr, hist

    def born(self, s0, s1, u):
        c = self.c
        a, b = u["a"].double(), u["b"].double()
        _, (dK, dr) = torch.func.jvp(lambda x, y: self.maps(c["pz"], x, y), (a, b), (u["da"].double(), u["db"].double()))
        dK, dr = self.spread(dK), self.spread(dr)
        dbx, dbz = (-0.5 * q * q * (dr + far(dr)) for q, far in ((self.bx, self.right), (self.bz, self.down)))
        z = lambda: torch.zeros((s1 - s0, self.Nz, self.Nx), device=DEV, dtype=torch.float64)
        p, vx, vz, q, ux, uz = z(), z(), z(), z(), z(), z()
        tr = torch.empty((s1 - s0, self.rec[0].shape[0], c["nt"]), device=DEV, dtype=torch.float64)
        for n in range(c["nt"]):
            gx, gz = self.diff(p, -1, True), self.diff(p, -2, True)
            ux = self.dvx * (ux - self.bx * self.diff(q, -1, True) - dbx * gx)
            uz = self.dvz * (uz - self.bz * self.diff(q, -2, True) - dbz * gz)
            vx, vz = self.dvx * (vx - self.bx * gx), self.dvz * (vz - self.bz * gz)
            dv = self.diff(vx, -1, False) + self.diff(vz, -2, False)
            q = self.dp * (q - self.K * (self.diff(ux, -1, False) + self.diff(uz, -2, False)) - dK * dv)
            p = self.dp * (p - self.K * dv)
            at, w = self.source(n, s0, s1)
            p.flatten(1).scatter_add_(1, at, w * self.K.flatten()[at])
            q.flatten(1).scatter_add_(1, at, w * dK.flatten()[at])
            tr[:, :, n] = self.sample(q)
        return tr

    def adjoint(self, hist, res):
        """(g_K, g_bx, g_bz) on the padded grid of sum(res * traces), from the kept history."""
        B = res.shape[0]
        z = lambda: torch.zeros((B, self.Nz, self.Nx), device=DEV, dtype=torch.float64)
        l, lx, lz = z(), z(), z()
        gK, gx, gz = (torch.zeros((self.Nz, self.Nx), device=DEV, dtype=torch.float64) for _ in range(3))
        at, w = self.rec
        at = at.flatten()[None].expand(B, -1)
        for n in range(self.c["nt"] - 1, -1, -1):
            l = l.clone()
            l.flatten(1).scatter_add_(1, at, (res[:, :, n, None] * w).flatten(1))
            gK += (l * (hist[n + 1] - self.dp * hist[n])).sum(0)      # K d p^{n+1} / d K
            q = self.dp * l
            lx = self.dvx * (lx + self.diff(self.K * q, -1, True))
            lz = self.dvz * (lz + self.diff(self.K * q, -2, True))
            gx -= (lx * self.diff(hist[n], -1, True)).sum(0)
            gz -= (lz * self.diff(hist[n], -2, True)).sum(0)
            l = q + self.diff(self.bx * lx, -1, False) + self.diff(self.bz * lz, -2, False)
        return gK / self.K, gx, gz

    def fold(self, f):
        """Sum of the padded cells onto the physical cell whose model they copy."""
        c = self.c
        o = torch.zeros((c["nz"], self.Nx), device=DEV, dtype=torch.float64).index_add_(0, self.iz, f)
        return torch.zeros((c["nz"], c["nx"]), device=DEV, dtype=torch.float64).index_add_(1, self.ix, o)

    def chain(self, gK, gx, gz):
        """The gradient in all five parameterizations, [5][2][nz][nx]."""
        gr = torch.zeros_like(gK)
        for b, g, ax in ((self.bx, gx, -1), (self.bz, gz, -2)):
            h, n = -0.5 * b * b * g, g.shape[ax]
            gr += h
            gr.narrow(ax, 1, n - 1).add_(h.narrow(ax, 0, n - 1))
            gr.narrow(ax, n - 1, 1).add_(h.narrow(ax, n - 1, 1))
        sK, sR = self.fold(gK), self.fold(gr)
        K, r, vo, ro = self.K0, self.rho0, self.vo, self.ro
        v, Ko, Io = torch.sqrt(K / r), ro * vo * vo, ro * vo
        return torch.stack([torch.stack(x) for x in (
            (vo * 2 * r * v * sK, ro * (sR + v * v * sK)), (Io * 2 * v * sK, ro * (sR - v * v * sK)),
            (vo * (r * v * sK - r / v * sR), Io * (v * sK + sR / v)), (Ko * sK, ro * sR),
            (-K * K / Ko * sK, -r * r / ro * sR))])

    def chunks(self, history):
        per = 8.0 * self.Nx * self.Nz * (self.c["nt"] + 2 if history else 24)
        B = max(1, min(self.c["ns"], int(40e9 / per)))
        return [(s, min(s + B, self.c["ns"])) for s in range(0, self.c["ns"], B)]

    def gradient(self, data):
        J, G, T = 0.0, 0, []
        for s0, s1 in self.chunks(True):
            tr, hist = self.forward(s0, s1, keep=True)
            r = tr - data[s0:s1].double()
            J = J + 0.5 * r.square().sum()
            G = [x + y for x, y in zip(G, self.adjoint(hist, r))] if G else self.adjoint(hist, r)
            T.append(tr)
        return J, self.chain(*G), torch.cat(T)


def _green(f, r):
    """G_o and dG_o/dr (complex128) at frequency f and distance r (vp_o = rho_o = 2000)."""
    k = 2.0 * math.pi * f / 2000.0
    x, s = k * r, torch.special
    return (torch.complex(-500.0 * s.bessel_y0(x), 500.0 * s.bessel_j0(x)),
            torch.complex(500.0 * k * s.bessel_y1(x), -500.0 * k * s.bessel_j1(x)))


def _inverse_map(pz, scheme, a, b):
    """(xi_1/K, xi_1/rho) of the contrasts, linearly (1) or exactly (2)."""
    if scheme == 1:
        return {0: (-2 * a - b, -b), 1: (-2 * a + b, -b), 2: (-a - b, a - b), 3: (-a, -b), 4: (a, b)}[pz]
    A, B = 1 + a, 1 + b
    return {0: (1 / (B * A * A) - 1, 1 / B - 1), 1: (B / (A * A) - 1, 1 / B - 1), 2: (1 / (A * B) - 1, A / B - 1),
            3: (1 / A - 1, 1 / B - 1), 4: (a, b)}[pz]


def _freq_exact(c, u):
    x = u["x0"] + c["dx"] * torch.arange(c["nx"], device=DEV, dtype=torch.float64)
    z = u["z0"] + c["dx"] * torch.arange(c["nz"], device=DEV, dtype=torch.float64)
    X = torch.stack([x.repeat(c["nz"]), z.repeat_interleave(c["nx"])], 1)
    pts = torch.from_numpy(np.concatenate([u["src"], u["rec"]])).to(DEV).double()
    d = X[None] - pts[:, None]
    r = d.norm(dim=-1)
    e, ns, dx2 = d / r[..., None], c["ns"], c["dx"] ** 2
    a, b = u["a"].double().flatten(), u["b"].double().flatten()
    x1, x2 = _inverse_map(c["pz"], c["scheme"], a, b)
    S = torch.from_numpy(u["spectrum"]).to(DEV).to(torch.complex128)
    rsr = torch.cdist(pts[:ns], pts[ns:])
    out, J, g1, g2 = [], 0.0, 0.0, 0.0
    for k, f in enumerate(u["freqs"].tolist()):
        w = 2.0 * math.pi * f
        G, D = _green(f, r)
        Dx, Dz = D * e[..., 0], D * e[..., 1]
        al, be = w * w / (2000.0 ** 3) * dx2, -dx2 / 2000.0
        p = al * (G[:ns] * x1) @ G[ns:].T + be * ((Dx[:ns] * x2) @ Dx[ns:].T + (Dz[:ns] * x2) @ Dz[ns:].T)
        p = S[k] * (p + _green(f, rsr)[0])
        out.append(p)
        if c["op"] == "fgradient":
            R = p - u["data"][k].to(torch.complex128)
            J = J + 0.5 * R.abs().square().sum()
            Rc = S[k] * R.conj()
            g1 = g1 + al * (G[:ns] * (Rc @ G[ns:])).sum(0).real
            g2 = g2 + be * (Dx[:ns] * (Rc @ Dx[ns:]) + Dz[:ns] * (Rc @ Dz[ns:])).sum(0).real
    if c["op"] == "fsurvey":
        return torch.stack(out)
    _, back = torch.func.vjp(lambda x, y: _inverse_map(c["pz"], c["scheme"], x, y), a, b)
    ga, gb = back((g1, g2))
    return J, (ga.reshape(c["nz"], c["nx"]), gb.reshape(c["nz"], c["nx"]))


def exact(case, seed):
    c, op = case, case["op"]
    if op in ("fgradient", "fsurvey"):
        return _freq_exact(c, _freq_inputs(c, seed))
    if op == "engine":
        out = []
        for k, j in enumerate(_mix(c)):
            u = _fd_inputs(j, seed + 17 * k)
            s = _Scheme(j, u)
            if j["op"] == "gradient":
                out.append(s.gradient(u["data"])[:2])
            else:
                out.append(s.forward(0, j["ns"])[0] if j["op"] == "model" else s.born(0, j["ns"], u))
        return out
    u = _fd_inputs(c, seed)
    if op == "linesearch":
        J = []
        for a, b in u["trials"]:
            s = _Scheme(c, dict(u, a=a, b=b))
            J.append(sum(0.5 * (s.forward(i, k)[0] - u["data"][i:k].double()).square().sum() for i, k in s.chunks(False)))
        return torch.stack(J)
    s = _Scheme(c, u)
    if op == "model":
        return torch.cat([s.forward(i, k)[0] for i, k in s.chunks(False)])
    if op == "born":
        return torch.cat([s.born(i, k, u) for i, k in s.chunks(False)])
    J, G, T = s.gradient(u["data"])
    if op == "gradient":
        return J, G
    if op == "inversion":
        return J, (G[c["pz"], 0], G[c["pz"], 1])
    return T, G[c["pz"], 0], G[c["pz"], 1]
