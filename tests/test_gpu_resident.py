"""The on-chip time-step kernels (csrc/fwi_resident.cuh): their results are bitwise the streaming
kernels' for every tiling -- one tile, ragged tiles, receivers on tile edges and corners and
more of them in a tile than its shared list holds -- and the launches that are meant to be on
chip are."""
import ctypes

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


def kernels(F, call):
    """(result, names of the kernels launched) of a call."""
    L, buf = F.lib(), ctypes.create_string_buffer(1 << 16)
    L.fwi_profile_report(buf, len(buf))
    L.fwi_profile(1)
    out = call()
    torch.cuda.synchronize()
    L.fwi_profile(0)
    assert L.fwi_profile_report(buf, len(buf)) > 0
    return out, {line.split(" ")[0] for line in buf.value.decode().splitlines()}


def both(F, call, name):
    """The call's outputs with the streaming kernels (a fixed strip height asks for them) and by default."""
    F.fwi_set_tile(40, 0)
    try:
        ref, used = kernels(F, call)
    finally:
        F.fwi_set_tile(0, 0)
    assert not any(name in k for k in used)
    got, used = kernels(F, call)
    assert any(name in k for k in used), used
    return ref, got


# grids on either side of one tile (30 column groups; 41 rows at 8th order, 57 at 4th), thin ones,
# and ones whose last group, tile column or tile row is short
GRIDS = [(2, 2, 4, 0), (2, 9, 8, 3), (104, 25, 8, 8), (105, 26, 8, 8), (112, 49, 4, 4), (114, 50, 4, 4), (33, 90, 8, 4),
         (7, 400, 8, 0), (400, 7, 8, 0), (201, 121, 8, 20), (121, 201, 4, 40)]


def case(nx, nz, order, sponge, ns=3, nr=9, nt=60, seed=7):
    w = I.small_case(seed=seed, nx=max(nx, 8), nz=max(nz, 8), nt=nt, order=order, sponge=sponge, ns=ns, nr=nr)
    if nx < 8 or nz < 8:
        rng = np.random.default_rng(seed)
        w.nx, w.nz = nx, nz
        w.xi_a, w.xi_b = (0.1 * rng.standard_normal((nz, nx)).astype(np.float32) for _ in range(2))
        hi = np.array([(nx - 1) * w.dx, (nz - 1) * w.dx])
        w.src_xy = (hi * rng.random((ns, 2))).astype(np.float32)
        w.rec_xy = (hi * rng.random((nr, 2))).astype(np.float32)
    return w


@pytest.mark.parametrize("nx,nz,order,sponge", GRIDS)
def test_forward_is_bitwise_the_streaming_kernels(F, nx, nz, order, sponge):
    w = case(nx, nz, order, sponge)
    # receivers on every cell of a row and a column, so that tile edges and corners are sampled
    x, z = np.arange(min(nx - 1, 90)) * w.dx + 0.4 * w.dx, np.arange(min(nz - 1, 60)) * w.dx + 0.3 * w.dx
    grid = np.stack(np.meshgrid(x[::7], z[::3]), -1).reshape(-1, 2)
    line = np.concatenate([np.stack([x, np.full_like(x, z[len(z) // 2])], 1), np.stack([np.full_like(z, x[len(x) // 2]), z], 1)])
    w.rec_xy = np.concatenate([w.rec_xy, line, grid]).astype(np.float32)
    g = gpu_grid(w)
    ref, got = both(F, lambda: F.fwi_model(g, w.pz, w.xi_a, w.xi_b, w.src_xy, w.wavelet, w.rec_xy), "k_res_fwd")
    assert ref.abs().max().item() > 0
    assert torch.equal(ref, got)


def test_corner_receivers_of_every_tile(F):
    """A receiver in every cell near the tiles' corners (the diagonal neighbour's cell)."""
    w = case(240, 150, 8, 6, ns=2, nr=3)
    x, z = np.arange(1, 239) * w.dx + 1.0, np.arange(1, 149) * w.dx + 2.0
    w.rec_xy = np.stack(np.meshgrid(x[::2], z), -1).reshape(-1, 2).astype(np.float32)
    g = gpu_grid(w)
    ref, got = both(F, lambda: F.fwi_model(g, w.pz, w.xi_a, w.xi_b, w.src_xy, w.wavelet, w.rec_xy), "k_res_fwd")
    assert torch.equal(ref, got)


@pytest.mark.parametrize("every", [0, 17])
def test_gradient_history_and_checkpoints(F, every):
    """The pressure history and the checkpoints that the on-chip forward steps write."""
    w = case(150, 96, 8, 12, ns=3, nr=20, nt=70)
    g = gpu_grid(w)
    data = I.random_like((w.ns, w.nr, w.nt), 5, 1.0)
    F.fwi_set_checkpoint(every)
    try:
        ref, got = both(F, lambda: F.fwi_gradient(g, w.pz, w.xi_a, w.xi_b, w.src_xy, w.wavelet, w.rec_xy, data),
                        "k_res_fwd")
    finally:
        F.fwi_set_checkpoint(0)
    assert torch.equal(ref[0], got[0]) and torch.equal(ref[1], got[1])


@pytest.mark.parametrize("nx,nz,order,sponge", GRIDS)
def test_adjoint_is_bitwise_the_streaming_kernels(F, nx, nz, order, sponge):
    """Two accumulation chunks, receivers that share cells and more of them than a tile lists."""
    w = case(nx, nz, order, sponge, nt=70)
    hi = np.array([(nx - 1) * w.dx, (nz - 1) * w.dx])
    more = (hi * np.random.default_rng(3).random((90, 2))).astype(np.float32)
    w.rec_xy = np.concatenate([w.rec_xy, more, more[::5]]).astype(np.float32)
    g = gpu_grid(w)
    res = I.random_like((w.ns, len(w.rec_xy), w.nt), 11, 1.0)
    ref, got = both(F, lambda: F.fwi_adjoint(g, w.pz, w.xi_a, w.xi_b, w.src_xy, w.wavelet, w.rec_xy, res), "k_res_adj")
    assert ref.abs().max().item() > 0
    assert torch.equal(ref, got)


@pytest.mark.parametrize("nx,nz,order,sponge", GRIDS)
def test_born_is_bitwise_the_streaming_kernels(F, nx, nz, order, sponge):
    w = case(nx, nz, order, sponge)
    hi = np.array([(nx - 1) * w.dx, (nz - 1) * w.dx])
    w.rec_xy = np.concatenate([w.rec_xy, (hi * np.random.default_rng(3).random((90, 2))).astype(np.float32)])
    g = gpu_grid(w)
    da, db = (I.random_like(w.xi_a.shape, s, 0.05) for s in (1, 2))
    ref, got = both(F, lambda: F.fwi_born(g, w.pz, w.xi_a, w.xi_b, da, db, w.src_xy, w.wavelet, w.rec_xy), "k_res_born")
    assert ref.abs().max().item() > 0
    assert torch.equal(ref, got)


@pytest.mark.parametrize("iterations", [1, 9, 64, 256])
def test_engine_runs_on_chip_equal_single_calls(F, iterations):
    """Runs of steps between engine calls of any length (odd remainders stream), several shot groups,
    checkpointed gradients with recomputation, jobs spread over launches."""
    from paper_1804_01184_gb300 import engine
    E = engine.Engine(2 << 30)
    E.arena.fill_(0xFF)
    want = []
    for k in range(9):
        w = I.small_case(seed=900 + k, nx=60 + 23 * k, nz=150 - 11 * k, nt=90 + 7 * k, order=4 if k % 4 == 3 else 8, sponge=6,
                         ns=2 + k % 4, nr=8)
        g = gpu_grid(w)
        ar = (g, w.pz, w.xi_a, w.xi_b)
        tail = (w.src_xy, w.wavelet, w.rec_xy)
        budget = 0 if k % 2 else 1 << 28
        op = (F.OP_MODEL, F.OP_BORN, F.OP_GRADIENT)[k % 3]
        work = torch.empty(F.fwi_workspace_bytes(g, w.ns, w.nr, op, budget), dtype=torch.uint8, device="cuda")
        if op == F.OP_MODEL:
            want.append((E.submit_model(*ar, *tail, work_budget=budget), F.fwi_model(*ar, *tail, work=work)))
        elif op == F.OP_BORN:
            d = tuple(I.random_like(w.xi_a.shape, 40 + k + s, 0.05) for s in (0, 1))
            want.append((E.submit_born(*ar, *d, *tail, work_budget=budget), F.fwi_born(*ar, *d, *tail, work=work)))
        else:
            data = I.random_like((w.ns, w.nr, w.nt), 50 + k, 1.0)
            want.append((E.submit_gradient(*ar, *tail, data, work_budget=budget),
                         F.fwi_gradient(*ar, *tail, data, work=work)))
    (res, used) = kernels(F, lambda: {r.ticket: r for r in E.drain(iterations)})
    if iterations >= 64:
        assert any("k_res" in k for k in used), used
    for t, ref in want:
        r = res[t]
        got = (r.traces,) if r.traces is not None else (r.misfit, r.grads)
        for x, y in zip(got, ref if isinstance(ref, tuple) else (ref,)):
            assert torch.equal(x, y)
    E.close()


def test_more_shots_than_a_launch_holds(F):
    w = case(201, 201, 8, 40, ns=33, nr=20, nt=30)
    g = gpu_grid(w)
    ref, got = both(F, lambda: F.fwi_model(g, w.pz, w.xi_a, w.xi_b, w.src_xy, w.wavelet, w.rec_xy), "k_res_fwd")
    assert torch.equal(ref, got)


def test_under_stream_capture(F):
    """A captured call replays: cooperative launches are legal graph nodes."""
    w = case(120, 90, 8, 10, ns=2, nr=8, nt=40)
    g = gpu_grid(w)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    ar = (g, w.pz, d(w.xi_a), d(w.xi_b), d(w.src_xy), d(w.wavelet), d(w.rec_xy))
    work = F.workspace(g, w.ns, w.nr, F.OP_MODEL)
    ref = F.fwi_model(*ar, work=work).clone()
    out = torch.zeros_like(ref)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        F.fwi_model(*ar, traces=out, work=work, check=False)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)


def test_two_threads_on_two_streams(F):
    """Cooperative launches that each nearly fill the GPU, from two threads on their own streams."""
    import threading

    w = case(161, 161, 8, 20, ns=10, nr=20, nt=60)
    g = gpu_grid(w)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    ar = (g, w.pz, d(w.xi_a), d(w.xi_b), d(w.src_xy), d(w.wavelet), d(w.rec_xy))
    ref = F.fwi_model(*ar)
    torch.cuda.synchronize()
    out, errors = [[], []], []

    def run(k):
        try:
            st, work = torch.cuda.Stream(), F.workspace(g, w.ns, w.nr, F.OP_MODEL)
            torch.cuda.synchronize()
            for _ in range(8):
                with torch.cuda.stream(st):
                    out[k].append(F.fwi_model(*ar, work=work, check=False))
            F.fwi_status(work, st)
        except Exception as e:   # noqa: BLE001 -- shown by the assertion below
            errors.append(e)

    threads = [threading.Thread(target=run, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    assert all(torch.equal(x, ref) for xs in out for x in xs)
