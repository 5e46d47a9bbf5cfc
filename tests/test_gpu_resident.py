"""The resident pass (every step of a call in one cooperative launch, fields on chip): the automatic
choice for FP32 grids that fit, against the warp-blocked pass (kernel 2, tiles of 16 rows) on the same problem.

The states and traces have to be the same bits (same operations per node).  The energies are sums of
the same FP32 chains, added up in FP64 (and in pairs of FP32 with their rounding errors) in another
order: at most 2e4 chains, partial sums good to 2^-46, terms of both signs that cancel to about 1e-3 of
their magnitude, so 1e-10 relative holds with room."""
import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import inputs, tsu

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.03, mollifier=inputs.GAUSS,
             sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5), (inputs.LINE_Y, 1, 1.0, 0.4, 0.4)])


def run(nx, ny, calls, kernel, energy=False, nrec=0, spoil=None):
    """u, v, energies and traces after the calls (numbers of steps) of one simulation."""
    sim = tsu.Simulation.create(nx, DEPTH, dtype="f32", ny=ny)
    u0 = tsu.empty_field(sim.g, "f32")
    rng = np.random.default_rng(nx * 10007 + ny)
    u0[:, :nx] = torch.from_numpy(rng.standard_normal((ny, nx)).astype(np.float32)).cuda()
    u0[0] = u0[-1] = 0
    u0[:, 0] = u0[:, nx - 1] = 0
    if spoil is not None:
        u0[ny // 2, 1] = spoil
        u0[1, nx // 2] = spoil
    rec = torch.from_numpy(rng.integers(-5, ny * sim.g.ld + 5, nrec)).cuda() if nrec else None
    sim.init(u0)
    es, ts = [], []
    for n in calls:
        e = torch.full((n,), -1.0, dtype=torch.float64, device="cuda") if energy else None
        t = torch.full((n, nrec), 7.0, device="cuda") if nrec else None
        sim.step(n, energy=e, rec_idx=rec, traces=t, kernel=kernel, rows=16 if kernel else 0)
        es.append(e)
        ts.append(t)
    torch.cuda.synchronize()
    return sim.u.clone(), sim.v.clone(), torch.cat(es) if energy else None, torch.cat(ts) if nrec else None


# 17 strips of columns leave 8 chunks of rows on 152 SMs: the rows per warp grow with ny, from 2 to 17
# without the energy (12 with it); the last ones are too large for either
SIZES = [(2001, ny) for ny in (130, 249, 300, 381, 400, 500, 561, 630, 700, 800, 881, 900, 1100, 1139, 1350, 1401,
                               1600, 2000, 2046)]
SIZES += [(3, 3), (4, 70), (5, 200), (64, 64), (65, 34), (97, 3001), (120, 130), (121, 2449), (3001, 97), (1025, 1023), (2200, 1700)]
SIZES += [(64, 723), (130, 724), (64, 725)]  # a last chunk of 1, 2, 3 rows: halos reach past it


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("energy", [False, True])
def test_states_and_energies(nx, ny, energy):
    a = run(nx, ny, (13, 8), 0, energy)
    b = run(nx, ny, (13, 8), 2, energy)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    if energy:
        assert torch.allclose(a[2], b[2], rtol=1e-10, atol=0)


@pytest.mark.parametrize("nx,ny,nrec,energy", [(2001, 300, 1, False), (2001, 1600, 512, False), (769, 769, 200, True),
                                               (130, 70, 512, True), (65, 2001, 33, False), (2001, 1139, 77, True)])
def test_receivers(nx, ny, nrec, energy):
    a = run(nx, ny, (13, 30), 0, energy, nrec)
    b = run(nx, ny, (13, 30), 2, energy, nrec)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and torch.equal(a[3], b[3])
    if energy:
        assert torch.allclose(a[2], b[2], rtol=1e-10, atol=0)


def test_long_calls():
    """More passes than the energy partials of one launch hold."""
    a = run(201, 333, (2500,), 0, True)
    b = run(201, 333, (2500,), 2, True)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert torch.allclose(a[2], b[2], rtol=1e-10, atol=0)


@pytest.mark.parametrize("spoil", [float("nan"), float("inf"), -3e38])
def test_not_finite(spoil):
    """Nodes that are not finite spread as in the other passes, and the boundary stays 0."""
    a = run(257, 130, (9,), 0, False, 0, spoil)
    b = run(257, 130, (9,), 2, False, 0, spoil)
    for x, y in zip(a[:2], b[:2]):
        assert torch.equal(x.isfinite(), y.isfinite())
        assert torch.equal(x[x.isfinite()], y[y.isfinite()])


def test_capture_and_side_stream():
    """Under stream capture and on a side stream, as the passes before it."""
    sim = tsu.Simulation.create(300, DEPTH, dtype="f32", ny=200)
    u0 = tsu.empty_field(sim.g, "f32")
    u0[1:-1, 1:299] = torch.rand(198, 298, device="cuda")
    sim.init(u0)
    start = [b.clone() for b in (sim.u, sim.v)]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        sim.step(16, stream=s)
        sim.step(16, stream=s)
    torch.cuda.synchronize()
    ref = sim.u.clone()
    sim.init(u0)
    assert torch.equal(sim.u, start[0]) and torch.equal(sim.v, start[1])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        sim.step(16, stream=s)
        sim.step(16, stream=s)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(sim.u, ref)


@pytest.mark.parametrize("dtype,nx,ny", [("f32", 300, 200), ("f32", 1025, 900), ("f64", 129, 257)])
@pytest.mark.parametrize("every,calls", [(16, (70, 21)), (10, (47, 30)), (5, (23,)), (64, (64, 64, 9))])
def test_checkpoints(dtype, nx, ny, every, calls):
    """A launch per stretch between checkpoints: the same checkpoints, states and traces as one step per
    pass, also when a call starts or ends between two, and when a stretch is too short for a launch."""
    out = []
    for kernel in (0, 1):
        sim = tsu.Simulation.create(nx, DEPTH, dtype=dtype, ny=ny)
        rng = np.random.default_rng(3)
        u0 = tsu.empty_field(sim.g, dtype)
        u0[1:-1, 1 : nx - 1] = torch.from_numpy(rng.standard_normal((ny - 2, nx - 2))).to(u0.dtype).cuda()
        rec = torch.from_numpy(rng.integers(0, ny * sim.g.ld, 9)).cuda()
        sim.init(u0)
        ck = torch.full((sum(calls) // every + 2, 2, sim.g.ny, sim.g.ld), 5.0, dtype=u0.dtype, device="cuda")
        tr = torch.zeros((sum(calls), 9), dtype=u0.dtype, device="cuda")
        at = 0
        for n in calls:
            sim.step(n, ckpt=ck, ckpt_every=every, rec_idx=rec, traces=tr[at : at + n], kernel=kernel)
            at += n
        torch.cuda.synchronize()
        other = sim.v if sim.form == tsu.TSU_FORM_INCREMENT else sim.u_prev
        out.append((sim.u.clone(), other.clone(), ck, tr))
    for a, b in zip(*out):
        assert torch.equal(a, b)


def test_several_streams_and_threads():
    """Resident launches of several problems from several threads and streams at once: each waits only
    for its own CTAs, so they give what they give one after another."""
    import threading

    cases = [("f32", 1025, 900), ("f32", 300, 200), ("f64", 201, 201), ("f64", 500, 499)]

    def build(dtype, nx, ny):
        sim = tsu.Simulation.create(nx, DEPTH, dtype=dtype, ny=ny)
        u0 = tsu.empty_field(sim.g, dtype)
        u0[1:-1, 1 : nx - 1] = torch.from_numpy(np.random.default_rng(nx).standard_normal((ny - 2, nx - 2))).to(u0.dtype)
        sim.init(u0)
        return sim

    alone, together = [build(*c) for c in cases], [build(*c) for c in cases]
    torch.cuda.synchronize()
    for sim in alone:
        for _ in range(5):
            sim.step(200)
    torch.cuda.synchronize()

    def work(sim):
        s = torch.cuda.Stream()
        for _ in range(5):
            sim.step(200, stream=s)
        s.synchronize()

    threads = [threading.Thread(target=work, args=(sim,)) for sim in together]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, b in zip(alone, together):
        tsu.tsu_sync_status(b.ws, b.ws.numel())
        assert torch.equal(a.u, b.u)
