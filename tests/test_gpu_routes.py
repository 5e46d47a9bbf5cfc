"""The passes that the automatic choice takes: on chip where the grid fits, and not where it does not (the tests
of results compare the automatic choice with a pass it would silently fall back to)."""
from collections import Counter

import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import inputs, tsu
from tests.routes import launches

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.05, mollifier=inputs.GAUSS, sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5)])


def route(dtype, nx, ny, steps, energy=False, nrec=0, every=0, first=0, slots=None, **kw):
    """Kernels of one tsu_step_n call of `steps` steps that starts `first` steps after the start."""
    sim = tsu.Simulation.create(nx, DEPTH, dtype=dtype, ny=ny, **kw)
    sim.init(tsu.empty_field(sim.g, dtype))
    if first:
        sim.step(first, kernel=1)
    o = dict(energy=torch.zeros(steps, dtype=torch.float64, device="cuda") if energy else None)
    if nrec:
        o["rec_idx"] = torch.arange(nrec, device="cuda") * 3 + sim.g.ld + 1
        o["traces"] = torch.zeros((steps, nrec), dtype=tsu.DTYPES[sim.dtype], device="cuda")
    if every:
        slots = slots or (first + steps) // every + 2
        o["ckpt"] = torch.zeros((slots, 2, ny, sim.g.ld), dtype=tsu.DTYPES[sim.dtype], device="cuda")
        o["ckpt_every"] = every
    return Counter(k for k in launches(lambda s: sim.step(steps, stream=s, **o)) if k.startswith("k_leapfrog"))


@pytest.mark.parametrize("nx,ny", [(64, 64), (1003, 517), (769, 769), (1400, 1400), (1536, 1536), (2048, 2048), (97, 3001)])
@pytest.mark.parametrize("energy", [False, True])
def test_fp32_on_chip(nx, ny, energy):
    assert route("f32", nx, ny, 64, energy) == {"k_leapfrog_res": 1}
    if nx * ny < 1700 ** 2:
        assert route("f32", nx, ny, 64, energy, nrec=9) == {"k_leapfrog_res": 1}


def test_fp32_streaming():
    """Too large for the chip, or an option that the pass on chip does not have."""
    assert route("f32", 2304, 2304, 64) == {"k_leapfrog_wtb_flow": 1}
    assert route("f32", 4096, 2048, 64, True) == {"k_leapfrog_wtb_flow": 1}
    assert "k_leapfrog_res" not in route("f32", 1900, 1900, 64, True, nrec=9)
    assert "k_leapfrog_res" not in route("f32", 513, 513, 64, True, every=16)
    assert "k_leapfrog_res" not in route("f32", 513, 513, 64, form=tsu.TSU_FORM_STANDARD)
    assert "k_leapfrog_res" not in route("f32", 513, 513, 64, nbuf=3)
    assert "k_leapfrog_res" not in route("f32", 513, 513, 64, nrec=513)
    assert "k_leapfrog_res" not in route("f32", 513, 513, 4)


@pytest.mark.parametrize("nx,ny", [(40, 40), (201, 201), (500, 499), (730, 720)])
@pytest.mark.parametrize("energy,nrec", [(False, 0), (True, 60)])
def test_fp64(nx, ny, energy, nrec):
    assert route("f64", nx, ny, 64, energy, nrec) == {"k_leapfrog_res64": 1}


def test_fp64_one_step_per_launch():
    assert route("f64", 800, 801, 20, True) == {"k_leapfrog64": 20}
    assert route("f64", 201, 201, 20, form=tsu.TSU_FORM_INCREMENT) == {"k_leapfrog64": 20}
    assert route("f64", 201, 201, 3) == {"k_leapfrog64": 3}


@pytest.mark.parametrize("nx,ny,chip", [(201, 201, True), (400, 390, True), (800, 801, False)])
def test_fp64_adjoint(nx, ny, chip):
    sim = tsu.Simulation.create(nx, DEPTH, dtype="f64", ny=ny)
    g, S, every = sim.g, 41, 20
    rec = torch.arange(9, device="cuda") * 3 + g.ld + 1
    z = lambda *shape: torch.zeros(shape, dtype=torch.float64, device="cuda")
    ck, dtr, out = z(tsu.tsu_ckpt_slots(S, every), 2, ny, g.ld), z(S, 9), [z(ny, g.ld) for _ in range(5)]
    wsb = tsu.tsu_adjoint_workspace(g, sim.dtype, sim.form, S, every, 9)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    call = lambda s: tsu.tsu_adjoint(g, sim.dtype, sim.form, sim.tau, sim.medium, S, every, ck, out[4], rec, dtr,
                                     *out[:4], ws, wsb, stream=s)
    call(torch.cuda.current_stream())  # this thread's recompute stream is created outside the capture
    n = Counter(launches(call))
    if chip:
        assert (n["k_leapfrog_res64"], n["k_adjoint_res64"]) == (2, 2) and not n["k_adjoint64"] and not n["k_leapfrog64"]
    else:
        assert not n["k_leapfrog_res64"] and not n["k_adjoint_res64"] and n["k_adjoint64"] == 41


@pytest.mark.parametrize("nx,ny,steps", [(2304, 2304, 61), (4096, 1500, 45)])
def test_persistent_streaming_pass_equals_one_step_passes(nx, ny, steps):
    """The automatic choice above the grids that fit on chip."""
    out = []
    for kernel in (0, 1):
        sim = tsu.Simulation.create(nx, DEPTH, dtype="f32", ny=ny)
        u0 = tsu.empty_field(sim.g, "f32")
        u0[1:-1, 1 : nx - 1] = torch.from_numpy(np.random.default_rng(2).standard_normal((ny - 2, nx - 2), dtype=np.float32))
        sim.init(u0)
        e = torch.zeros(steps, dtype=torch.float64, device="cuda")
        sim.step(steps, energy=e, kernel=kernel)
        tsu.tsu_sync_status(sim.ws, sim.ws.numel())
        out.append((sim.u.clone(), sim.v.clone(), e))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert torch.allclose(out[0][2], out[1][2], rtol=1e-6, atol=0)  # FP32 sums of other nodes
