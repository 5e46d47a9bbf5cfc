"""Stretches between checkpoints on chip: which of them run there, and that states, traces, checkpoints and (FP64)
energies are those of one step per pass."""
import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import tsu
from tests.test_gpu_routes import DEPTH, route

pytestmark = pytest.mark.gpu


def outputs(dtype, nx, ny, first, steps, every, slots, kernel, energy):
    sim = tsu.Simulation.create(nx, DEPTH, dtype=dtype, ny=ny)
    rng = np.random.default_rng(nx)
    u0 = tsu.empty_field(sim.g, dtype)
    u0[1:-1, 1 : nx - 1] = torch.from_numpy(rng.standard_normal((ny - 2, nx - 2))).to(u0.dtype)
    rec = torch.from_numpy(rng.integers(0, ny * sim.g.ld, 9)).cuda()
    sim.init(u0)
    sim.step(first, kernel=1)
    ck = torch.full((slots, 2, ny, sim.g.ld), 5.0, dtype=u0.dtype, device="cuda")
    tr = torch.zeros((steps, 9), dtype=u0.dtype, device="cuda")
    e = torch.zeros(steps, dtype=torch.float64, device="cuda") if energy else None
    sim.step(steps, energy=e, ckpt=ck, ckpt_every=every, rec_idx=rec, traces=tr, kernel=kernel)
    torch.cuda.synchronize()
    return sim.u.clone(), sim.bufs[sim.state.aux].clone(), ck, tr, e


def same(dtype, nx, ny, first, steps, every, slots):
    energy = dtype == "f64"
    a, b = (outputs(dtype, nx, ny, first, steps, every, slots, k, energy) for k in (0, 1))
    for x, y in zip(a[:4], b[:4]):
        assert torch.equal(x, y)
    if energy:
        assert torch.allclose(a[4], b[4], rtol=1e-11, atol=0)


@pytest.mark.parametrize("dtype,nx,ny", [("f32", 300, 200), ("f64", 129, 257)])
def test_short_stretch_before_a_checkpoint(dtype, nx, ny):
    chip, one = ("k_leapfrog_res", "k_leapfrog") if dtype == "f32" else ("k_leapfrog_res64", "k_leapfrog64")
    # 3 + 4 x 16; the same and 5 more; 7 + 5 x 10 + 3; 1 + 12 + 7
    for first, steps, every, n_chip, n_one in ((13, 67, 16, 4, 3), (13, 72, 16, 4, 8), (3, 60, 10, 5, 10), (11, 20, 12, 1, 8)):
        got = route(dtype, nx, ny, steps, nrec=9, every=every, first=first)
        assert got == {chip: n_chip, one: n_one}, (first, steps, every)
        same(dtype, nx, ny, first, steps, every, (first + steps) // every + 2)
    # no stretch is long enough
    assert chip not in route(dtype, nx, ny, 40, nrec=9, every=7, first=3)
    same(dtype, nx, ny, 3, 40, 7, 9)


@pytest.mark.parametrize("dtype,nx,ny", [("f32", 300, 200), ("f64", 129, 257)])
def test_full_store(dtype, nx, ny):
    """Behind the last slot no checkpoint cuts the call: 2 slots of 16 steps (states 1 and 17), then one launch."""
    chip, one = ("k_leapfrog_res", "k_leapfrog") if dtype == "f32" else ("k_leapfrog_res64", "k_leapfrog64")
    assert route(dtype, nx, ny, 100, nrec=9, every=16, slots=2) == {chip: 2}
    assert route(dtype, nx, ny, 100, nrec=9, every=16, first=40, slots=2) == {chip: 1}
    assert route(dtype, nx, ny, 103, nrec=9, every=16, first=13, slots=2) == {one: 3, chip: 1}
    for first, steps in ((0, 100), (40, 100), (13, 103), (16, 50)):
        same(dtype, nx, ny, first, steps, 16, 2)


def test_fewest_steps():
    """With receivers or checkpoints the tiles of 17 rows per warp start at 16 steps, the others at 8; without
    them all at 8."""
    for n, fewest in ((1800, 8), (1900, 16), (2048, 16)):
        assert route("f32", n, n, fewest, nrec=9) == {"k_leapfrog_res": 1}
        assert route("f32", n, n, 48, every=fewest) == {"k_leapfrog_res": 48 // fewest}
        assert route("f32", n, n, 8) == route("f32", n, n, 8, True) == {"k_leapfrog_res": 1}
        assert "k_leapfrog_res" not in route("f32", n, n, fewest - 4, nrec=9)
        assert "k_leapfrog_res" not in route("f32", n, n, 48, every=fewest - 4)
    # an interval that the four-step pass cannot take
    assert route("f32", 1900, 1900, 45, every=9) == {"k_leapfrog_res": 5}
