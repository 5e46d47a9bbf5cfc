"""The on-chip FP32 pass where its tests had not been: values that are not finite on every kind of tile, with the
energy, and launches on streams of different priority."""
import threading

import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import inputs, tsu

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.03, mollifier=inputs.GAUSS, sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5)])


def start(dtype, nx, ny, spoil=None):
    sim = tsu.Simulation.create(nx, DEPTH, dtype=dtype, ny=ny)
    u0 = tsu.empty_field(sim.g, dtype)
    u0[1:-1, 1 : nx - 1] = torch.from_numpy(np.random.default_rng(nx).standard_normal((ny - 2, nx - 2))).to(u0.dtype)
    if spoil is not None:  # beside the last column and the last row, and in the middle of a tile
        u0[ny // 3, nx - 2] = u0[ny - 2, nx // 3] = u0[ny // 2, nx // 2] = spoil
    sim.init(u0)
    return sim


# 2 rows per warp, 8 and 12 in tensor memory, 17 (lean)
@pytest.mark.parametrize("nx,ny", [(301, 200), (1301, 1203), (1501, 1502), (2045, 1990)])
@pytest.mark.parametrize("energy", [False, True])
@pytest.mark.parametrize("spoil", [float("nan"), float("-inf"), 3e38])
def test_not_finite(nx, ny, energy, spoil):
    out = []
    for kernel in (0, 2):
        sim = start("f32", nx, ny, spoil)
        e = torch.zeros(9, dtype=torch.float64, device="cuda") if energy else None
        sim.step(9, energy=e, kernel=kernel, rows=16 if kernel else 0)
        out.append((sim.u.clone(), sim.v.clone(), e))
    for x, y in zip(out[0][:2], out[1][:2]):
        ok = y.isfinite()
        assert torch.equal(x.isfinite(), ok) and torch.equal(x[ok], y[ok]) and not ok.all()
    if energy:
        assert torch.equal(out[0][2].isfinite(), out[1][2].isfinite())


def test_streams_of_different_priority():
    cases = [("f32", 1025, 900, 0), ("f32", 1400, 1400, -1), ("f64", 500, 499, -1), ("f32", 300, 200, 0)]
    alone, together = ([start(*c[:3]) for c in cases] for _ in range(2))
    for sim in alone:
        for _ in range(20):
            sim.step(100)
    torch.cuda.synchronize()

    def work(sim, priority):
        s = torch.cuda.Stream(priority=priority)
        for _ in range(20):
            sim.step(100, stream=s)
        s.synchronize()

    threads = [threading.Thread(target=work, args=(sim, c[3])) for sim, c in zip(together, cases)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, b in zip(alone, together):
        tsu.tsu_sync_status(b.ws, b.ws.numel())
        assert torch.equal(a.u, b.u)
