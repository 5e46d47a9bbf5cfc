"""Values and tags travel between the CTAs of the on-chip passes as aligned 8-byte words, with no flag, fence or
barrier: thousands of exchanges through tiles of few rows (a step takes little longer than an exchange, so
readers poll words that are being written), the same bits as one launch per pass or step."""
import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import inputs, tsu

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.05, mollifier=inputs.GAUSS, sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5)])


@pytest.mark.parametrize("dtype,nx,ny,kernel", [("f32", 2001, 130, 2), ("f32", 130, 2400, 2), ("f32", 1025, 300, 2),
                                                ("f64", 1000, 60, 1), ("f64", 62, 2200, 1), ("f64", 201, 201, 1)])
def test_many_exchanges(dtype, nx, ny, kernel):
    out = []
    for k in (0, kernel):
        sim = tsu.Simulation.create(nx, DEPTH, dtype=dtype, ny=ny)
        u0 = tsu.empty_field(sim.g, dtype)
        u0[1:-1, 1 : nx - 1] = torch.from_numpy(np.random.default_rng(ny).standard_normal((ny - 2, nx - 2))).to(u0.dtype)
        sim.init(u0)
        sim.step(6000, kernel=k)
        torch.cuda.synchronize()
        tsu.tsu_sync_status(sim.ws, sim.ws.numel())
        out.append((sim.u.clone(), sim.bufs[sim.state.aux].clone()))
    for x, y in zip(*out):
        assert torch.equal(x, y) and torch.isfinite(x).all()
