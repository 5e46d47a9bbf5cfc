"""The FP32 energies of the on-chip pass against kernel 2's at 16 rows per tile: sums of the same chains, there in
FP64, here in three FP32 numbers that hold more, then both over the CTAs in FP64.  The additions that matter
are the last few near the top of each FP64 tree and the scale, roundings of 6.4e-17 rms each: about 2e-16 rms of
the difference, 2e-15 with room for the largest of 400 steps and for terms of both signs."""
import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import inputs, tsu

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.05, mollifier=inputs.GAUSS,
             sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5), (inputs.LINE_Y, 1, 1.0, 0.4, 0.4)])


# the terms of a pass together (up to 8 rows per warp), one step behind, lean tiles
@pytest.mark.parametrize("nx,ny", [(64, 64), (1003, 517), (1024, 1024), (1400, 1400), (2048, 2048), (3001, 97)])
@pytest.mark.parametrize("noise", [0.0, 0.05])
def test_sums(nx, ny, noise):
    out = []
    for kernel in (0, 2):
        sim = tsu.Simulation.create(nx, DEPTH, dtype="f32", ny=ny)
        u0 = inputs.gaussian_hump(nx, ny, sim.g.ld, 0.4, 0.45, 0.1)
        u0[1:-1, 1 : nx - 1] += noise * np.random.default_rng(nx).standard_normal((ny - 2, nx - 2))
        sim.init(torch.from_numpy(u0).float().cuda())
        e = torch.zeros(400, dtype=torch.float64, device="cuda")
        sim.step(400, energy=e, kernel=kernel, rows=16 if kernel else 0)
        out.append(e)
    assert torch.allclose(*out, rtol=2e-15, atol=0)
