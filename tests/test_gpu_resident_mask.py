"""What lies in the padding and in faces that border no interior node never reaches a result: the steps on
chip mask nothing but the rows, so they have to drop it when they read the fields."""
import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import inputs, tsu

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.03, mollifier=inputs.GAUSS, sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5)])


def run(dtype, nx, ny, ld, kernel, spoil):
    sim = tsu.Simulation.create(nx, DEPTH, dtype=dtype, ny=ny, ld=ld)
    u0 = tsu.empty_field(sim.g, dtype)
    u0[1:-1, 1 : nx - 1] = torch.from_numpy(np.random.default_rng(nx).standard_normal((ny - 2, nx - 2))).to(u0.dtype)
    sim.init(u0)
    if spoil is not None:  # hx: faces 0 .. nx - 2 of rows 1 .. ny - 2; hy: faces 0 .. ny - 2 of columns 1 .. nx - 2
        sim.hx[:, nx - 1 :] = sim.hx[0] = sim.hx[-1] = spoil
        sim.hy[:, nx - 1 :] = sim.hy[:, 0] = sim.hy[ny - 1] = spoil
        sim.u[:, nx:] = sim.bufs[sim.state.aux][:, nx:] = spoil
    e = torch.zeros(13, dtype=torch.float64, device="cuda")
    sim.step(13, energy=e, kernel=kernel)
    torch.cuda.synchronize()
    return sim.u[:, :nx].clone(), sim.bufs[sim.state.aux][:, :nx].clone(), e


# FP32: fields in registers, in tensor memory (5 to 17 rows per warp, 17 being the lean tile); FP64; the last
# column of the grid first, within and last in a lane's four columns, with and without padding
@pytest.mark.parametrize("dtype,nx,ny,ld", [("f32", 257, 130, None), ("f32", 258, 131, None), ("f32", 259, 90, 320),
                                            ("f32", 256, 130, 256), ("f32", 1102, 1100, None), ("f32", 2045, 1990, None),
                                            ("f64", 257, 130, None), ("f64", 302, 300, 352)])
@pytest.mark.parametrize("spoil", [float("nan"), float("inf")])
def test_unused_entries(dtype, nx, ny, ld, spoil):
    a, b = (run(dtype, nx, ny, ld, 0, s) for s in (spoil, None))
    for x, y in zip(a, b):
        assert torch.equal(x, y)
