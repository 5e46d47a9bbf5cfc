"""FP64 energies against binary128 on the same states.  A correctly rounded sum is off by its last two roundings
(the sum, times the scale), 4.6e-17 rms each, and by those of the terms, which average out: 6.5e-17 rms.
1e-16 allows for half as much again; plain additions near the top of the tree give 1.1e-16 to 1.6e-16."""
import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import inputs, tsu

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(np.finfo(np.longdouble).nmant < 100, reason="long double is not binary128 here")]
DEPTH = dict(background=1.0, eps=0.05, mollifier=inputs.GAUSS,
             sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5), (inputs.LINE_Y, 1, 1.0, 0.4, 0.4)])


def exact(sim):
    q = np.longdouble
    nx, ny, g = sim.g.nx, sim.g.ny, sim.g
    u, p, hx, hy = (t.cpu().numpy()[:, :nx].astype(q) for t in (sim.u, sim.u_prev, sim.hx, sim.hy))
    cx, cy = q(sim.tau * sim.tau / (g.dx * g.dx)), q(sim.tau * sim.tau / (g.dy * g.dy))
    fx = hx[1:-1, :-1] * (u[1:-1, 1:] - u[1:-1, :-1])
    fy = hy[:-1, 1:-1] * (u[1:, 1:-1] - u[:-1, 1:-1])
    b = cx * (fx[:, 1:] - fx[:, :-1]) + cy * (fy[1:] - fy[:-1])
    d = u[1:-1, 1:-1] - p[1:-1, 1:-1]
    return (d * d - b * p[1:-1, 1:-1]).sum() * q(g.dx * g.dy / (2.0 * sim.tau * sim.tau))


# on chip; one step per launch with the sums of several steps together (1024^2), and each by itself (2200 x 2100)
@pytest.mark.parametrize("nx,ny,fields", [(101, 101, 40), (201, 201, 40), (330, 331, 16), (1024, 1024, 6), (2200, 2100, 6)])
def test_energy(nx, ny, fields):
    err = []
    sim = tsu.Simulation.create(nx, DEPTH, dtype="f64", ny=ny)
    for seed in range(fields):
        rng = np.random.default_rng(seed)
        u0 = inputs.gaussian_hump(nx, ny, sim.g.ld, rng.uniform(0.3, 0.7), rng.uniform(0.3, 0.7), rng.uniform(0.03, 0.2))
        if seed % 2:
            u0[1:-1, 1 : nx - 1] += 0.05 * rng.standard_normal((ny - 2, nx - 2))
        sim.init(torch.from_numpy(u0).cuda())
        ref = exact(sim)
        e = torch.zeros(8, dtype=torch.float64, device="cuda")
        sim.step(8, energy=e)
        err.append(float((np.longdouble(e[0].item()) - ref) / ref))
    assert np.sqrt(np.mean(np.square(err))) <= 1e-16


def test_infinite_energy():
    """A sum that is infinite stays so (its rounding errors are not numbers)."""
    sim = tsu.Simulation.create(101, DEPTH, dtype="f64")
    u0 = tsu.empty_field(sim.g, "f64")
    u0[50, 50] = 1e200
    sim.init(u0)
    e = torch.zeros(8, dtype=torch.float64, device="cuda")
    sim.step(8, energy=e)
    assert torch.isinf(e).all()
