"""FP64 steps on chip (k_step_res64.cu, the automatic choice for small grids in the standard form) against
one step per launch (kernel 1): the same operations per node, so the same bits in states and traces; the
energies are FP64 sums of the same terms in another order (at most 3e5 terms, of both signs that cancel to
about 1e-3 of their magnitude: 1e-11 holds with room)."""
import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import inputs, tsu

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.05, mollifier=inputs.GAUSS,
             sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5), (inputs.LINE_Y, 1, 1.0, 0.4, 0.4)])


def run(nx, ny, calls, kernel, energy, nrec):
    sim = tsu.Simulation.create(nx, DEPTH, dtype="f64", ny=ny)
    rng = np.random.default_rng(nx * 10007 + ny)
    u0 = tsu.empty_field(sim.g, "f64")
    u0[1:-1, 1 : nx - 1] = torch.from_numpy(rng.standard_normal((ny - 2, nx - 2))).cuda()
    rec = torch.from_numpy(rng.integers(-5, ny * sim.g.ld + 5, nrec)).cuda() if nrec else None
    sim.init(u0)
    es, ts = [], []
    for n in calls:
        e = torch.full((n,), -1.0, dtype=torch.float64, device="cuda") if energy else None
        t = torch.full((n, nrec), 7.0, dtype=torch.float64, device="cuda") if nrec else None
        sim.step(n, energy=e, rec_idx=rec, traces=t, kernel=kernel)
        es.append(e)
        ts.append(t)
    torch.cuda.synchronize()
    return sim.u.clone(), sim.u_prev.clone(), torch.cat(es) if energy else None, torch.cat(ts) if nrec else None


# rows per warp 1 .. 16, ragged strips and chunks, more chunks than a warp has lanes, and grids too large
@pytest.mark.parametrize("nx,ny", [(3, 3), (4, 90), (31, 32), (32, 9), (33, 600), (62, 63), (63, 1201), (201, 201),
                                   (330, 331), (400, 401), (500, 499), (1000, 180), (121, 2400), (600, 601), (730, 720), (800, 801)])
@pytest.mark.parametrize("energy,nrec", [(False, 0), (True, 0), (True, 60)])
def test_same_as_one_step_per_launch(nx, ny, energy, nrec):
    a, b = (run(nx, ny, (41, 8, 33), k, energy, nrec) for k in (0, 1))
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    if energy:
        assert torch.allclose(a[2], b[2], rtol=1e-11, atol=0)
    if nrec:
        assert torch.equal(a[3], b[3])


@pytest.mark.parametrize("steps", [512, 513, 1100])
def test_long_calls(steps):
    a, b = (run(90, 100, (steps,), k, True, 3) for k in (0, 1))
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and torch.equal(a[3], b[3])
    assert torch.allclose(a[2], b[2], rtol=1e-11, atol=0)


# the reverse sweep (k_adjoint_res64.cu) of a checkpoint segment on chip (20 steps) against one launch per
# step (segments of 7): the same operations in the same order, so the same bits; receivers on the edges of
# tiles, several on one node, and more than a tile's list holds
@pytest.mark.parametrize("nx,ny,nrec", [(3, 3, 2), (31, 32, 9), (33, 600, 40), (63, 64, 200), (201, 180, 0), (257, 300, 512),
                                        (400, 390, 30), (500, 499, 64), (520, 200, 513), (121, 2400, 25), (700, 690, 8)])
def test_adjoint_on_chip(nx, ny, nrec):
    from tests.test_gpu_adjoint import gpu_forward_adjoint

    S = 47
    rng = np.random.default_rng(nx)
    u0, u1 = inputs.random_field(nx, ny, None, rng), inputs.random_field(nx, ny, None, rng)
    rec = np.stack([rng.integers(0, nx, max(nrec, 1)), rng.integers(0, ny, max(nrec, 1))], 1)[:nrec]
    if nrec > 4:
        rec[:4] = [[1, 1], [nx - 2, ny - 2], [min(30, nx - 2), ny // 2], [min(30, nx - 2), ny // 2]]
    dtr = rng.standard_normal((S, nrec))
    a, _ = gpu_forward_adjoint(nx, ny, DEPTH, u0, u1, S, rec, dtr, "f64", tsu.TSU_FORM_STANDARD, 20)
    b, _ = gpu_forward_adjoint(nx, ny, DEPTH, u0, u1, S, rec, dtr, "f64", tsu.TSU_FORM_STANDARD, 7)
    for k in a:
        assert np.array_equal(a[k], b[k]), k
