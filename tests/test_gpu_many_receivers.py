"""Grouping the adjoint's receivers is linear in their number, and keeps their order within a tile: long lists,
several on one node, against the oracle; and the time of a list of 300 000."""
import numpy as np
import pytest
import torch

import oracle
from paper_2005_11931_gb300 import inputs, tsu
from tests.gpu_helpers import relerr
from tests.test_gpu_adjoint import gpu_forward_adjoint

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.06, mollifier=0, sings=[(0, 1, 0.5, 0.5, 0.5)])


# fewer than a warp, whole warps and one more or less, more than the on-chip sweep keeps, far more than threads; FP32
# and FP64 group by other units.  Many of the nodes repeat: FP32 sums are compared at the tolerance of its adjoint
@pytest.mark.parametrize("dtype,tol", [("f64", 1e-12), ("f32", 2e-5)])
@pytest.mark.parametrize("nrec", [1, 31, 32, 33, 64, 513, 1025, 5000])
def test_grouping(dtype, tol, nrec):
    nx, ny, S = 97, 90, 9
    rng = np.random.default_rng(nrec)
    u0, u1 = inputs.random_field(nx, ny, None, rng), inputs.random_field(nx, ny, None, rng)
    rec = np.stack([rng.integers(0, nx, nrec), rng.integers(0, ny, nrec)], 1)
    rec[nrec // 2 :] = rec[: nrec - nrec // 2]
    dtr = rng.standard_normal((S, nrec))
    form = tsu.TSU_FORM_STANDARD if dtype == "f64" else tsu.TSU_FORM_INCREMENT
    out, tau = gpu_forward_adjoint(nx, ny, DEPTH, u0, u1, S, rec, dtr, dtype, form, 5)
    g = oracle.grid(nx, ny)
    hx, hy, _ = oracle.make_depth(g, DEPTH)
    ref = oracle.adjoint(g, tau, hx, hy, u0[:, :nx], u1[:, :nx], S, inputs.flat_index(rec, g.ld), dtr)
    for k in ("g_hx", "g_hy", "g_u0", "g_u1"):
        assert relerr(out[k], ref[k][:, :nx]) <= tol, k


def test_time_of_a_long_list():
    """300 000 receivers, 180 a tile: 10 000 rounds of a warp at 2 us are 20 ms, and the three injections as
    long again; 0.25 s leaves room for both, and none for a count over all earlier ones (0.87 s)."""
    n, nrec, S = 600, 300000, 3
    sim = tsu.Simulation.create(n, DEPTH, dtype="f64")
    g = sim.g
    rng = np.random.default_rng(0)
    rec = torch.from_numpy(rng.integers(1, n - 1, nrec) * g.ld + rng.integers(1, n - 1, nrec)).cuda()
    dtr = torch.zeros((S, nrec), dtype=torch.float64, device="cuda")
    ck = torch.zeros((1, 2, g.ny, g.ld), dtype=torch.float64, device="cuda")
    out = [torch.zeros((g.ny, g.ld), dtype=torch.float64, device="cuda") for _ in range(5)]
    wsb = tsu.tsu_adjoint_workspace(g, sim.dtype, sim.form, S, 64, nrec)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for _ in range(2):
        ev[0].record()
        tsu.tsu_adjoint(g, sim.dtype, sim.form, sim.tau, sim.medium, S, 64, ck, out[4], rec, dtr, *out[:4], ws, wsb)
        ev[1].record()
        torch.cuda.synchronize()
    assert ev[0].elapsed_time(ev[1]) < 250
