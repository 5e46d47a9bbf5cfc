"""Waits of the on-chip passes that run out (with a test hook no CTA recognises its neighbours' edges; the limit is
then 20 ms): the launch ends soon after the first of them, says so, and the next call on the same workspace is as
good as any."""
import ctypes as C
import time

import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import inputs, tsu

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.05, mollifier=inputs.GAUSS, sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5)])


def problem(dtype, nx, ny):
    sim = tsu.Simulation.create(nx, DEPTH, dtype=dtype, ny=ny)
    u0 = tsu.empty_field(sim.g, dtype)
    u0[1:-1, 1 : nx - 1] = torch.from_numpy(np.random.default_rng(nx).standard_normal((ny - 2, nx - 2))).to(u0.dtype)
    return sim, u0


def other(sim):
    return sim.bufs[sim.state.aux]


def expired(sim, u0, steps, energy):
    """One call in which no CTA gets its neighbours' edges; returns what it left."""
    sim.init(u0)
    e = torch.zeros(steps, dtype=torch.float64, device="cuda") if energy else None
    torch.cuda.synchronize()
    t0 = time.time()
    sim.step(steps, energy=e, debug=4)
    with pytest.raises(tsu.TsuError) as err:
        tsu.tsu_sync_status(sim.ws, sim.ws.numel())
    assert err.value.code == tsu.TSU_ETIMEOUT
    assert time.time() - t0 < 0.5  # one limit, not one after another
    return sim.u.clone(), other(sim).clone()


# FP32 with 2, 6, 12 and 17 rows per warp (with the energy: terms of a pass together, one step behind, lean tiles)
@pytest.mark.parametrize("dtype,nx,ny", [("f32", 300, 200), ("f32", 1200, 1100), ("f32", 1500, 1500), ("f32", 2001, 2000),
                                         ("f64", 201, 201), ("f64", 500, 490)])
@pytest.mark.parametrize("energy", [False, True])
def test_forward(dtype, nx, ny, energy):
    sim, u0 = problem(dtype, nx, ny)
    u, o = expired(sim, u0, 24, energy)
    if dtype == "f64":
        assert u.isnan().any() and o.isnan().any()
    out = []
    for kernel in (0, 1):
        sim.init(u0)
        sim.step(24, kernel=kernel)
        tsu.tsu_sync_status(sim.ws, sim.ws.numel())  # the status was cleared
        out.append((sim.u.clone(), other(sim).clone()))
    for x, y in zip(*out):
        assert torch.equal(x, y)


# a call of two passes and one of several: what is not NaN does not depend on what never arrived
@pytest.mark.parametrize("nx,ny", [(300, 200), (1200, 1100), (1500, 1500), (2001, 2000)])
@pytest.mark.parametrize("energy", [False, True])
@pytest.mark.parametrize("steps", [8, 24])
def test_forward_leaves_no_valid_looking_values(nx, ny, energy, steps):
    sim, u0 = problem("f32", nx, ny)
    u, v = expired(sim, u0, steps, energy)
    assert u.isnan().any() and v.isnan().any()
    sim.init(u0)
    sim.step(steps, kernel=1)
    for x, y in ((u, sim.u), (v, sim.v)):
        ok = ~x.isnan()
        assert torch.equal(x[ok], y[ok])


def adjoint(sim, u0, S, every, hooks):
    """Gradients of a seeded receiver functional; hooks: see tsu_adjoint_hooks."""
    g = sim.g
    rec = torch.arange(20, device="cuda") * 5 + (g.ny // 2) * g.ld + 7
    ck = torch.zeros((tsu.tsu_ckpt_slots(S, every), 2, g.ny, g.ld), dtype=torch.float64, device="cuda")
    sim.init(u0)
    sim.step(S - 1, ckpt=ck, ckpt_every=every)
    dtr = torch.from_numpy(np.random.default_rng(1).standard_normal((S, 20))).cuda()
    out = [torch.zeros((g.ny, g.ld), dtype=torch.float64, device="cuda") for _ in range(4)]
    wsb = tsu.tsu_adjoint_workspace(g, sim.dtype, sim.form, S, every, 20)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    f = tsu.load().tsu_adjoint_hooks
    vp = C.c_void_p
    f.argtypes = tsu.load().tsu_adjoint.argtypes[:-1] + [C.c_int32, vp]
    f.restype = C.c_int
    torch.cuda.synchronize()
    t0 = time.time()
    rc = f(C.byref(g), sim.dtype, sim.form, sim.tau, C.byref(sim.medium), S, every, ck.data_ptr(), u0.data_ptr(), 20,
           rec.data_ptr(), dtr.data_ptr(), *(t.data_ptr() for t in out), ws.data_ptr(), wsb, hooks,
           torch.cuda.current_stream().cuda_stream)
    assert rc == tsu.TSU_OK
    torch.cuda.synchronize()
    assert time.time() - t0 < 0.5
    return out


@pytest.mark.parametrize("nx,ny", [(130, 200), (400, 390)])
def test_adjoint(nx, ny):
    """tsu_adjoint has no status word: an expired wait shows as NaN in the gradients that depend on it."""
    sim, u0 = problem("f64", nx, ny)
    S = 41
    g_hx, g_hy, g_u0, g_u1 = adjoint(sim, u0, S, 20, 4)  # recompute: the states, hence the face gradients
    assert g_hx.isnan().any() and g_hy.isnan().any()
    g_hx, g_hy, g_u0, g_u1 = adjoint(sim, u0, S, 20, 8)  # sweep: the multipliers, hence all of them
    assert all(g.isnan().any() for g in (g_hx, g_hy, g_u0, g_u1))
    for a, b in zip(adjoint(sim, u0, S, 20, 0), adjoint(sim, u0, S, 7, 0)):  # on chip; one step per launch
        assert torch.equal(a, b) and torch.isfinite(a).all()
