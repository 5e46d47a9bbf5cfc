"""tsu_step_n_noalloc in FP64 where the tiles are more than its fixed array holds partial sums (a CTA then takes
several) against tsu_step_n with a workspace: the same states, and energies that are FP64 sums of the same
terms in another order (each lane's sum compensated, then a tree of about 30 additions of terms of both signs:
1e-11 holds with room)."""
import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import inputs, tsu

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.05, mollifier=inputs.GAUSS, sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5)])


# 8 200 001 x 4: 66130 CTAs of one chunk; 124 x 100: far fewer than the array holds
@pytest.mark.parametrize("nx,ny", [(8200001, 4), (124, 100)])
@pytest.mark.parametrize("form", [tsu.TSU_FORM_STANDARD, tsu.TSU_FORM_INCREMENT])
@pytest.mark.parametrize("energy", [True, False])
def test_equals_step_n(nx, ny, form, energy):
    sim = tsu.Simulation.create(nx, DEPTH, dtype="f64", form=form, ny=ny, nbuf=2 if form == tsu.TSU_FORM_STANDARD else 3)
    u0 = tsu.empty_field(sim.g, "f64")
    u0[1:-1, 1 : nx - 1] = torch.from_numpy(np.random.default_rng(1).standard_normal((ny - 2, nx - 2))).cuda()
    out = []
    for fixed in (True, False):
        sim.init(u0)
        e = torch.zeros(3, dtype=torch.float64, device="cuda") if energy else None
        if fixed:
            tsu.tsu_step_n_noalloc(sim.g, "f64", sim.tau, sim.medium, sim.state, 3, energy=e)
        else:
            sim.step(3, energy=e, kernel=1)
        torch.cuda.synchronize()
        out.append((sim.u.clone(), sim.bufs[sim.state.aux].clone(), e))
    (u, p, e), (ru, rp, re) = out
    assert torch.equal(u, ru) and torch.equal(p, rp)
    if energy:
        assert torch.allclose(e, re, rtol=1e-11, atol=0)
