"""A bounded wait of a forward run that runs out is reported to callers of the autograd function and of the
studies, which keep the workspace with the status word to themselves."""
import numpy as np
import pytest
import torch

from paper_2005_11931_gb300 import autograd, inputs, study, tsu

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.05, mollifier=inputs.GAUSS, sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5)])


@pytest.mark.parametrize("dtype,n", [("f32", 300), ("f64", 201)])
def test_autograd(dtype, n):
    sim = tsu.Simulation.create(n, DEPTH, dtype=dtype)
    g = sim.g
    u0 = torch.from_numpy(inputs.gaussian_hump(n, n, g.ld, 0.4, 0.5, 0.1)).to(sim.hx.dtype).cuda().requires_grad_()
    rec = torch.arange(10, device="cuda") * 9 + (n // 2) * g.ld + 20
    out = []
    for debug in (4, 0):
        cfg = autograd.TsunamiConfig(g, sim.tau, 40, rec, tuple(sim.ext), form=sim.form, ckpt_every=16, debug=debug)
        out.append(autograd.tsunami_traces(sim.hx, sim.hy, u0, None, cfg))
    with pytest.raises(tsu.TsuError) as err:
        autograd.sync_status(out[0])
    assert err.value.code == tsu.TSU_ETIMEOUT
    autograd.sync_status(out[0])  # read and cleared
    autograd.sync_status(out[1])
    assert torch.isfinite(out[1]).all()
    with pytest.raises(ValueError):
        autograd.sync_status(out[1].detach())


def test_studies(monkeypatch):
    step = tsu.Simulation.step
    monkeypatch.setattr(tsu.Simulation, "step", lambda self, n, **kw: step(self, n, debug=4, **kw))
    u0 = inputs.gaussian_hump(201, 201, None, 0.3, 0.5, 0.1)
    rec = np.array([[60, 100], [80, 120]])
    calls = [lambda: study.reflected_pulse(0.03, n=257, T=0.05)]
    calls += [lambda d=d: study.misfit_eps_gradient(201, DEPTH, u0, 40, rec, 0.06, dtype=d) for d in ("f64", "f32")]
    for call in calls:
        with pytest.raises(tsu.TsuError) as err:
            call()
        assert err.value.code == tsu.TSU_ETIMEOUT
