"""The work that users of this framework have it do, as a list of cases that can be timed.

Every case is a dict of plain values with a "kind":

- "forward":  one problem, ``Simulation.init`` (Taylor start) and ``steps - 1`` leapfrog steps, with the
  discrete energy of every step and / or receiver traces where the case asks for them.
- "family":   the eps-regularised family of problems of mixed sizes, started one by one and advanced
  together by ``batch_run``.
- "gradient": a receiver misfit J = 1/2 sum (traces - observed)^2 and its gradients in both face depths
  and the initial displacement, through the ``torch.autograd`` entry point (forward with traces and
  checkpoints, then the reverse sweep).
- "implicit": the implicit comparator of the paper's Table 1, ``init`` and ``steps - 1`` steps.

A pass always starts from the initial displacement, so it can be repeated on the same state.  The
sizes, depths and humps are those of ``inputs.py``, ``bench.py`` and the tests, with step counts cut
to what a timed pass can hold; the hump's place, the widths and the receivers come from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2005_11931_gb300 import autograd, inputs, tsu

CFL = 0.4
TYPES = {"f32": torch.float32, "f64": torch.float64}


# ---------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------
def listed():
    return [
        # the 201^2 FP64 parity run, whole: 1000 steps with the energy of every step (the smallest problem)
        dict(name="fwd64_201", kind="forward", nx=201, ny=201, dtype="f64", depth="line", steps=1000, energy=True,
             nrec=0),
        # FP64 reference solution of a mid-size problem (what FP32 runs are validated against)
        dict(name="fwd64_2048", kind="forward", nx=2048, ny=2048, dtype="f64", depth="point", steps=100, energy=True,
             nrec=0),
        # a small study grid of odd, ragged shape, as in interactive work and parameter studies
        dict(name="fwd32_ragged", kind="forward", nx=1003, ny=517, dtype="f32", depth="lines", steps=1000, energy=True,
             nrec=0),
        # reflected-pulse study: receivers between source and singularity, no energy
        dict(name="fwd32_769_rec", kind="forward", nx=769, ny=769, dtype="f32", depth="line", steps=800, energy=False,
             nrec=4),
        # mid-size production run
        dict(name="fwd32_2048", kind="forward", nx=2048, ny=2048, dtype="f32", depth="point", steps=1000, energy=True,
             nrec=0),
        # the headline workload: 8192^2 point singularity with the energy of every step
        dict(name="fwd32_8192", kind="forward", nx=8192, ny=8192, dtype="f32", depth="point", steps=500, energy=True,
             nrec=0),
        # the largest grid: 16384^2 crossing lines
        dict(name="fwd32_16384", kind="forward", nx=16384, ny=16384, dtype="f32", depth="lines", steps=200, energy=True,
             nrec=0),
        # the eps-family: 64 problems of 512^2 .. 2048^2 in one batched call
        dict(name="family_64", kind="family", count=64, nmin=512, nmax=2048, steps=500),
        # the 2048^2 gradient workload (128 receivers, a checkpoint every 64 steps)
        dict(name="grad32_2048", kind="gradient", nx=2048, ny=2048, dtype="f32", steps=1000, nrec=128, every=64),
        # an FP64 gradient of a small problem, as in gradient checks and small inversions
        dict(name="grad64_257", kind="gradient", nx=257, ny=257, dtype="f64", steps=300, nrec=32, every=32),
        # Table 1 of the paper, smallest and largest size (FP32), and a middle one in FP64
        dict(name="imp32_256", kind="implicit", nx=256, ny=256, dtype="f32", steps=100),
        dict(name="imp32_4096", kind="implicit", nx=4096, ny=4096, dtype="f32", steps=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: every kind, sizes spread over their logarithm, mostly odd."""
    kind = rng.choice(["forward"] * 5 + ["family", "gradient", "gradient", "implicit", "implicit"])
    dtype = rng.choice(["f32", "f32", "f32", "f64"])
    if kind == "forward":
        nx = _log_int(rng, 64, 16384 if dtype == "f32" else 2048)
        ny = max(64, min(16384 if dtype == "f32" else 2048, int(nx * rng.uniform(0.5, 1.5))))
        cap = 3.0e10 if dtype == "f32" else 4.0e8
        steps = _log_int(rng, 8, max(9, min(1000, int(cap / (nx * ny)))))
        nrec = rng.choice([0, 0, 1, _log_int(rng, 2, 200)])
        return dict(kind=kind, nx=nx, ny=ny, dtype=dtype, depth=rng.choice(["line", "point", "lines"]), steps=steps,
                    energy=rng.random() < 0.6, nrec=min(nrec, nx - 2))
    if kind == "family":
        nmin = _log_int(rng, 128, 600)
        count = _log_int(rng, 4, 64)
        return dict(kind=kind, count=count, nmin=nmin, nmax=int(nmin * rng.uniform(1.5, 3.4)),
                    steps=_log_int(rng, 40, 500))
    if kind == "gradient":
        nx = _log_int(rng, 100, 2048 if dtype == "f32" else 512)
        ny = max(64, int(nx * rng.uniform(0.6, 1.0)))
        return dict(kind=kind, nx=nx, ny=ny, dtype=dtype, steps=_log_int(rng, 30, 1000 if dtype == "f32" else 300),
                    nrec=_log_int(rng, 1, min(200, nx - 2)), every=rng.choice([16, 32, 64, rng.randint(5, 80)]))
    nx = _log_int(rng, 65, 4096 if dtype == "f32" else 1536)
    return dict(kind=kind, nx=nx, ny=max(65, int(nx * rng.uniform(0.6, 1.0))), dtype=dtype,
                steps=_log_int(rng, 8, 100))


# ---------------------------------------------------------------------------------------------
# what a case's seed decides, shared by prepare() and exact()
# ---------------------------------------------------------------------------------------------
def _rng(case, seed):
    return np.random.default_rng([seed, case.get("nx", case.get("count", 0)), case["steps"]])


def _depth(which, n, rng):
    """Depth descriptors of the repository's workloads, the width scaled by up to 30 %."""
    s = float(rng.uniform(0.85, 1.3))
    dx = 1.0 / (n - 1)
    if which == "line":
        return dict(background=1.0, eps=max(0.02 * s, 2 * dx), mollifier=inputs.GAUSS,
                    sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5)])
    if which == "point":
        return dict(background=0.5, eps=4 * dx * s, mollifier=inputs.GAUSS, sings=[(inputs.POINT, 1, 0.01, 0.5, 0.5)])
    return dict(background=1.0, eps=8 * dx * s, mollifier=inputs.GAUSS,
                sings=[(inputs.LINE_X, 1, 1.0, 0.5, 0.5), (inputs.LINE_Y, 1, 1.0, 0.5, 0.5)])


def _hump(rng, width):
    return float(rng.uniform(0.2, 0.8)), float(rng.uniform(0.2, 0.8)), width * float(rng.uniform(0.8, 1.2))


def _tau(nx, ny, depth):
    """Courant number CFL against the largest depth the descriptor can reach (Gaussian mollifiers)."""
    e = depth["eps"]
    top = depth["background"]
    for kind, power, amp, _, _ in depth["sings"]:
        top += amp * (1.0 / (math.pi * e * e) if kind == inputs.POINT else 1.0 / (e * math.sqrt(math.pi)))
    return CFL * min(1.0 / (nx - 1), 1.0 / (ny - 1)) / math.sqrt(top)


def _u0(nx, ny, ld, hump, dtype, amplitude=1.0):
    """The Gaussian hump at the nodes [ny][ld] on the GPU, computed in FP64, padding and edges 0."""
    x0, y0, w = hump
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") / (nx - 1) - x0) ** 2
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") / (ny - 1) - y0) ** 2
    out = torch.zeros((ny, ld), dtype=TYPES[dtype], device="cuda")
    out[1 : ny - 1, 1 : nx - 1] = (amplitude * torch.exp(-y / (w * w))[1:-1, None]
                                   * torch.exp(-x / (w * w))[None, 1:-1]).to(out.dtype)
    return out


def _ld(nx):
    return (nx + 31) // 32 * 32


def _receivers(case, rng, hump):
    """Receiver nodes on a row just above the hump, in the half of the columns around it, none twice."""
    nx, ny, m = case["nx"], case["ny"], case["nrec"]
    near = np.argsort(np.abs(np.arange(1, nx - 1) - hump[0] * (nx - 1)), kind="stable") + 1
    i = np.sort(rng.choice(near[: max(m, nx // 2)], size=m, replace=False)).astype(np.int64)
    return int(round((hump[1] + 0.03) * (ny - 1))) * _ld(nx) + i


def _observed(case, rng):
    """Observed pulses: one smooth bump of seeded arrival and height per receiver, [steps, nrec]."""
    S, n = case["steps"], case["nrec"]
    t = np.arange(1, S + 1)[:, None] / S
    return 0.2 * rng.uniform(-1, 1, n)[None, :] * np.exp(-((t - rng.uniform(0.2, 0.9, n)[None, :]) / 0.15) ** 2)


def _family_problems(case, seed):
    """Widths log-spaced in [1/512, 1/16], four singularity types, sizes drawn in [nmin, nmax]."""
    rng = _rng(case, seed)
    size_rng = np.random.default_rng(case["count"])  # the sizes belong to the case, not to the seed
    eps = np.logspace(math.log10(1 / 512), math.log10(1 / 16), max(2, (case["count"] + 3) // 4))
    sings = [[(inputs.LINE_X, 1, 1.0, 0.5, 0.5)], [(inputs.LINE_Y, 1, 1.0, 0.5, 0.5)],
             [(inputs.POINT, 1, 0.01, 0.5, 0.5)],
             [(inputs.LINE_X, 1, 1.0, 0.5, 0.5), (inputs.POINT, 1, 0.01, 0.5, 0.5)]]
    probs = []
    steps = [s for s in (512, 768, 1024, 1536, 2048) if case["nmin"] <= s <= case["nmax"]]
    for k in range(case["count"]):
        n = int(size_rng.choice(steps)) if len(steps) == 5 else int(size_rng.integers(case["nmin"], case["nmax"] + 1))
        depth = dict(background=1.0, eps=float(max(eps[k // 4] * rng.uniform(0.9, 1.1), 1.5 / n)),
                     mollifier=inputs.GAUSS, sings=sings[k % 4])
        probs.append((n, depth, _hump(rng, 0.03)))
    return probs


def _implicit_problem(case, seed):
    """Table 1: depth 100 left of the step, 10 right of it (Friedrichs, eps 0.008), tau = 5e-4 as the paper
    has it, with the hump (height 50) at a seeded place."""
    rng = _rng(case, seed)
    depth = dict(background=10.0, eps=0.8 / 100.0, mollifier=inputs.FRIEDRICHS, sings=[(inputs.STEP_X, 1, 90.0, 0.75, 0.5)])
    return depth, _hump(rng, math.sqrt(8) / 100), 0.05 / 100.0


# ---------------------------------------------------------------------------------------------
# preparation and one pass
# ---------------------------------------------------------------------------------------------
def prepare(case, seed):
    rng = _rng(case, seed)
    kind = case["kind"]
    if kind == "family":
        sims, u0s = [], []
        for n, depth, hump in _family_problems(case, seed):
            sims.append(tsu.Simulation.create(n, depth, dtype="f32", tau=_tau(n, n, depth)))
            u0s.append(_u0(n, n, sims[-1].g.ld, hump, "f32"))
        return dict(kind=kind, sims=sims, u0s=u0s, nsteps=[case["steps"] - 1] * len(sims))
    nx, ny, dtype, S = case["nx"], case["ny"], case["dtype"], case["steps"]
    if kind == "implicit":
        depth, hump, tau = _implicit_problem(case, seed)
        sim = tsu.ImplicitSimulation.create(nx, depth, dtype=dtype, ny=ny, tau=tau)
        return dict(kind=kind, sim=sim, u0=_u0(nx, ny, sim.g.ld, hump, dtype, 50.0), steps=S)
    if kind == "forward":
        depth = _depth(case["depth"], min(nx, ny), rng)
        hump = _hump(rng, 0.05 if max(nx, ny) < 512 else 0.02)
        sim = tsu.Simulation.create(nx, depth, dtype=dtype, ny=ny, tau=_tau(nx, ny, depth))
        st = dict(kind=kind, sim=sim, u0=_u0(nx, ny, sim.g.ld, hump, dtype), steps=S)
        if case["energy"]:
            st["energy"] = torch.zeros(S, dtype=torch.float64, device="cuda")
        if case["nrec"]:
            st["rec"] = torch.from_numpy(_receivers(case, rng, hump)).cuda()
            st["traces"] = torch.zeros((S, case["nrec"]), dtype=TYPES[dtype], device="cuda")
        return st
    depth = dict(background=1.0, eps=max(0.01 * float(rng.uniform(0.85, 1.3)), 1.5 / nx), mollifier=inputs.GAUSS,
                 sings=[(inputs.LINE_X, 1, 0.5, 0.5, 0.5)])
    hump = _hump(rng, 0.03 if nx >= 512 else 0.06)
    g = tsu.grid(nx, ny)
    hx, hy = tsu.empty_field(g, dtype), tsu.empty_field(g, dtype)
    ext = tsu.tsu_make_depth(g, depth, dtype, hx, hy, torch.zeros(4, dtype=torch.float64, device="cuda"))
    form = tsu.TSU_FORM_STANDARD if dtype == "f64" else tsu.TSU_FORM_INCREMENT
    cfg = autograd.TsunamiConfig(grid=g, tau=_tau(nx, ny, depth), steps=S, rec_idx=torch.from_numpy(_receivers(case, rng, hump)).cuda(),
                                 ext=tuple(ext), form=form, ckpt_every=case["every"])
    u0 = _u0(nx, ny, g.ld, hump, dtype)
    obs = torch.from_numpy(_observed(case, rng)).to(u0.dtype).cuda()
    return dict(kind=kind, cfg=cfg, hx=hx.requires_grad_(), hy=hy.requires_grad_(), u0=u0.requires_grad_(), obs=obs)


def run(st):
    kind = st["kind"]
    if kind == "family":
        for sim, u0 in zip(st["sims"], st["u0s"]):
            sim.init(u0)
        tsu.batch_run(st["sims"], st["nsteps"])
        return [sim.u for sim in st["sims"]]
    if kind == "implicit":
        sim = st["sim"]
        sim.init(st["u0"])
        sim.step(st["steps"] - 1)
        return dict(u=sim.u, v=sim.v)
    if kind == "gradient":
        traces = autograd.tsunami_traces(st["hx"], st["hy"], st["u0"], None, st["cfg"])
        misfit = 0.5 * ((traces - st["obs"]) ** 2).sum()
        g_hx, g_hy, g_u0 = torch.autograd.grad(misfit, (st["hx"], st["hy"], st["u0"]))
        return dict(misfit=misfit.detach(), traces=traces.detach(), g_hx=g_hx, g_hy=g_hy, g_u0=g_u0)
    sim, S, e, tr, rec = st["sim"], st["steps"], st.get("energy"), st.get("traces"), st.get("rec")
    sim.init(st["u0"])
    sim.step(S - 1, energy=None if e is None else e[: S - 1], rec_idx=rec, traces=None if tr is None else tr[: S - 1])
    if e is not None or tr is not None:
        sim.observe(energy=None if e is None else e[S - 1 :], rec_idx=rec, trace=None if tr is None else tr[S - 1])
    out = dict(u=sim.u, other=sim.v if sim.form == tsu.TSU_FORM_INCREMENT else sim.u_prev)
    if e is not None:
        out["energy"] = e
    if tr is not None:
        out["traces"] = tr
    return out


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def work(case):
    """Fields read and written once, and the scheme's own operations: per node and step 11 for the step
    (4 for the two face fluxes, 2 + 3 to combine them, 2 for the update), 5 more for the energy; 17 for a
    reverse step (9 for B lambda, 2 for the update, 6 for both face gradients); 21 for an implicit step
    (9 for B u, 5 for each line solve, 2 for the update)."""
    if case["kind"] == "family":
        nodes = sum(n * n for n, _, _ in _family_problems(case, 0))
        return {"bytes": 4 * 4 * nodes, "flops": 11 * nodes * case["steps"]}
    nodes, S, esz = case["nx"] * case["ny"], case["steps"], 4 if case["dtype"] == "f32" else 8
    if case["kind"] == "implicit":  # u0, both depths, three factor fields in; u, v out
        return {"bytes": 8 * esz * nodes, "flops": 21 * nodes * S}
    if case["kind"] == "gradient":  # u0, both depths, observations in; three gradients, traces out
        return {"bytes": 6 * esz * nodes + 2 * esz * S * case["nrec"], "flops": (11 + 17) * nodes * S}
    per = 11 + (5 if case["energy"] else 0)
    return {"bytes": 5 * esz * nodes + S * (8 * case["energy"] + esz * case["nrec"]), "flops": per * nodes * S}


# ---------------------------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------------------------
def _faces(nx, ny, depth, dtype):
    """Face depths hx [ny][nx - 1], hy [ny - 1][nx]: evaluated in FP64, rounded to the case's type."""
    dev = "cuda"
    xn = torch.arange(nx, dtype=torch.float64, device=dev) / (nx - 1)
    yn = torch.arange(ny, dtype=torch.float64, device=dev) / (ny - 1)
    xf, yf = xn[:-1] + 0.5 / (nx - 1), yn[:-1] + 0.5 / (ny - 1)
    e = depth["eps"]

    def at(x, y):
        h = torch.full((y.numel(), x.numel()), depth["background"], dtype=torch.float64, device=dev)
        for kind, power, amp, cx, cy in depth["sings"]:
            dx, dy = x - cx, y - cy
            if kind == inputs.LINE_X:
                h += (amp * torch.exp(-((dx / e) ** 2)) / (e * math.sqrt(math.pi)))[None, :]
            elif kind == inputs.LINE_Y:
                h += (amp * torch.exp(-((dy / e) ** 2)) / (e * math.sqrt(math.pi)))[:, None]
            elif kind == inputs.POINT:
                h += amp * torch.exp(-((dy / e) ** 2))[:, None] * torch.exp(-((dx / e) ** 2))[None, :] / (math.pi * e * e)
            else:  # the Friedrichs step in x: amp times the bump's mass left of (cx - x) / eps
                h += amp * torch.from_numpy(_bump_mass((-dx / e).cpu().numpy())).to(dev)[None, :]
        return h.to(TYPES[dtype]).double()

    return at(xf, yn), at(xn, yf)


def _bump_mass(s):
    """int_{-1}^{s} bump / int_{-1}^{1} bump, bump(t) = exp(1 / (t^2 - 1)), by Gauss-Legendre on 32 panels."""
    z, w = np.polynomial.legendre.leggauss(24)

    def integral(to):
        lo = np.full_like(to, -1.0)
        total = np.zeros_like(to)
        for p in range(32):
            a, b = lo + (to - lo) * p / 32, lo + (to - lo) * (p + 1) / 32
            t = 0.5 * (a + b)[:, None] + 0.5 * (b - a)[:, None] * z[None, :]
            q = t * t - 1.0
            f = np.where(q < -1e-12, np.exp(1.0 / np.minimum(q, -1e-12)), 0.0)
            total += 0.5 * (b - a) * (f * w[None, :]).sum(1)
        return total

    s = np.clip(np.asarray(s, dtype=np.float64), -1.0, 1.0)
    return integral(s) / integral(np.ones(1))


class _Plain:
    """u_tt = d_x(hx d_x u) + d_y(hy d_y u) on unpadded fields [ny][nx], edges 0."""

    def __init__(self, nx, ny, tau, hx, hy):
        self.nx, self.ny, self.tau, self.hx, self.hy = nx, ny, tau, hx, hy
        self.cx, self.cy = (tau * (nx - 1)) ** 2, (tau * (ny - 1)) ** 2

    def b(self, u):
        fx = self.hx[1:-1] * (u[1:-1, 1:] - u[1:-1, :-1])
        fy = self.hy[:, 1:-1] * (u[1:, 1:-1] - u[:-1, 1:-1])
        out = torch.zeros_like(u)
        out[1:-1, 1:-1] = self.cx * (fx[:, 1:] - fx[:, :-1]) + self.cy * (fy[1:] - fy[:-1])
        return out

    def start(self, u0):
        v = 0.5 * self.b(u0)
        return u0 + v, v

    def energy(self, u, v, bu):
        """E^{n-1/2} of (u^n, v^n = u^n - u^{n-1}), bu = B u^n."""
        return ((v * v).sum() - (bu * (u - v)).sum()) / ((self.nx - 1) * (self.ny - 1) * 2.0 * self.tau ** 2)


def _padded(u, nx, ny):
    out = torch.zeros((ny, _ld(nx)), dtype=torch.float64, device=u.device)
    out[: u.shape[0], : u.shape[1]] = u
    return out


def _plain_forward(nx, ny, tau, hx, hy, u0, S, energy=False, rec=None):
    p = _Plain(nx, ny, tau, hx, hy)
    u, v = p.start(u0)
    es, tr = [], []
    ij = None if rec is None else (rec // _ld(nx), rec % _ld(nx))
    for n in range(1, S + 1):  # u = u^n
        if ij is not None:
            tr.append(u[ij])
        if n < S or energy:
            bu = p.b(u)
        if energy:
            es.append(p.energy(u, v, bu))
        if n < S:
            v = v + bu
            u = u + v
    return u, v, torch.stack(es) if energy else None, torch.stack(tr) if ij is not None else None


def _plain_gradient(nx, ny, tau, hx, hy, u0, S, rec, obs):
    """The discrete adjoint, states recomputed from a checkpoint every 100 steps."""
    p = _Plain(nx, ny, tau, hx, hy)
    i, j = rec % _ld(nx), rec // _ld(nx)
    every = 100
    u, v = p.start(u0)
    saved, tr = {}, []
    for n in range(1, S + 1):
        if (n - 1) % every == 0:
            saved[n] = (u, v)
        tr.append(u[j, i])
        if n < S:
            v = v + p.b(u)
            u = u + v
    tr = torch.stack(tr)
    res = tr - obs
    gx, gy = torch.zeros_like(hx), torch.zeros_like(hy)
    lam, lam1 = torch.zeros_like(u0), torch.zeros_like(u0)  # lam^{n+1}, lam^{n+2}
    states, lo = [], S + 1
    for n in range(S, 0, -1):
        if n < lo:
            lo = (n - 1) // every * every + 1
            states = [saved[lo]]
            for _ in range(n - lo):
                u, v = states[-1]
                v = v + p.b(u)
                states.append((u + v, v))
        un = states[n - lo][0]
        gx -= p.cx * (lam[:, 1:] - lam[:, :-1]) * (un[:, 1:] - un[:, :-1])
        gy -= p.cy * (lam[1:] - lam[:-1]) * (un[1:] - un[:-1])
        new = 2.0 * lam + p.b(lam) - lam1
        new.index_put_((j, i), res[n - 1], accumulate=True)
        lam, lam1 = new, lam
    gx -= 0.5 * p.cx * (lam[:, 1:] - lam[:, :-1]) * (u0[:, 1:] - u0[:, :-1])
    gy -= 0.5 * p.cy * (lam[1:] - lam[:-1]) * (u0[1:] - u0[:-1])
    gu0 = lam - lam1 + 0.5 * p.b(lam)
    return 0.5 * (res * res).sum(), tr, gx, gy, gu0


def _plain_implicit(nx, ny, tau, hx, hy, u0, S, sigma=0.25):
    """(I - s B_x)(I - s B_y) w = B u with a depth that varies in x only: the x systems are one matrix
    for all rows, and the y systems are diagonal in the discrete sine basis."""
    p = _Plain(nx, ny, tau, hx, hy)
    m, h = nx - 2, hx[0]
    a = torch.diag(1.0 + sigma * p.cx * (h[:-1] + h[1:]))
    k = torch.arange(m - 1, device=a.device)
    a[k, k + 1] = a[k + 1, k] = -sigma * p.cx * h[1:-1]
    inv = torch.linalg.inv(a)
    l = torch.arange(1, ny - 1, dtype=torch.float64, device=a.device)
    sine = torch.sin(math.pi / (ny - 1) * torch.remainder(l[:, None] * l[None, :], 2 * (ny - 1))) * math.sqrt(2.0 / (ny - 1))
    eig = 1.0 + sigma * p.cy * 4.0 * torch.sin(0.5 * math.pi * l / (ny - 1))[:, None] ** 2 * hy[0, 1:-1][None, :]

    def solve(u):
        z = p.b(u)[1:-1, 1:-1] @ inv.T
        w = torch.zeros_like(u)
        w[1:-1, 1:-1] = sine @ ((sine @ z) / eig)
        return w

    v = 0.5 * solve(u0)
    u = u0 + v
    for _ in range(S - 1):
        v = v + solve(u)
        u = u + v
    return u, v


def exact(case, seed):
    kind = case["kind"]
    if kind == "family":
        out = []
        for n, depth, hump in _family_problems(case, seed):
            hx, hy = _faces(n, n, depth, "f32")
            u0 = _u0(n, n, n, hump, "f32").double()
            out.append(_padded(_plain_forward(n, n, _tau(n, n, depth), hx, hy, u0, case["steps"])[0], n, n))
        return out
    nx, ny, dtype, S = case["nx"], case["ny"], case["dtype"], case["steps"]
    rng = _rng(case, seed)
    if kind == "implicit":
        if nx * ny * nx * S > 9e11:  # dense solves: up to about 2048^2
            return None
        depth, hump, tau = _implicit_problem(case, seed)
        hx, hy = _faces(nx, ny, depth, dtype)
        u, v = _plain_implicit(nx, ny, tau, hx, hy, _u0(nx, ny, nx, hump, dtype, 50.0).double(), S)
        return dict(u=_padded(u, nx, ny), v=_padded(v, nx, ny))
    if kind == "forward":
        depth = _depth(case["depth"], min(nx, ny), rng)
        hump = _hump(rng, 0.05 if max(nx, ny) < 512 else 0.02)
        rec = torch.from_numpy(_receivers(case, rng, hump)).cuda() if case["nrec"] else None
        hx, hy = _faces(nx, ny, depth, dtype)
        u, v, e, tr = _plain_forward(nx, ny, _tau(nx, ny, depth), hx, hy, _u0(nx, ny, nx, hump, dtype).double(), S,
                                     case["energy"], rec)
        out = dict(u=_padded(u, nx, ny), other=_padded(v if dtype == "f32" else u - v, nx, ny))
        if e is not None:
            out["energy"] = e
        if tr is not None:
            out["traces"] = tr
        return out
    depth = dict(background=1.0, eps=max(0.01 * float(rng.uniform(0.85, 1.3)), 1.5 / nx), mollifier=inputs.GAUSS,
                 sings=[(inputs.LINE_X, 1, 0.5, 0.5, 0.5)])
    hump = _hump(rng, 0.03 if nx >= 512 else 0.06)
    rec = torch.from_numpy(_receivers(case, rng, hump)).cuda()
    obs = torch.from_numpy(_observed(case, rng)).to(TYPES[dtype]).double().cuda()
    hx, hy = _faces(nx, ny, depth, dtype)
    j, tr, gx, gy, gu0 = _plain_gradient(nx, ny, _tau(nx, ny, depth), hx, hy, _u0(nx, ny, nx, hump, dtype).double(), S,
                                         rec, obs)
    return dict(misfit=j, traces=tr, g_hx=_padded(gx, nx, ny), g_hy=_padded(gy, nx, ny), g_u0=_padded(gu0, nx, ny))
