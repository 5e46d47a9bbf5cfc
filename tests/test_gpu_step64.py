"""FP64 steps and reverse steps (k_step64.cu: tiles of 31 columns, a warp each) against the oracle, at
sizes around the tile edges: one column more or less than whole strips, the smallest grids, few and
many rows, rows per tile chosen by the caller.  1e-12 relative, the FP64 tolerance of the other parity
tests (a few hundred roundings of 1.1e-16 per node over 40 steps)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2005_11931_gb300 import inputs, tsu
from tests.gpu_helpers import relerr, run_gpu, run_oracle
from tests.test_gpu_adjoint import gpu_forward_adjoint

pytestmark = pytest.mark.gpu
DEPTH = dict(background=1.0, eps=0.06, mollifier=0, sings=[(0, 1, 0.5, 0.5, 0.5), (2, 1, 0.002, 0.4, 0.6)])
SIZES = [(3, 3), (3, 40), (40, 3), (31, 9), (32, 33), (33, 8), (62, 37), (63, 5), (64, 64), (94, 30), (125, 257),
         (400, 61)]


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("form", [tsu.TSU_FORM_STANDARD, tsu.TSU_FORM_INCREMENT])
@pytest.mark.parametrize("kernel,rows", [(1, 0), (1, 5), (0, 0)])
def test_forward(nx, ny, form, kernel, rows):
    S = 40
    rng = np.random.default_rng(nx * 1009 + ny)
    u0 = inputs.random_field(nx, ny, None, rng)
    rec = np.array([[1, 1], [nx - 2, ny - 2], [nx // 2, ny // 2], [nx // 2, ny // 2], [0, ny // 2]])
    gpu = run_gpu(nx, DEPTH, u0, S, dtype="f64", form=form, ny=ny, rec_ij=rec, rows=rows, kernel=kernel)
    ref = run_oracle(nx, DEPTH, u0, S, ny=ny, rec_ij=rec, tau=gpu["tau"])
    assert relerr(gpu["u"], ref["u"]) <= 1e-12
    assert relerr(gpu["traces"], ref["traces"]) <= 1e-12
    assert np.max(np.abs(gpu["energy"] - ref["energy"]) / ref["energy"]) <= 1e-12


@pytest.mark.parametrize("nx,ny", SIZES)
def test_adjoint(nx, ny):
    S, every = 40, 7
    rng = np.random.default_rng(nx * 1009 + ny)
    u0, u1 = inputs.random_field(nx, ny, None, rng), inputs.random_field(nx, ny, None, rng)
    rec = np.array([[1, 1], [nx - 2, ny - 2], [nx // 2, ny // 2], [nx // 2, ny // 2], [0, ny // 2]])
    dtr = rng.standard_normal((S, len(rec)))
    out, tau = gpu_forward_adjoint(nx, ny, DEPTH, u0, u1, S, rec, dtr, "f64", tsu.TSU_FORM_STANDARD, every)
    g = oracle.grid(nx, ny)
    hx, hy, _ = oracle.make_depth(g, DEPTH)
    ref = oracle.adjoint(g, tau, hx, hy, u0[:, :nx], u1[:, :nx], S, inputs.flat_index(rec, g.ld), dtr)
    for k in ("g_hx", "g_hy", "g_u0", "g_u1"):
        assert relerr(out[k], ref[k][:, :nx]) <= 1e-12, k


def test_many_receivers():
    """More receivers than a bucket count, several on one node: injected in receiver order."""
    nx, ny, S = 97, 90, 12
    rng = np.random.default_rng(5)
    u0, u1 = inputs.random_field(nx, ny, None, rng), inputs.random_field(nx, ny, None, rng)
    rec = np.stack([rng.integers(0, nx, 1500), rng.integers(0, ny, 1500)], 1)
    dtr = rng.standard_normal((S, len(rec)))
    out, tau = gpu_forward_adjoint(nx, ny, DEPTH, u0, u1, S, rec, dtr, "f64", tsu.TSU_FORM_STANDARD, 5)
    g = oracle.grid(nx, ny)
    hx, hy, _ = oracle.make_depth(g, DEPTH)
    ref = oracle.adjoint(g, tau, hx, hy, u0[:, :nx], u1[:, :nx], S, inputs.flat_index(rec, g.ld), dtr)
    for k in ("g_hx", "g_hy", "g_u0", "g_u1"):
        assert relerr(out[k], ref[k][:, :nx]) <= 1e-12, k
