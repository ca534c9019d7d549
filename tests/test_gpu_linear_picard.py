"""The elastic Picard predictor's polynomial form against the oracle's space-time iteration: any
number of iterations, both guesses, a point source, several cells per block at low order and a
cell count that leaves the last block partly empty."""
import numpy as np
import pytest
import torch

from cases import Case, rel_linf
from oracle.adjoint import step_vjp
from paper_1905_07987_gb300 import synth

pytestmark = pytest.mark.gpu


def run(order, iters, guess, precision, bc="absorbing"):
    nc = (3, 3, 1) if order < 5 else (2, 1, 2)
    mat = synth.elastic_material(nc, seed=order)
    c = Case("elastic", 3, order, nc, hi=tuple(0.5 * k for k in nc), bc=bc, material=mat,
             picard_iters=iters, initial_guess=guess, precision=precision)
    c.point_source([0.7, 0.2, 0.3], synth.moment_tensor(5) * 1e-2, 2.0, 0.02)
    u = np.random.default_rng(7).standard_normal(c.shape)
    c.set(u)
    dt = float(c.oracle.cfl_dt(torch.from_numpy(u)))
    c.ctx.step(dt)
    out, ref = c.get(), c.oracle_step(u, dt)
    return out, ref, u


@pytest.mark.parametrize("guess", ["constant", "cerk"])
@pytest.mark.parametrize("order,iters", [(1, 0), (1, 5), (2, 1), (3, 2), (3, 7), (4, 0), (5, 3), (6, 0)])
def test_fp64(order, iters, guess):
    out, ref, _ = run(order, iters, guess, "fp64", "periodic" if order % 2 else "absorbing")
    assert rel_linf(out, ref) < 1e-12


@pytest.mark.parametrize("guess", ["constant", "cerk"])
@pytest.mark.parametrize("order,iters", [(1, 1), (2, 4), (4, 1), (5, 0), (6, 2)])
def test_mixed(order, iters, guess):
    out, ref, u = run(order, iters, guess, "mixed")
    assert np.abs(out - ref).max() < 2e-6 * np.abs(ref - u).max()


# iterations enough for the last weights to leave the range: the levels end before
@pytest.mark.parametrize("guess", ["constant", "cerk"])
@pytest.mark.parametrize("iters", [1021, 1024, 1025, 1100])
def test_many_iterations(iters, guess):
    out, ref, _ = run(1, iters, guess, "fp64")
    assert rel_linf(out, ref) < 1e-12


def device(a):
    return torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).cuda()


def adjoint(c, u, lam, dt, t, static):
    lam_d = device(lam)
    gm = torch.zeros(c.ctx.cells * 3, dtype=torch.float64, device="cuda")
    gM = torch.zeros(6, dtype=torch.float64, device="cuda")
    c.ctx.adjoint_step(t, dt, device(u), lam_d, gm, gM, static=static)
    c.ctx.sync()
    return lam_d.cpu().numpy(), gm.cpu().numpy(), gM.cpu().numpy()


def close(a, b):
    return np.abs(a - b).max() <= 1e-12 * np.abs(b).max()


# 40 iterations: more levels than fit, the adjoint that keeps the iterates
@pytest.mark.parametrize("static", [False, True])
@pytest.mark.parametrize("order,iters", [(1, 1), (1, 4), (2, 7), (3, 1), (4, 3), (5, 6), (2, 40)])
def test_adjoint(order, iters, static):
    nc = (3, 3, 1) if order < 4 else (2, 1, 2)
    mat = synth.elastic_material(nc, seed=order)
    c = Case("elastic", 3, order, nc, hi=tuple(0.5 * k for k in nc), bc="absorbing", material=mat,
             picard_iters=iters)
    c.point_source([0.7, 0.2, 0.3], synth.moment_tensor(5), 2.0, 0.4)
    rng = np.random.default_rng(order)
    u, lam = rng.standard_normal(c.shape), rng.standard_normal(c.shape)
    dt = 0.7 * float(c.oracle.cfl_dt(torch.from_numpy(u)))
    ref = step_vjp(c.oracle, torch.from_numpy(u), torch.from_numpy(lam), dt, 0.35)
    out = adjoint(c, u, lam, dt, 0.35, static)
    for a, b in zip(out, ref):
        assert close(a, b.numpy().reshape(-1))


def test_adjoint_static_beyond_the_projections():
    # 16 x 16 x 16 cells at order 4: the projections do not fit the fixed array, the iterate slabs do
    nc = (16, 16, 16)
    mat = synth.elastic_material(nc, seed=2)
    c = Case("elastic", 3, 4, nc, hi=(8.0,) * 3, bc="periodic", material=mat)
    rng = np.random.default_rng(1)
    u, lam = rng.standard_normal(c.shape), rng.standard_normal(c.shape)
    a, b = (adjoint(c, u, lam, 1e-3, 0.0, s) for s in (False, True))
    assert close(a[0], b[0]) and close(a[1], b[1])
