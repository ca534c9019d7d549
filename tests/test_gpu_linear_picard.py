"""The elastic Picard predictor's polynomial form against the oracle's space-time iteration: any
number of iterations, both guesses, a point source, several cells per block at low order and a
cell count that leaves the last block partly empty."""
import numpy as np
import pytest
import torch

from cases import Case, rel_linf
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
