"""The FP64 predictor's integer contractions against the oracle: every order, one and several
iterations, both guesses, and the states that leave its scale and are recomputed by the FP64 form
(magnitudes outside binary32, a flux that grows past the room, non-finite values)."""
import numpy as np
import pytest
import torch

from cases import Case, rel_linf
from paper_1905_07987_gb300 import synth

pytestmark = pytest.mark.gpu


def smooth_state(c, scale=1.0, speed=1.0):
    """Euler / shallow water data with every term active; rho and E scaled by `scale`, velocities
    by `speed` (pressure by scale * speed^2)."""
    X = c.X
    s = sum(X)
    f = [0.3 * np.sin(2 * np.pi * (s + 0.37 * i)) for i in range(c.ctx.nvar)]
    if c.pde == "swe":
        h = 1.0 + 0.1 * f[0]
        return np.stack([h, 0.4 * h * (1 + f[1]), -0.3 * h * (1 + f[2]), 0.2 + 0.1 * f[3]], axis=-1)
    rho = scale * (1.0 + f[0])
    vel = [speed * (0.5 - 0.4 * d + f[1 + d]) for d in range(c.dim)]
    p = scale * speed ** 2 * (1.0 + f[-1])
    return np.stack([rho] + [rho * v for v in vel] + [p / 0.4 + 0.5 * rho * sum(v * v for v in vel)], axis=-1)


def step(c, u, dt=None):
    c.set(u)
    dt = float(c.oracle.cfl_dt(torch.from_numpy(u))) if dt is None else dt
    c.ctx.step(dt)
    return c.get(), c.oracle_step(u, dt)


@pytest.mark.parametrize("order", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("pde,dim", [("euler", 2), ("euler", 3), ("swe", 2)])
def test_orders(pde, dim, order):
    nc = (3, 2, 2)[:dim]
    c = Case(pde, dim, order, nc, hi=(1.3, 0.7, 1.0)[:dim], bc="absorbing")
    out, ref = step(c, smooth_state(c))
    assert rel_linf(out, ref) < 1e-12


@pytest.mark.parametrize("guess,iters", [("constant", 1), ("constant", 2), ("cerk", 1), ("cerk", 3)])
def test_iterations(guess, iters):
    c = Case("euler", 3, 3, (2, 3, 2), picard_iters=iters, initial_guess=guess)
    out, ref = step(c, smooth_state(c))
    assert rel_linf(out, ref) < 1e-12


# 1e-60 and 1e60: outside binary32; 1e-3 and 1e4: far apart scales of the variables
@pytest.mark.parametrize("scale,speed", [(1e-60, 1.0), (1e60, 1.0), (1.0, 1e-3), (1e4, 340.0)])
def test_magnitudes(scale, speed):
    c = Case("euler", 2, 4, (3, 2))
    out, ref = step(c, smooth_state(c, scale, speed))
    assert rel_linf(out, ref) < 1e-12


def test_flux_past_the_room():
    # a step far above the stability limit: the iterates, and their fluxes, grow by more than the
    # room left for them
    c = Case("euler", 2, 3, (4, 3))
    u = smooth_state(c)
    out, ref = step(c, u, 40.0 * float(c.oracle.cfl_dt(torch.from_numpy(u))))
    assert np.abs(ref).max() > 1e4 * np.abs(u).max()
    assert np.abs(out - ref).max() < 1e-9 * np.abs(ref).max()


def test_non_finite():
    # the cells that hold them stay non-finite; cells that share no face with one are unaffected
    c = Case("euler", 2, 2, (5, 5), bc="absorbing", picard_iters=1)
    u = smooth_state(c)
    u[12, 1, 1, 0] = np.nan
    u[0, 0, 0, 3] = np.inf
    out, ref = step(c, u, 1e-3)
    far = [k for k in range(25) if min(abs(k % 5 - b % 5) + abs(k // 5 - b // 5) for b in (0, 12)) > 1]
    assert rel_linf(out[far], ref[far]) < 1e-12
    assert not np.isfinite(out[12]).all() and not np.isfinite(out[0]).all()


# the mixed elastic predictor: its lowest order in fixed point, the largest, odd and even numbers of
# nodes; a block that is part full; 30 stable steps: levels past the room, the block in the node form
@pytest.mark.parametrize("predictor", ["picard", "ck"])
@pytest.mark.parametrize("order,stretch", [(3, 1), (4, 1), (5, 1), (6, 1), (4, 30), (5, 30)])
def test_mixed_elastic(order, stretch, predictor):
    nc = (3, 3, 3)
    c = Case("elastic", 3, order, nc, hi=(1.3, 0.7, 1.0), predictor=predictor, precision="mixed",
             material=synth.elastic_material(nc, seed=order))
    s = sum(c.X)
    # stresses of the size of the impedance times the velocities
    u = np.stack([(3.0 if i >= 3 else 1.0) * np.sin(2 * np.pi * (s + 0.37 * i)) for i in range(9)], axis=-1)
    dt = stretch * float(c.oracle.cfl_dt(torch.from_numpy(u)))
    c.set(u)
    c.ctx.step(dt)
    ref = c.oracle_step(u, dt)
    # the levels after the first carry binary32's rounding, 2^-24 each operation
    assert np.abs(c.get() - ref).max() < 2e-6 * np.abs(ref - u).max()
