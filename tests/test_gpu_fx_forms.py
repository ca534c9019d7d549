"""The fixed-point form and the FP64 form of a predictor on the same data.  Scaled by powers of two that
leave the fixed-point range, the data take the FP64 form, whose results scale exactly (every
operation of the step does): bits that differ from it show that the fixed-point form was taken, bits
that agree that it was not, and the difference is the two forms' rounding."""
import numpy as np
import pytest
import torch

from cases import Case, rel_linf

pytestmark = pytest.mark.gpu


def step(c, u, dt):
    c.set(u)
    c.ctx.step(dt)
    return c.get()


def swe_fp64_form(c, u, dt, m=60):
    """h, b scale as 2^(2 m), momenta as 2^(3 m), times as 2^-m (g and the grid stay)."""
    e = np.array([2 * m, 3 * m, 3 * m, 2 * m])
    return np.ldexp(step(c, np.ldexp(u, e), np.ldexp(dt, -m)), -e)


def swe_state(c, kind):
    x, y = (2 * np.pi * a for a in c.X)
    depth = 1.0 + 0.3 * np.sin(x) * np.cos(y)
    eta = {"datum": 0.0 * x, "wave": 1e-3 * np.sin(x + y), "residue": 1e-16 * np.sin(5 * x),
           "high": 2.0 + 0.1 * np.sin(y)}[kind]
    h = depth + eta
    return np.stack([h, 0.2 * h * np.cos(x), -0.1 * h * np.sin(y), -depth], axis=-1)


# a surface at the datum (h + b = 0 where the water moves), near it, and above it
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("kind", ["datum", "wave", "residue", "high"])
def test_shallow_water_surface(order, kind):
    c = Case("swe", 2, order, (3, 2), hi=(1.3, 0.7))
    u = swe_state(c, kind)
    dt = float(c.oracle.cfl_dt(torch.from_numpy(u)))
    out, ref = step(c, u, dt), c.oracle_step(u, dt)
    assert rel_linf(out, ref) < 1e-12
    fp64 = swe_fp64_form(c, u, dt)
    assert all((out[k] != fp64[k]).any() for k in range(c.ctx.cells))


# The forms round the last iterate, the time averages, the volume sum and the corrector differently: four
# sums of at most 21 products of at most half the scale, each rounded at 2^-53 (FP64; the fixed-point form
# less): about 4 sqrt(21) / 2 / 2 = 5 units as a random walk, 32 for the largest of all values.  A
# fixed-point form that lost ten of its bits would be off by 64.
ROUNDING = 32 * 2.0 ** -53


def euler_state(c):
    f = [0.3 * np.sin(2 * np.pi * (sum(c.X) + 0.37 * i)) for i in range(c.ctx.nvar)]
    rho = 1.0 + f[0]
    vel = [0.5 - 0.4 * d + f[1 + d] for d in range(c.dim)]
    p = 1.0 + f[-1]
    s = np.abs(np.array(vel)).sum(axis=0).max() + np.sqrt(1.4 * p / rho).max()
    u = np.stack([rho] + [rho * v for v in vel] + [2.5 * p + 0.5 * rho * sum(v * v for v in vel)], axis=-1)
    return u, [rho.max()] + [rho.max() * s] * c.dim + [(u[..., -1] + p).max()]


@pytest.mark.parametrize("dim,order,guess", [(2, n, "constant") for n in range(1, 7)] +
                         [(3, n, "constant") for n in range(1, 6)] + [(2, 4, "cerk"), (3, 3, "cerk")])
def test_euler(dim, order, guess):
    c = Case("euler", dim, order, (3, 2, 2)[:dim], hi=(1.3, 0.7, 1.0)[:dim], initial_guess=guess)
    u, scale = euler_state(c)
    dt = float(c.oracle.cfl_dt(torch.from_numpy(u)))
    out = step(c, u, dt)
    fp64 = np.ldexp(step(c, np.ldexp(u, 120), dt), -120)
    assert all((out[k] != fp64[k]).any() for k in range(c.ctx.cells))
    assert (np.abs(out - fp64) <= ROUNDING * np.array(scale)).all()


@pytest.mark.parametrize("order", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("kind", ["wave", "high"])
def test_shallow_water(order, kind):
    c = Case("swe", 2, order, (3, 2), hi=(1.3, 0.7), bc="absorbing")
    u = swe_state(c, kind)
    h = u[..., 0]
    s = (np.abs(u[..., 1:3] / h[..., None]).sum(axis=-1) + np.sqrt(9.81 * h)).max()
    dt = float(c.oracle.cfl_dt(torch.from_numpy(u)))
    out, fp64 = step(c, u, dt), swe_fp64_form(c, u, dt)
    assert all((out[k] != fp64[k]).any() for k in range(c.ctx.cells))
    top = max(h.max(), np.abs(h + u[..., 3]).max())
    assert (np.abs(out - fp64) <= ROUNDING * np.array([top, top * s, top * s, top])).all()


# magnitudes outside the fixed-point range
def test_shallow_water_in_fp64():
    c = Case("swe", 2, 3, (4, 3))
    u = swe_state(c, "high")
    dt = float(c.oracle.cfl_dt(torch.from_numpy(u)))
    assert rel_linf(swe_fp64_form(c, u, dt), c.oracle_step(u, dt)) < 1e-12


# rough data and several stable steps: the iterates, and their fluxes, leave the range on the way
def test_shallow_water_past_the_room():
    c = Case("swe", 2, 3, (4, 3))
    r = np.random.default_rng(3)
    h = 3.0 * (1.0 + 0.2 * r.uniform(-1, 1, c.shape[:-1]))
    b = -1.0 + 0.2 * r.uniform(-1, 1, h.shape)
    u = np.stack([h, 0.2 * h * r.uniform(-1, 1, h.shape), -0.1 * h * r.uniform(-1, 1, h.shape), b], axis=-1)
    dt = 8.0 * float(c.oracle.cfl_dt(torch.from_numpy(u)))
    out, ref = step(c, u, dt), c.oracle_step(u, dt)
    assert np.isfinite(ref).all() and np.abs(ref).max() > 1e3 * np.abs(u).max()
    assert np.abs(out - ref).max() < 1e-9 * np.abs(ref).max()


def elastic_case(order, predictor, precision="fp64"):
    # 18 cells: the last block of 16 (order 1) or 4 (order 2) is part full; the impedance is 2
    mat = np.tile(np.array([1.0, 2.0, 1.0]), (18, 1))
    return Case("elastic", 3, order, (3, 3, 2), hi=(1.5, 1.5, 1.0), bc="absorbing", predictor=predictor,
                precision=precision, material=mat)


def elastic_state(c, rough):
    """Stresses twice the velocities.  Rough: signs that alternate from node to node, mirrored in each
    direction, just below a power of two: the levels pass the room above it.  Smooth: values above a
    power of two, with a factor of two of room."""
    u = np.empty(c.shape)
    n = c.order + 1
    k = np.arange(n)
    alt = np.where(np.minimum(k, n - 1 - k) % 2, -1.0, 1.0)
    odd = alt * np.sign(n - 1 - 2 * k)
    for v in range(9):
        a = alt if v % 2 else odd
        f = 0.995 * a[:, None, None] * a[:, None] * a if rough else 0.505 * np.sin(0.6 * sum(c.X) + 2.3 * v)
        u[..., v] = f * (2.0 if v >= 3 else 1.0)
    return u


STRETCH = {1: 3.5, 2: 2.5, 3: 2.0, 4: 2.0, 5: 2.0, 6: 1.5}  # of the stable step: the coefficients still fit


@pytest.mark.parametrize("predictor", ["picard", "ck"])
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5, 6])
def test_elastic(order, predictor):
    c = elastic_case(order, predictor)
    u = elastic_state(c, False)
    dt = STRETCH[order] * float(c.oracle.cfl_dt(torch.from_numpy(u)))
    out = step(c, u, dt)
    fp64 = np.ldexp(step(c, np.ldexp(u, 900), dt), -900)
    assert all((out[k] != fp64[k]).any() for k in range(c.ctx.cells))
    assert (np.abs(out - fp64) <= ROUNDING * np.array([1.0] * 3 + [2.0] * 6)).all()
    # small enough for the corrector (fixed point from order 3) to take its FP64 form as well
    low = np.ldexp(step(c, np.ldexp(u, -850), dt), 850)
    assert (np.abs(out - low) <= ROUNDING * np.array([1.0] * 3 + [2.0] * 6)).all()
    assert np.array_equal(low, fp64) == (order < 3)


@pytest.mark.parametrize("predictor", ["picard", "ck"])
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5, 6])
def test_elastic_levels_past_the_room(order, predictor):
    c = elastic_case(order, predictor)
    u = elastic_state(c, True)
    dt = STRETCH[order] * float(c.oracle.cfl_dt(torch.from_numpy(u)))
    out = step(c, u, dt)
    assert np.array_equal(out, np.ldexp(step(c, np.ldexp(u, 900), dt), -900))
    assert rel_linf(out, c.oracle_step(u, dt)) < 1e-12


@pytest.mark.parametrize("predictor,order", [("picard", 4), ("picard", 5), ("picard", 6), ("ck", 5), ("ck", 6)])
def test_mixed_elastic_levels_past_the_room(order, predictor):
    c = elastic_case(order, predictor, "mixed")
    u = elastic_state(c, True)
    dt = STRETCH[order] * float(c.oracle.cfl_dt(torch.from_numpy(u)))
    out, ref = step(c, u, dt), c.oracle_step(u, dt)
    # the levels after the first carry binary32's rounding, 2^-24 each operation
    assert np.abs(out - ref).max() < 2e-6 * np.abs(ref - u).max()
