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
