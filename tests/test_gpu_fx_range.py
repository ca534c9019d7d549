"""States near the ends of binary64's range: what the fixed-point forms leave to the FP64 forms."""
import numpy as np
import pytest
import torch

from cases import Case, rel_linf
from oracle.limiter import Limiter
from paper_1905_07987_gb300 import ader, synth

pytestmark = pytest.mark.gpu


def layered(shape, order):
    """Elastic data constant in each cell (no volume term), every component of the size of 1."""
    u = np.random.default_rng(order).uniform(0.5, 1.0, (shape[0], 1, 1, 1, 9))
    return np.broadcast_to(u * np.random.default_rng(7).choice([-1.0, 1.0], u.shape), shape).copy()


# dt = 8, far above the stable one: the face terms are some 60 times the fluxes
@pytest.mark.parametrize("order", [3, 4, 5, 6])
@pytest.mark.parametrize("exponent", [900, 1000, 1016])
def test_corrector_at_the_upper_end(order, exponent):
    nc = (3, 2, 2)
    mat = np.tile(np.array([1.0, 1.0, 1.0]), (12, 1))
    c = Case("elastic", 3, order, nc, hi=(1.5, 1.0, 1.0), bc="absorbing", material=mat, picard_iters=1)
    u = layered(c.shape, order)
    ref = c.oracle_step(u, 8.0)  # the step is linear: the result of u 2^exponent is ref 2^exponent
    c.set(np.ldexp(u, exponent))
    c.ctx.step(8.0)
    out = c.get()
    big = np.abs(ref) >= 2.0 ** (1024 - exponent)
    assert not np.isfinite(out[big]).any()
    if exponent < 1016:
        assert rel_linf(np.ldexp(out, -exponent), ref) < 1e-12
    else:
        assert big.any()
        with pytest.raises(ader.AderError) as e:
            c.ctx.sync()
        assert e.value.status == ader.ENONFINITE


def smooth(c, seed):
    s = sum(c.X)
    u = np.stack([np.sin(2 * np.pi * (s + 0.37 * i)) for i in range(9)], axis=-1)
    u[..., 4] = 0.0  # a component of zeros
    u[3] = 0.0       # and a quiet cell
    return u


# all values below the fixed-point forms' smallest scale: as exact as any others
@pytest.mark.parametrize("predictor", ["picard", "ck"])
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("exponent", [-600, -780, -860, -950])
def test_elastic_at_the_lower_end(order, exponent, predictor):
    nc = (3, 2, 2)
    c = Case("elastic", 3, order, nc, hi=(1.5, 1.0, 1.0), bc="absorbing", predictor=predictor,
             material=synth.elastic_material(nc, seed=order))
    u = smooth(c, order)
    dt = float(c.oracle.cfl_dt(torch.from_numpy(u)))
    ref = c.oracle_step(u, dt)
    c.set(np.ldexp(u, exponent))
    c.ctx.step(dt)
    assert rel_linf(np.ldexp(c.get(), -exponent), ref) < 1e-12


@pytest.mark.parametrize("dim,order", [(2, 1), (2, 3), (3, 2), (3, 3)])
def test_projection_at_the_lower_end(dim, order):
    # one variable small, one of zeros, the others of the size of 1
    c = Case("euler", dim, order, (3, 2, 2)[:dim], limiter=1)
    lim = Limiter(c.oracle)
    u = np.random.default_rng(order).standard_normal(c.shape)
    u[..., 1] = np.ldexp(u[..., 1], -860)
    u[..., 2] = 0.0
    c.set(u)
    n = (c.ctx.cells,) + (lim.ns,) * dim + (c.ctx.nvar,)
    c.ctx.set_subcell_state(torch.zeros(int(np.prod(n)), dtype=torch.float64, device="cuda"),
                            torch.zeros(c.ctx.cells, dtype=torch.uint8, device="cuda"))
    rep = torch.empty(int(np.prod(n)), dtype=torch.float64, device="cuda")
    c.ctx.get_subcell_state(rep)
    torch.cuda.synchronize()
    assert rel_linf(rep.cpu().numpy(), lim.project(torch.from_numpy(u)).numpy()) < 1e-12
