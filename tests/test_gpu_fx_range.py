"""States near the ends of binary64's range: what the fixed-point forms leave to the FP64 forms."""
import numpy as np
import pytest
import torch

from cases import Case, rel_linf
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
