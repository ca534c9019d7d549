"""Gradients in materials whose shear modulus or bulk modulus vanishes: the derivative of a step with
respect to (rho, lambda, mu) is finite there, and as exact as elsewhere (against the oracle)."""
import numpy as np
import pytest
import torch

from cases import Case
from oracle.adjoint import step_vjp
from paper_1905_07987_gb300 import synth

pytestmark = pytest.mark.gpu

# (lambda, mu): a fluid, nearly one, 3 lambda + 2 mu = 0 and nearly so
MATERIALS = [(2.0, 0.0), (2.0, 2e-9), (-1.0, 1.5), (-1.0, 1.5 + 1e-9)]


def device(a):
    return torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).cuda()


def check(order, lam, mu, predictor, source, static, precision="fp64", tol=1e-12):
    nc = (3, 2, 2)
    mat = synth.elastic_material(nc, seed=order)
    mat[::2, 1] = lam  # the other cells keep an ordinary material
    mat[::2, 2] = mu
    c = Case("elastic", 3, order, nc, hi=(1.5, 1.0, 1.0), bc="absorbing", material=mat, predictor=predictor,
             precision=precision)
    if source:
        c.point_source([0.3, 0.2, 0.3], synth.moment_tensor(5), 2.0, 0.4)
    rng = np.random.default_rng(order)
    u, adj = rng.standard_normal(c.shape), rng.standard_normal(c.shape)
    dt = 0.7 * float(c.oracle.cfl_dt(torch.from_numpy(u)))
    ref = step_vjp(c.oracle, torch.from_numpy(u), torch.from_numpy(adj), dt, 0.35)
    lam_d = device(adj)
    gm = torch.zeros(c.ctx.cells * 3, dtype=torch.float64, device="cuda")
    gM = torch.zeros(6, dtype=torch.float64, device="cuda")
    c.ctx.adjoint_step(0.35, dt, device(u), lam_d, gm, gM, static=static)
    c.ctx.sync()
    out = (lam_d.cpu().numpy(), gm.cpu().numpy(), gM.cpu().numpy())
    for a, b in zip(out, ref):
        b = b.numpy().reshape(-1)
        assert np.abs(a - b).max() <= tol * np.abs(b).max()
    if precision != "fp64":
        return
    # each material parameter by its own size too
    a, b = gm.cpu().numpy().reshape(-1, 3), ref[1].numpy()
    assert (np.abs(a - b).max(axis=0) <= 1e-12 * np.abs(b).max(axis=0)).all()


@pytest.mark.parametrize("lam,mu", MATERIALS)
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5])
def test_picard(order, lam, mu):
    check(order, lam, mu, "picard", source=order % 2 == 1, static=order == 2)


@pytest.mark.parametrize("lam,mu", MATERIALS)
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5])
def test_ck(order, lam, mu):
    check(order, lam, mu, "ck", source=order % 2 == 1, static=order == 2)


# binary32 levels: a few of its roundings relative to the largest value, on states that are not smooth
@pytest.mark.parametrize("lam,mu", MATERIALS)
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5])
def test_ck_mixed(order, lam, mu):
    check(order, lam, mu, "ck", source=order % 2 == 1, static=order == 2, precision="mixed", tol=2e-6)
