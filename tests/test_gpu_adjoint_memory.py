"""The Picard adjoint on a device whose free memory holds the face adjoints and the iterate slabs, but
not lambda's face projections as well: the form with the slabs takes the step."""
import pytest
import torch

from paper_1905_07987_gb300 import ader, synth

pytestmark = pytest.mark.gpu


def context(side, order):
    cfg = ader.make_config("elastic", 3, order, (side,) * 3, (0,) * 3, (0.5 * side,) * 3, "absorbing",
                           synth.cfl_number(order))
    c = ader.Context(cfg)
    c.set_material(torch.from_numpy(synth.elastic_material((side,) * 3, seed=1).reshape(-1).copy()).cuda())
    c.set_point_source((0.6 * side / 2,) * 3, synth.moment_tensor(seed=2), 2.0, 0.5)
    return c


def adjoint(c, u, lam0, out):
    out[0].copy_(lam0)
    out[1].zero_()
    out[2].zero_()
    c.adjoint_step(0.3, 2e-3, u, *out)
    c.sync()
    return [o.cpu() for o in out]


def test_picard_adjoint_without_room_for_the_projections():
    side, order = 32, 5
    gen = torch.Generator("cuda").manual_seed(1)
    c = context(side, order)
    u, lam0, lam = (torch.randn(c.count, dtype=torch.float64, device="cuda", generator=gen) for _ in range(3))
    out = [lam] + [torch.empty(n, dtype=torch.float64, device="cuda") for n in (c.cells * 3, 6)]
    ref = adjoint(c, u, lam0, out)
    c.close()
    c = context(side, order)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    faces = c.cells * 3 * 2 * 36 * 9 * 8  # the face adjoints; the projections are as many
    rest = torch.empty(torch.cuda.mem_get_info()[0] - faces - 3 * faces // 4, dtype=torch.uint8, device="cuda")
    try:
        first, second = adjoint(c, u, lam0, out), adjoint(c, u, lam0, out)
    finally:
        del rest
        torch.cuda.empty_cache()
        c.close()
    for a, b, r in zip(first, second, ref):
        assert torch.equal(a, b)
        assert (a - r).abs().max() <= 1e-12 * r.abs().max()
