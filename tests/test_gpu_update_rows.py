"""The solver's block updates with one, two and four rows a thread and several
blocks a launch: the modes, put through the operators, have the residual that the
solver reports, ||H x - t M x|| / (t ||M x||) <= tol, to a hundredth (the products
are good to ~1e-9 of it at these sizes)."""
import pytest

from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k", [(101, 6), (1003, 66), (5003, 20), (7003, 12), (9002, 30)])
def test_residuals_of_the_returned_modes(n, k):
    import torch
    from paper_2605_29318_gb300 import binding
    c = synth.unit_cube(n, seed=n)
    a = synth.support_floor(c.X, c.a, factor=1.5)
    ctx = binding.Context(0, "fp64")
    ctx.rkpm_build(*(torch.from_numpy(x).cuda() for x in (c.X, c.v, a)))
    ctx.assemble_hessian(None, None, 1e6, 0.4)
    ev, modes, rep, st = ctx.eigenmodes(k, binding.default_opts(tol=1e-6))
    assert st == 0 and rep["max_residual"] <= 1e-6
    x = modes.double()
    HX, MX = ctx.apply_operators(x)
    t = torch.from_numpy(ev).to(x)
    r = (HX - MX * t).norm(dim=0) / (t.abs() * MX.norm(dim=0))
    assert r[1:].max().item() <= 1.01e-6
