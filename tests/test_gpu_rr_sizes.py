"""The eigensolver at every size class of its dense step: bases of 3 nb columns
for nb = (k - 1 + 8) rounded up to four, from one block's registers (64, 96,
128, 160, 192 and 224 columns in FP32, 64 and 96 in double-float) to the
cluster's."""
import numpy as np
import pytest

from oracle import assembly, eigen, rkpm
from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu

_ORACLE = {}


def _cloud():
    if not _ORACLE:
        c = synth.unit_cube(2000, seed=1)
        ptr, idx = rkpm.neighbours(c.X, c.a)
        phi, dphi, _ = rkpm.shape_functions(c.X, c.a, ptr, idx)
        H, M = assembly.assemble(c.n, ptr, idx, phi, dphi, c.v, c.E, c.nu)
        _ORACLE["x"] = (c, eigen.eigh_dense(H, M, 72)[0])
    return _ORACLE["x"]


@pytest.mark.parametrize("k", [2, 12, 14, 24, 26, 34, 36, 44, 46, 56, 58, 66, 70])
def test_eigenvalues_at_every_basis_size(k):
    """A residual of 1e-7 (the bar of the 2,000-particle cube's parity tests)
    leaves eigenvalues within its square over the gap, and their double-float
    Rayleigh quotients within 1e-9; 1e-7 is asked for."""
    import torch
    from paper_2605_29318_gb300 import binding
    c, lam = _cloud()
    ctx = binding.Context(0, "fp64")
    ctx.rkpm_build(*(torch.from_numpy(x).cuda() for x in (c.X, c.v, c.a)))
    ctx.assemble_hessian(None, None, c.E, c.nu)
    ev, _, rep, st = ctx.eigenmodes(k, binding.default_opts(tol=1e-7))
    assert st == 0 and rep["max_residual"] <= 1e-7
    assert np.max(np.abs(ev[1:] - lam[1:k]) / lam[1:k]) < 1e-7


def test_a_wide_basis():
    """876 columns (256 modes, the most that a call may ask for, with 36 guard
    vectors): the modes, put through the operators, have the residual that was
    asked for, to a hundredth."""
    import torch
    from paper_2605_29318_gb300 import binding
    c = synth.unit_cube(3100, seed=2)
    a = synth.support_floor(c.X, c.a, factor=1.5)
    ctx = binding.Context(0, "fp64")
    ctx.rkpm_build(*(torch.from_numpy(x).cuda() for x in (c.X, c.v, a)))
    ctx.assemble_hessian(None, None, c.E, c.nu)
    ev, modes, rep, st = ctx.eigenmodes(256, binding.default_opts(tol=1e-6, guard=36))
    assert st == 0 and rep["max_residual"] <= 1e-6
    x = modes.double()
    HX, MX = ctx.apply_operators(x)
    t = torch.from_numpy(ev).to(x)
    r = (HX - MX * t).norm(dim=0) / (t.abs() * MX.norm(dim=0))
    assert r[1:].max().item() <= 1.01e-6
