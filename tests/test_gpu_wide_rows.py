"""Nodal matrices of clouds between what a tile of rows may list and what its block can
hold: one wide support gives some rows more than 1,200 columns, which eight warps of
double-float sums do not fit beside the tile's tables."""
import numpy as np
import pytest

from oracle import assembly, rkpm
from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu


def _one_wide(n, support, factor):
    """A cube whose most central particle has its support widened."""
    c = synth.unit_cube(n, seed=7, support=support)
    c.a = synth.support_floor(c.X, c.a, factor=1.5)
    c.a[np.argmin(((c.X - 0.5) ** 2).sum(1))] *= factor
    return c


# the most a tile lists: 499 points, 1,222 columns, 20,300 entries (235,248 bytes of 232,448
# in double-float); 509, 1,250 and 20,462 (228,976 bytes); 575 points, more than a tile of
# any type may have
CLOUDS = {"1222-columns": (4000, 2.1, 2.3), "1250-columns": (4000, 2.1, 2.25),
          "575-points": (4000, 2.0, 2.4)}


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("name", list(CLOUDS))
def test_matrices_with_wide_rows(name, prec):
    """The bars of the matrix parity tests: the same pattern, values within
    1e-5 (FP32) or 1e-10 (double-float) of a row's largest."""
    import torch
    from paper_2605_29318_gb300 import binding
    c = _one_wide(*CLOUDS[name])
    ptr, idx = rkpm.neighbours(c.X, c.a)
    phi, dphi, _ = rkpm.shape_functions(c.X, c.a, ptr, idx)
    H, M = assembly.assemble(c.n, ptr, idx, phi, dphi, c.v, c.E, c.nu)
    ctx = binding.Context(0, prec)
    ctx.rkpm_build(*(torch.from_numpy(x).cuda() for x in (c.X, c.v, c.a)))
    ctx.assemble_hessian(None, None, c.E, c.nu)
    rp, col, Hg, Mg = ctx.export_matrices()
    assert np.array_equal(rp, H.indptr) and np.array_equal(col, H.indices)
    rows = np.repeat(np.arange(c.n), np.diff(rp))
    tol = 1e-5 if prec == "fp32" else 1e-10
    for got, want in ((Hg, H), (Mg, M)):
        scale = np.maximum.reduceat(np.abs(want.data), want.indptr[:-1])[rows]
        assert np.max(np.abs(got - want.data) / scale) < tol
