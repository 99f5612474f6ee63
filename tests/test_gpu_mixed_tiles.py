"""Nodal matrices of clouds of which some tiles of rows are beyond the tiles'
capacities: only the rows of those take the row-owner passes."""
import numpy as np
import pytest

from oracle import assembly, rkpm
from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu


def _cube(n):
    c = synth.unit_cube(n, seed=11)
    c.a = synth.support_floor(c.X, c.a, factor=1.5)
    return c


def _one_wide(n, at, factor):
    """The support of the particle nearest to `at` widened: tiles of more than 512
    points, 1,200 columns or 20,480 list entries in one to twelve places."""
    c = _cube(n)
    c.a[np.argmin(((c.X - np.asarray(at)) ** 2).sum(1))] *= factor
    return c


def _spot(n):
    """The last 203 particles in a spot past the far corner, each covering all of them:
    the last tiles, the ragged one among them, have 41,209 list entries and more."""
    c = _cube(n)
    c.X[-203:] = 1.05 + 0.01 * np.random.default_rng(1).standard_normal((203, 3))
    c.a[-203:] = 0.1
    c.v[-203:] = 1e-6
    return c


CLOUDS = {"near": lambda: _one_wide(3003, (0, 0, 0), 4.5),
          "far": lambda: _one_wide(3000, (1, 1, 1), 3.6),
          "spot": lambda: _spot(2803)}


def _launches(ctx, c):
    import torch
    from paper_2605_29318_gb300 import binding
    ctx.rkpm_build(*(torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (c.X, c.v, c.a)))
    before = binding.launch_count()
    ctx.assemble_hessian(None, None, c.E, c.nu)
    return binding.launch_count() - before


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("name", list(CLOUDS))
def test_matrices_of_mixed_tiles(name, prec):
    """The bars of the matrix parity tests: the same pattern, values within
    1e-5 (FP32) or 1e-10 (double-float) of a row's largest.  Beside the launches for a
    cloud whose tiles all fit, the rows of the wide tiles are counted and filled."""
    from paper_2605_29318_gb300 import binding
    c = CLOUDS[name]()
    ctx = binding.Context(0, prec)
    fit = _launches(ctx, _cube(c.n))
    assert _launches(ctx, c) == fit + 2
    ptr, idx = rkpm.neighbours(c.X, c.a)
    phi, dphi, _ = rkpm.shape_functions(c.X, c.a, ptr, idx)
    H, M = assembly.assemble(c.n, ptr, idx, phi, dphi, c.v, c.E, c.nu)
    rp, col, Hg, Mg = ctx.export_matrices()
    assert np.array_equal(rp, H.indptr) and np.array_equal(col, H.indices)
    rows = np.repeat(np.arange(c.n), np.diff(rp))
    tol = 1e-5 if prec == "fp32" else 1e-10
    for got, want in ((Hg, H), (Mg, M)):
        scale = np.maximum.reduceat(np.abs(want.data), want.indptr[:-1])[rows]
        assert np.max(np.abs(got - want.data) / scale) < tol
