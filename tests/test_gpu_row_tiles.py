"""The nodal assembly in tiles of rows against the oracle, at the edges of its
tiles and of its capacities: rows that do not fill a tile, lists longer than a
warp takes at once, a row's columns across several words, and clouds whose
tiles do not fit (these take the row-owner passes)."""
import numpy as np
import pytest

from oracle import assembly, rkpm
from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu


def _spots():
    """A dense cluster inside a sparse cloud: wide supports reach into it."""
    rng = np.random.default_rng(3)
    c = synth.unit_cube(900, seed=4, support=2.6)
    dense = 0.5 + 0.05 * rng.standard_normal((300, 3))
    c.X = np.concatenate([c.X, dense.astype(np.float32)])
    c.v = np.concatenate([c.v, np.full(300, 1e-6, np.float32)])
    c.a = np.concatenate([c.a, np.full(300, 0.12, np.float32)])
    return c


CLOUDS = {
    "5": lambda: synth.unit_cube(5, seed=2, support=6.0),
    "16": lambda: synth.unit_cube(16, seed=5, support=4.0),
    "17": lambda: synth.unit_cube(17, seed=6, support=4.0),
    "1000-lists-past-64": lambda: synth.unit_cube(1000, seed=7, support=2.9),
    "3001": lambda: synth.torus(3001, seed=8),
    "2000-tiles-too-wide": lambda: synth.unit_cube(2000, seed=9, support=4.2),
    "cluster": _spots,
}


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("name", list(CLOUDS))
def test_matrices_of_row_tiles(name, prec):
    """The bars of the matrix parity tests: the same pattern, values within
    1e-5 (FP32) or 1e-10 (double-float) of a row's largest."""
    import torch
    from paper_2605_29318_gb300 import binding
    c = CLOUDS[name]()
    c.a = synth.support_floor(c.X, c.a, m=min(8, c.n - 1), factor=1.5)
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
