"""Solves of thin and of tiny clouds: their row blocks' unions have fewer k-steps of
16 columns than a block has warps, so that some warps of the tensor-core step copy
the block's own rows without a k-step of their own.  A solve by itself takes the
polynomial in one launch, the same object twice in a batch the single steps; the
results are the same bit for bit."""
import numpy as np
import pytest

from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu


def _bar(nx, ny, nz):
    """nx x ny x nz particles 0.1 apart, each moved by up to a tenth of that."""
    g = np.stack(np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij"), -1)
    g = g.reshape(-1, 3)
    X = 0.1 * (g + 0.1 * np.random.default_rng(nz).uniform(-1, 1, g.shape))
    n = len(X)
    return X.astype(np.float32), np.full(n, 1e-3, np.float32), np.full(n, 0.2, np.float32)


def _torus(n):
    c = synth.torus(n, seed=n)
    return c.X, c.v, synth.support_floor(c.X, c.a, factor=1.5)


CLOUDS = {
    "bar-3x3x60": (lambda: _bar(3, 3, 60), (36, 48, 80)),  # unions of 3 to 6 k-steps
    "torus-500": (lambda: _torus(500), (64, 80, 104)),     # 8 to 21
    "torus-150": (lambda: _torus(150), (36,)),             # 5 to 9
    "bar-2x2x1300": (lambda: _bar(2, 2, 1300), (20, 44)),  # 2 to 4, the form of four warps
}


@pytest.mark.parametrize("name,k", [(c, k) for c, (_, ks) in CLOUDS.items() for k in ks])
def test_small_unions_in_a_batch_match_alone(name, k):
    import torch
    from paper_2605_29318_gb300 import binding
    X, v, a = (torch.from_numpy(x).cuda() for x in CLOUDS[name][0]())
    opts = binding.default_opts(tol=1e-6, cheb_degree=16, cheb_degree_fp64=48, max_iter=30)
    ctx = binding.Context(0, "fp64")
    ctx.rkpm_build(X, v, a)
    ctx.assemble_hessian(None, None, 1e6, 0.4)
    first = ctx.eigenmodes(k, opts, check=False)
    again = ctx.eigenmodes(k, opts, check=False)
    o = {"X": X, "v": v, "a": a, "E0": 1e6, "nu0": 0.4, "k": k}
    _, res = binding.eigenmodes_batched([o, dict(o)], "fp64", opts, workers=2)
    for ev2, modes2, rep2, st2, *_ in [again] + list(res):
        assert st2 == first[3] and rep2["iterations"] == first[2]["iterations"]
        assert np.array_equal(ev2, first[0]) and torch.equal(modes2, first[1])
