"""The preconditioner's polynomial in one launch against its single steps: a
solve by itself takes the one, the same object twice in a batch the others; the
results are the same bit for bit.  Row counts around one block and around the
limit of the one launch (304 row blocks of 16), widths of one and of several
column tiles, odd steps and more steps than one launch takes."""
import numpy as np
import pytest

from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,degree,degree2", [(60, 2, 16, 48), (333, 9, 17, 48), (2000, 4, 2, 3),
                                                (2433, 30, 16, 48), (2433, 66, 16, 32),
                                                (3001, 10, 16, 66), (4864, 20, 16, 48),
                                                (4880, 20, 16, 48)])
def test_one_launch_gives_the_steps_bits(n, k, degree, degree2):
    import torch
    from paper_2605_29318_gb300 import binding
    c = synth.unit_cube(n, seed=n)
    a = synth.support_floor(c.X, c.a, factor=1.5)
    X, v, a = (torch.from_numpy(x).cuda() for x in (c.X, c.v, a))
    opts = binding.default_opts(tol=1e-6, cheb_degree=degree, cheb_degree_fp64=degree2,
                                max_iter=60)
    ctx = binding.Context(0, "fp64")
    ctx.rkpm_build(X, v, a)
    ctx.assemble_hessian(None, None, 1e6, 0.4)
    ev, modes, rep, st = ctx.eigenmodes(k, opts, check=False)
    o = {"X": X, "v": v, "a": a, "E0": 1e6, "nu0": 0.4, "k": k}
    _, res = binding.eigenmodes_batched([o, dict(o)], "fp64", opts, workers=2)
    for ev2, modes2, rep2, st2, _ in res:
        assert st2 == st and rep2["iterations"] == rep["iterations"]
        assert np.array_equal(ev2, ev) and torch.equal(modes2, modes)


@pytest.mark.parametrize("n,k", [(4865, 4), (4879, 20), (6001, 30), (5003, 66)])
def test_single_steps_in_a_row_match_steps_apart(n, k):
    """Row counts that end inside a block, over the limit of the one launch: steps
    that start while the one before drains give, alone and beside another solve on
    the GPU, the same bits, at the tensor-core step's widths of one to several tiles."""
    import torch
    from paper_2605_29318_gb300 import binding
    c = synth.unit_cube(n, seed=n)
    a = synth.support_floor(c.X, c.a, factor=1.5)
    X, v, a = (torch.from_numpy(x).cuda() for x in (c.X, c.v, a))
    opts = binding.default_opts(tol=1e-6, cheb_degree=16, cheb_degree_fp64=48, max_iter=40)
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
