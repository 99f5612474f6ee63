"""Farthest-point sampling on GB300 against the oracle's plain loop, index by
index, where its rounds can go wrong: lattices (many exact ties), duplicates,
sizes around one block's points, other start points, tiny and large scales."""
import numpy as np
import pytest

from oracle import twoset

pytestmark = pytest.mark.gpu


def _lattice(m, h):
    g = np.arange(m) * h
    return np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)


def _random(n, seed):
    return np.random.default_rng(seed).random((n, 3))


CASES = {
    "lattice-8000": (lambda: _lattice(20, 0.05), 300, 0),
    "lattice-262144": (lambda: _lattice(64, 0.25), 150, 77),
    "one-block-500": (lambda: _random(500, 1), 200, 7),
    "one-block-1024": (lambda: _random(1024, 2), 400, 1023),
    "two-blocks-1025": (lambda: _random(1025, 3), 300, 1024),
    "blocks-9000": (lambda: _random(9000, 4), 500, 3),
    "sorted-40000": (lambda: np.array(sorted(map(tuple, _random(40000, 5)))), 200, 0),
    "duplicates-6300": (lambda: np.repeat(_random(700, 6), 9, 0), 650, 2),
    "lattice-and-random": (lambda: np.concatenate([_lattice(16, 1 / 16), _random(9000, 7)]), 300, 0),
    "tiny-5000": (lambda: _random(5000, 8) * 1e-15, 150, 0),
    "large-5000": (lambda: _random(5000, 9) * 1e17, 150, 0),
    "whole-slice-in-global-memory": (lambda: _random(1_700_000, 10), 12, 5),
}


@pytest.mark.parametrize("name", list(CASES))
def test_centres_are_the_oracles(name):
    import torch
    from paper_2605_29318_gb300 import binding
    make, K, start = CASES[name]
    X = make().astype(np.float32)
    ctx = binding.Context(0, "fp32")
    # the whole Gaussian where K centres cover the points thinly
    ctx.rkpm_build_twoset(torch.from_numpy(X).cuda(), torch.ones(len(X), device="cuda"), K,
                          0.0 if K < 100 else 3.0, start)
    _, cen, _ = ctx.twoset()
    assert np.array_equal(cen, twoset.farthest_point_sampling(X, K, start))


@pytest.mark.parametrize("repeat", [3, 60])
def test_as_many_centres_as_distinct_points(repeat):
    """40 distinct positions (one block's points, and several blocks'): 40
    centres are found, 41 are refused at step 40."""
    import torch
    from paper_2605_29318_gb300 import binding
    X = np.repeat(_random(40, 11).astype(np.float32), repeat, 0)
    Xd, v = torch.from_numpy(X).cuda(), torch.ones(len(X), device="cuda")
    ctx = binding.Context(0, "fp32")
    ctx.rkpm_build_twoset(Xd, v, 40, 0.0, 0)
    assert np.array_equal(ctx.twoset()[1], twoset.farthest_point_sampling(X, 40, 0))
    with pytest.raises(binding.FreeformError, match="step 40"):
        ctx.rkpm_build_twoset(Xd, v, 41, 0.0, 0)


@pytest.mark.parametrize("n,K,trunc", [(513, 31, 3.0), (512, 32, 3.0), (777, 33, 3.0),
                                       (1300, 256, 3.0), (1300, 257, 2.5), (600, 64, 0.0),
                                       (1025, 1024, 3.0), (3400, 3201, 3.0)])
def test_covering_lists_at_the_edges_of_their_words(n, K, trunc):
    """Lists from the bits (K up to 3,200) and from the two passes beyond, pair
    by pair the oracle's."""
    import torch
    from paper_2605_29318_gb300 import binding
    X = _random(n, n + K).astype(np.float32)
    ctx = binding.Context(0, "fp32")
    ctx.rkpm_build_twoset(torch.from_numpy(X).cuda(), torch.ones(n, device="cuda"), K, trunc, 0)
    _, cen, rad = ctx.twoset()
    ptr, idx = twoset.covering(X, X[cen], rad, trunc or None)
    got_ptr, got_idx, _, _ = ctx.export_rkpm()
    assert np.array_equal(got_ptr, ptr) and np.array_equal(got_idx, idx)
