"""What a weights call leaves on the device beside its lists: the bits and hits that
a pass keeps for the next stay within 256 MB, and more points than fit at once give
the same weights as in two calls."""
import pytest

from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu


def _two_set():
    """1,200,000 points on 3,000 centres: 451 MB of bits."""
    import torch
    from paper_2605_29318_gb300 import binding
    g = torch.Generator(device="cuda").manual_seed(5)
    X = torch.rand((20_000, 3), generator=g, device="cuda")
    ctx = binding.Context(0, "fp32")
    ctx.rkpm_build_twoset(X, torch.full((20_000,), 5e-5, device="cuda"), 3000)
    _, cen, rad = ctx.twoset()
    reach = 3.0 * torch.from_numpy(rad).float().cuda()
    return ctx, X[torch.from_numpy(cen).cuda()], reach, 1_200_000


def _nodal():
    """1,200,000 points: 461 MB of hits."""
    import torch
    from paper_2605_29318_gb300 import binding
    c = synth.unit_cube(2000, seed=4)
    a = synth.support_floor(c.X, c.a, factor=1.5)
    ctx = binding.Context(0, "fp32")
    X, v, a = (torch.from_numpy(x).cuda() for x in (c.X, c.v, a))
    ctx.rkpm_build(X, v, a)
    return ctx, X, a, 1_200_000


@pytest.mark.parametrize("build", [_two_set, _nodal])
def test_scratch_of_many_query_points(build):
    """The lists: 8 bytes a pair and 24 a point; 64 MB for what the allocators round up."""
    import torch
    ctx, nodes, reach, nq = build()
    n = len(nodes)
    g = torch.Generator(device="cuda").manual_seed(6)
    Q = 0.1 + 0.8 * torch.rand((nq, 3), generator=g, device="cuda")
    C = torch.randn((n, 2), generator=g, device="cuda")
    pairs = sum(int((torch.cdist(q, nodes) < reach).sum()) for q in Q.split(40_000))
    ctx.skinning_weights(Q[:64], C)
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    W = ctx.skinning_weights(Q, C)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= 8 * pairs + 24 * nq + (320 << 20)
    half = nq // 2 + 7
    again = torch.cat([ctx.skinning_weights(q, C) for q in (Q[:half], Q[half:])])
    assert torch.equal(W, again)
