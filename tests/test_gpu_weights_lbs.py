"""Skinning weights and linear blend skinning on GB300 at the sizes where their
kernels change path: widths around the vector lanes of a row, points around the
blocks, aligned and unaligned weights."""
import numpy as np
import pytest

from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
EPS = {"fp32": 2.0 ** -24, "fp64": 2.0 ** -53}


def _ctx(prec):
    import torch
    from paper_2605_29318_gb300 import binding
    c = synth.unit_cube(1500, seed=11)
    c.a = synth.support_floor(c.X, c.a, factor=1.5)
    ctx = binding.Context(0, prec)
    ctx.rkpm_build(*(torch.from_numpy(x).to(DEV) for x in (c.X, c.v, c.a)))
    return c, ctx


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("m", [1, 3, 16, 17, 33, 64, 65, 130])
def test_weights_at_every_lane_split(prec, m):
    """W = phi C with phi the exported shape functions: queries at the
    particles.  A row's sum of c terms is within (c + 2) eps sum |phi C| of the
    exact one; the query's shape functions sum their moments in another order
    than the build's, each within 1e3 condition-weighted roundings (the redo
    limit is 1e2 in FP32; FP64 contexts carry 2^-47)."""
    import torch
    c, ctx = _ctx(prec)
    ptr, idx, phi, _ = ctx.export_rkpm()
    C = torch.randn(c.n, m, device=DEV, dtype=ctx.dtype,
                    generator=torch.Generator(device=DEV).manual_seed(m))
    nq = 257
    Q = torch.from_numpy(c.X[:nq]).to(DEV)
    W = ctx.skinning_weights(Q, C).double().cpu().numpy()
    Cd = C.double().cpu().numpy()
    unit = 2.0 ** -24 if prec == "fp32" else 2.0 ** -47
    for q in range(nq):
        s = slice(ptr[q], ptr[q + 1])
        exact = phi[s] @ Cd[idx[s]]
        bound = 1e3 * unit * (np.abs(phi[s]) @ np.abs(Cd[idx[s]]))
        assert (np.abs(W[q] - exact) <= bound).all(), (q, np.abs(W[q] - exact).max())


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_failed_weights_leave_the_output_alone(prec):
    import torch
    from paper_2605_29318_gb300 import binding
    c, ctx = _ctx(prec)
    Q = torch.from_numpy(c.X[:40]).to(DEV).clone()
    Q[17] = 50.0                       # covered by nothing
    W = torch.full((40, 5), 7.0, dtype=ctx.dtype, device=DEV)
    C = torch.ones((5, c.n), dtype=ctx.dtype, device=DEV)
    st = ctx.L.ff_skinning_weights(ctx.h, Q.data_ptr(), 40, C.data_ptr(), 5, W.data_ptr())
    assert binding.STATUS[st] == "FF_ERR_SINGULAR_MOMENT"
    assert "query point 17 " in ctx.L.ff_last_error(ctx.h).decode()
    assert bool((W == 7.0).all())


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("m", [1, 2, 4, 5, 8, 9, 33, 62, 64, 65, 100])
@pytest.mark.parametrize("nq", [1, 33, 80001])
@pytest.mark.parametrize("shift", [0, 1])
def test_lbs_in_every_read_form(prec, m, nq, shift):
    """Each mode adds one product of a four-term form: the sum is within
    (m + 6) eps of the sum of absolute terms.  shift = 1 takes the weights off
    their 16-byte boundary."""
    import torch
    from paper_2605_29318_gb300 import binding
    ctx = binding.Context(0, prec)
    g = torch.Generator(device=DEV).manual_seed(100 * m + shift)
    Q = torch.randn(nq, 3, device=DEV, generator=g)
    room = torch.randn(nq * m + shift, device=DEV, dtype=ctx.dtype, generator=g)
    W = room[shift:].view(nq, m)
    Z = torch.randn(m, 3, 4, device=DEV, dtype=ctx.dtype, generator=g)
    x = ctx.lbs(Q, W, Z).double()
    h = torch.cat([Q.double(), torch.ones(nq, 1, device=DEV, dtype=torch.float64)], 1)
    Wd, Zd = W.double(), Z.double()
    exact = Q.double() + torch.einsum("qm,mrc,qc->qr", Wd, Zd, h)
    terms = Q.double().abs() + torch.einsum("qm,mrc,qc->qr", Wd.abs(), Zd.abs(), h.abs())
    assert bool(((x - exact).abs() <= (m + 6) * EPS[prec] * terms).all())


@pytest.mark.parametrize("crowd", [0, 40, 130])
def test_query_lists_in_and_past_the_kept_rounds(crowd):
    """Weights at the particles are phi C of the build's own lists: with cells of
    about ten nodes, of some forty (two rounds of 32) and of more than three rounds'
    worth, which are searched twice.  The bound of the lane-split test."""
    import torch
    from paper_2605_29318_gb300 import binding
    c = synth.unit_cube(1500, seed=12)
    rng = np.random.default_rng(crowd)
    near = (0.5 + 0.02 * rng.standard_normal((crowd, 3))).astype(np.float32)
    X = np.concatenate([c.X, near])
    v = np.concatenate([c.v, np.full(crowd, 1e-6, np.float32)])
    a = np.concatenate([c.a, np.full(crowd, 0.1, np.float32)])
    a = synth.support_floor(X, a, factor=1.5)
    ctx = binding.Context(0, "fp64")
    ctx.rkpm_build(*(torch.from_numpy(x).to(DEV) for x in (X, v, a)))
    ptr, idx, phi, _ = ctx.export_rkpm()
    C = torch.randn(len(X), 7, device=DEV, dtype=torch.float64,
                    generator=torch.Generator(device=DEV).manual_seed(crowd))
    W = ctx.skinning_weights(torch.from_numpy(X).to(DEV), C).cpu().numpy()
    Cd = C.cpu().numpy()
    for q in range(len(X)):
        s = slice(ptr[q], ptr[q + 1])
        bound = 1e3 * 2.0 ** -47 * (np.abs(phi[s]) @ np.abs(Cd[idx[s]]))
        assert (np.abs(W[q] - phi[s] @ Cd[idx[s]]) <= bound).all(), q
