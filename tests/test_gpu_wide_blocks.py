"""H_w on constant columns of wide FP64 blocks.  Past 128 columns, and at widths that
are not whole fours, the products sum h (x_l - x_k): a constant column gives zero,
not a rounding of it, and a large common part costs no digits."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [37, 130, 132, 192, 256, 512])
@pytest.mark.parametrize("n", [700, 2600])
def test_constant_columns_of_wide_blocks(n, m):
    """A row of c entries is summed with c + 8 roundings of terms |h| |x_l - x_k|, the
    differences exact where the block is a multiple of 2^-20 around 2^10."""
    import torch
    from paper_2605_29318_gb300 import binding
    c = synth.unit_cube(n, seed=n)
    a = synth.support_floor(c.X, c.a, factor=1.5)
    ctx = binding.Context(0, "fp64")
    ctx.rkpm_build(*(torch.from_numpy(x).cuda() for x in (c.X, c.v, a)))
    ctx.assemble_hessian(None, None, 1e5, 0.4)
    rng = np.random.default_rng(m)
    flat = np.tile(rng.uniform(0.5, 2.0, m), (n, 1))
    d = rng.integers(-4096, 4096, (n, m)) * 2.0 ** -20
    rp, col, Hv, _ = ctx.export_matrices()
    rows = np.repeat(np.arange(n), np.diff(rp))
    width = np.diff(rp).max()
    H = sp.csr_matrix((np.where(rows == col, 0.0, Hv), col, rp), shape=(n, n))
    want = H @ d - np.asarray(H.sum(1)) * d
    terms = abs(H) @ np.abs(d) + np.asarray(abs(H).sum(1)) * np.abs(d)
    calls = [ctx.apply_operators]
    if 3 * n * m * 8 <= (32 << 20) - 768:
        calls.append(ctx.apply_operators_noalloc)
    for call in calls:
        YH, _ = call(torch.from_numpy(flat).cuda())
        assert YH.abs().max().item() == 0.0
        YH, _ = call(torch.from_numpy(1024.0 + d).cuda())
        err = np.abs(YH.cpu().numpy() - want)
        assert (err <= (2 * width + 16) * 2.0 ** -53 * terms).all(), (err / terms).max()
