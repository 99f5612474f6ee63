"""The operators on blocks of every width class (lanes of 16 bytes a row, whole
fours and not, pieces of wide blocks): the assembled product against the exported
matrices, the allocation-free and the matrix-free ones against it."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu

EPS = {"fp32": 2.0 ** -24, "fp64": 2.0 ** -53}


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 8, 10, 16, 17, 33, 63, 66, 130, 131])
@pytest.mark.parametrize("n", [700, 2600])
def test_products_at_every_width(prec, m, n):
    """A row of c entries is summed with c + 8 roundings of terms up to |h| (|x_l|
    + |x_k|): the bound.  n = 700 takes the kernels for few rows, 2,600 those for
    many.  The matrix-free product reads tables, not matrices: both carry their
    build's rounding (1e-5 of a row's terms in FP32, 1e-11 in double-float)."""
    import torch
    from paper_2605_29318_gb300 import binding
    c = synth.unit_cube(n, seed=n)
    a = synth.support_floor(c.X, c.a, factor=1.5)
    ctx = binding.Context(0, prec)
    ctx.rkpm_build(*(torch.from_numpy(x).cuda() for x in (c.X, c.v, a)))
    ctx.assemble_hessian(None, None, 1e5, 0.4)
    rp, col, Hv, Mv = ctx.export_matrices()
    X = torch.randn(n, m, dtype=ctx.dtype, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(m))
    x = X.double().cpu().numpy()
    width = np.diff(rp).max()
    out = {"assembled": ctx.apply_operators(X)}
    if 3 * n * m * X.element_size() <= (32 << 20) - 768:
        out["static"] = ctx.apply_operators_noalloc(X)
    out["tables"] = ctx.apply_operators_matfree(X, None, None, 1e5, 0.4)
    for q, val in enumerate((Hv, Mv)):
        A = sp.csr_matrix((val, col, rp), shape=(n, n))
        B = abs(A)
        exact = A @ x
        terms = B @ np.abs(x) + np.asarray(B.sum(1)) * np.abs(x)
        for name, ys in out.items():
            tol = ((width + 8) * EPS[prec] if name != "tables"
                   else {"fp32": 1e-5, "fp64": 1e-11}[prec])
            err = np.abs(ys[q].double().cpu().numpy() - exact)
            assert (err <= tol * terms).all(), (name, "HM"[q], (err / terms).max())
