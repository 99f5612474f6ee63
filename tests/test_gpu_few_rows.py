"""Nodal shape functions where a row takes a whole warp and where it takes eight lanes:
sizes on both sides of each line against the oracle, and the launches of a build (an FP32
build of few rows redoes its ill-conditioned ones in place, without a second launch)."""
import numpy as np
import pytest

from oracle import rkpm
from paper_2605_29318_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {"fp32": 2e-5, "fp64": 1e-10}  # the bars of the shape-function parity tests


def _build(n, prec):
    import torch
    from paper_2605_29318_gb300 import binding
    c = synth.unit_cube(n, seed=n)
    a = synth.support_floor(c.X, c.a, m=min(8, n - 1), factor=1.5)
    ctx = binding.Context(0, prec)
    d = [torch.from_numpy(x).cuda() for x in (c.X, c.v, a)]
    ctx.rkpm_build(*d)
    before = binding.launch_count()
    ctx.rkpm_build(*d)
    return ctx, c.X, a, binding.launch_count() - before


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("prec,waves", [("fp32", 64), ("fp64", 16)])
@pytest.mark.parametrize("past", [None, -1, 0, 1])
def test_rows_on_both_sides_of_the_line(prec, waves, past):
    n = 61 if past is None else waves * _sms() + past
    ctx, X, a, _ = _build(n, prec)
    ptr, idx = rkpm.neighbours(X, a)
    phi, dphi, _ = rkpm.shape_functions(X, a, ptr, idx)
    got = ctx.export_rkpm()
    assert np.array_equal(got[0], ptr) and np.array_equal(got[1], idx)
    assert np.abs(got[2] - phi).max() <= TOL[prec] * np.abs(phi).max()
    assert np.abs(got[3] - np.asarray(dphi)).max() <= TOL[prec] * np.abs(dphi).max()


def test_launches_of_a_small_build():
    """The same in both precisions: no second launch for the FP64 rows of an FP32 build."""
    assert _build(2000, "fp32")[3] == _build(2000, "fp64")[3]
