"""Refined solves at the limits of the float range, against the oracle (needs a GB300).

They hold the matrix's inverse, right-hand sides and corrections as floats; numbers that floats
cannot hold take the FP64 LU. The bounds are those of rtol 1e-8 runs of the oracle's own builds.
"""
import numpy as np
import pytest

import oracle
from tests import tinymech
from tests.test_gpu_parity import assert_parity, dlb, run_gpu

pytestmark = pytest.mark.gpu


def decay(tmp_path, k, hf=0.0):
    """A -> B at k /s"""
    sp = dict(atoms=[1, 0, 0, 0], s0=200.0, a=30.0, b=0.0)
    tinymech.make(tmp_path / "m.bin", [dict(sp, hf=0.0), dict(sp, hf=hf)],
                  [dict(reac=[(0, 1)], prod=[(1, 1)], lnA=np.log(k), rev=0)])
    return str(tmp_path / "m.bin")


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("wpc", [1, 2, 4])
@pytest.mark.parametrize("atol,y", [(1e-30, 1e-24), (1e-60, 1e-50)])
def test_traces_far_below_the_float_range_react(tmp_path, wpc, precision, atol, y):
    """A trace decays by 1/e within its tolerance, whatever the size of the trace and of atol."""
    mech = decay(tmp_path, 1e7)
    T, p, Y = np.full(3, 1000.0), np.full(3, 1e5), np.array([[y, 0.3 * y, 0.0], [1.0, 1.0, 1.0]])
    opts = dict(rtol=1e-8, atol=atol)
    o = oracle.Oracle(mech).integrate(T, p, Y, 1e-7, **opts)
    assert abs(o[1][0, 0] / (y * np.exp(-1.0)) - 1.0) < 1e-6
    g = run_gpu(dlb().Context(mech, team_warps=wpc, precision=precision, **opts), T, p, Y, 1e-7)
    assert_parity(g, o)
    assert np.all(np.abs(g[1][0] - o[1][0]) <= 1e-6 * o[1][0])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("wpc", [1, 2, 4])
def test_pivots_whose_reciprocal_is_no_normal_float(tmp_path, wpc, precision):
    """1.5e-38 s in one step: the diagonal, 1/(gamma h) = 1.2e38, is a float and its reciprocal is
    below 2^-126, where the hardware reciprocal gives zero."""
    mech = decay(tmp_path, 1e36, hf=-1000.0)
    T, p, Y = np.full(3, 1000.0), np.full(3, 1e5), np.array([[1.0, 0.5, 0.2], [0.0, 0.5, 0.8]])
    opts = dict(rtol=1e-8, atol=1e-12)
    o = oracle.Oracle(mech).integrate(T, p, Y, 1.5e-38, **opts)
    assert abs(o[1][0, 0] / np.exp(-0.015) - 1.0) < 1e-7
    ctx = dlb().Context(mech, team_warps=wpc, precision=precision, **opts)
    assert_parity(run_gpu(ctx, T, p, Y, 1.5e-38), o)
