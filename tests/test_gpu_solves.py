"""Refined solves with the FP32 inverse against the oracle, at the sizes where the path changes (needs a GB300).

A team of W warps takes them up to 32 W unknowns, in kernels padded to fixed
sizes; beyond, and where the refinement cannot converge, the FP64 LU runs. At
rtol 1e-8 two legal builds of the oracle agree within 1.5e-10 in Y
(tests/test_oracle_rounding.py), so the parity bar of 1e-9 holds on every cell.
"""
import numpy as np
import pytest

import oracle
from synth import mechgen, states, write_mech
from tests import tinymech
from tests.test_gpu_parity import assert_parity, dlb, run_gpu

pytestmark = pytest.mark.gpu

# unknowns N = species + 1: both sides of every padded size, and of the limit 32 W
SIZES = [(1, n) for n in (12, 13, 20, 21, 32, 33)] + [(2, n) for n in (33, 40, 41, 56, 57, 64, 65)] + \
        [(4, n) for n in (33, 80, 81, 104, 105, 128, 129)]


@pytest.mark.parametrize("wpc,unknowns", SIZES)
def test_solve_sizes_match_oracle(tmp_path, wpc, unknowns):
    d = dlb()
    mech = str(tmp_path / "m.bin")
    write_mech(mech, mechgen.generate_mechanism(unknowns - 1, 3 * unknowns, 1 if unknowns == 65 else 2))
    T, p, Y = states.uniform_states(unknowns - 1, 12, unknowns)
    o = oracle.Oracle(mech).integrate(T, p, Y, 1e-7, rtol=1e-8, atol=1e-12, nthreads=16)
    for precision in (0, 1):
        ctx = d.Context(mech, rtol=1e-8, atol=1e-12, team_warps=wpc, precision=precision)
        assert_parity(run_gpu(ctx, T, p, Y, 1e-7), o)


@pytest.mark.parametrize("wpc", [1, 2, 4])
def test_rates_beyond_the_float_range_take_the_fp64_lu(tmp_path, wpc):
    """A <-> B at 1e39 /s over 1e-38 s: the iteration matrix overflows FP32, so no
    refined solve converges; the FP64 LU gives the oracle's relaxation."""
    d = dlb()
    sp = dict(atoms=[1, 0, 0, 0], s0=200.0, a=30.0, b=0.0)
    tinymech.make(tmp_path / "m.bin", [dict(sp, hf=0.0), dict(sp, hf=-1000.0)],
                  [dict(reac=[(0, 1)], prod=[(1, 1)], lnA=39.0 * np.log(10.0))])
    mech = str(tmp_path / "m.bin")
    T, p, Y = np.full(3, 1000.0), np.full(3, 1e5), np.array([[1.0, 0.5, 0.2], [0.0, 0.5, 0.8]])
    opts = dict(rtol=1e-8, atol=1e-12)
    o = oracle.Oracle(mech).integrate(T, p, Y, 1e-38, **opts)
    for precision in (0, 1):
        ctx = d.Context(mech, team_warps=wpc, precision=precision, **opts)
        assert_parity(run_gpu(ctx, T, p, Y, 1e-38), o)
        if precision:
            assert ctx.last_stats()["fp64_fallbacks"] > 0


def test_overlapping_calls_on_two_streams_keep_their_matrices():
    """Two plain calls of one context at once, more cells than fit the GPU: every
    resident team has a matrix of its own, so the results are those of one call."""
    import torch
    d = dlb()
    mech = states.mech_path(53, 325, 0)
    T, p, Y = (torch.tensor(a, device="cuda:0") for a in states.uniform_states(53, 700, 3))
    ctx = d.Context(mech, rtol=1e-6, atol=1e-10)
    ref = ctx.integrate(T, p, Y, 1e-7)
    torch.cuda.synchronize()
    s = [torch.cuda.Stream() for _ in range(2)]
    out = [ctx.integrate(T, p, Y, 1e-7, T_out=torch.empty_like(T), Y_out=torch.empty_like(Y), stream=q) for q in s]
    torch.cuda.synchronize()
    for o in out:
        assert torch.equal(o[0], ref[0]) and torch.equal(o[1], ref[1])
