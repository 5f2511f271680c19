"""Steps that leave the refined solves for the FP64 LU are counted (needs a GB300).

Parity with the oracle does not tell the two apart: the LU satisfies it too.
"""
import numpy as np
import pytest

from synth import mechgen, states, write_mech
from tests.test_gpu_parity import dlb, run_gpu
from tests.test_gpu_solve_limits import decay
from tests.test_gpu_solves import SIZES

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wpc,unknowns", SIZES)
def test_every_padded_size_converges(tmp_path, wpc, unknowns):
    """The states of the parity test at these sizes: no step leaves the refined solves."""
    d = dlb()
    mech = str(tmp_path / "m.bin")
    write_mech(mech, mechgen.generate_mechanism(unknowns - 1, 3 * unknowns, 1 if unknowns == 65 else 2))
    T, p, Y = states.uniform_states(unknowns - 1, 12, unknowns)
    for precision in (0, 1):
        ctx = d.Context(mech, rtol=1e-8, atol=1e-12, team_warps=wpc, precision=precision)
        run_gpu(ctx, T, p, Y, 1e-7)
        assert ctx.last_stats()["fp64_fallbacks"] == 0


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("wpc", [1, 2, 4])
def test_steps_that_do_not_converge_are_counted(tmp_path, wpc, precision):
    """1e39 /s overflows the float matrix: every attempted step takes the LU."""
    ctx = dlb().Context(decay(tmp_path, 1e39), rtol=1e-8, atol=1e-12, team_warps=wpc, precision=precision)
    T, p, Y = np.full(3, 1000.0), np.full(3, 1e5), np.array([[1.0, 0.5, 0.2], [0.0, 0.5, 0.8]])
    steps = run_gpu(ctx, T, p, Y, 1e-38)[2]
    assert ctx.last_stats()["fp64_fallbacks"] == steps.sum()


@pytest.mark.parametrize("wpc,unknowns", [(1, 11), (1, 54), (2, 54), (4, 54)])
def test_contexts_without_matrices_take_the_lu(wpc, unknowns):
    """An atol below 1e-30 leaves the kernel no matrices, as a failed allocation does."""
    d = dlb()
    mech = states.mech_path(10, 20, 0) if unknowns == 11 else states.mech_path(53, 325, 0)
    T, p, Y = states.uniform_states(10 if unknowns == 11 else 53, 20, 4)
    for precision in (0, 1):
        with_matrices = d.Context(mech, rtol=1e-6, atol=1e-30, team_warps=wpc, precision=precision)
        without = d.Context(mech, rtol=1e-6, atol=0.99e-30, team_warps=wpc, precision=precision)
        a, b = (run_gpu(c, T, p, Y, 1e-8) for c in (with_matrices, without))
        counted = precision == 1 or unknowns <= 32 * wpc   # 54 unknowns in one warp: the LU is the rule
        assert without.last_stats()["fp64_fallbacks"] == (b[2].sum() if counted else 0)
        assert np.all(np.abs(a[0] - b[0]) <= 1e-5 * b[0]) and np.all(np.abs(a[1] - b[1]) <= 1e-6)
        static = [torch.tensor(v, device="cuda:0") for v in (T, p, Y)]
        steps = torch.zeros(T.size, dtype=torch.int32, device="cuda:0")
        without.integrate_static(*static, 1e-8, torch.empty_like(static[0]), torch.empty_like(static[2]), steps=steps)
        assert without.last_stats()["fp64_fallbacks"] == (int(steps.sum()) if counted else 0)
