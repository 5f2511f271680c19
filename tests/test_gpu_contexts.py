"""Contexts side by side (needs a GB300)."""
import pytest

from synth import states
from tests.test_gpu_parity import dlb

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wpc", [1, 2, 4])
def test_a_smaller_context_leaves_the_larger_one_its_shared_memory(wpc):
    """The shared-memory limit belongs to the kernel function, which contexts of one team size have
    in common: creating a smaller one must not lower it under the larger one's next calls."""
    d = dlb()
    T, p, Y = (torch.tensor(a, device="cuda:0") for a in states.uniform_states(53, 40, 1))
    big = d.Context(states.mech_path(53, 325, 0), team_warps=wpc)
    want = [*big.integrate(T, p, Y, 1e-8), *big.rhs(T, p, Y)]
    small = d.Context(states.mech_path(10, 20, 0), team_warps=wpc)
    got = [*big.integrate(T, p, Y, 1e-8), *big.rhs(T, p, Y)]
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, got))
    small.close()
    big.close()
