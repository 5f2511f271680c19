"""Flops of an integrator step by unit, as the benchmark counts them (CPU)."""
import types

import pytest

import bench


def mech(nsp, nrx):
    return types.SimpleNamespace(nsp=nsp, nrx=nrx)


@pytest.mark.parametrize("nsp,nrx,f64,f32", [
    # rates, Jacobian and assembly; residuals in FP64; inverse, products (and the paired residual)
    (53, 325, 26760 + 29250 + 8748 + 23328, 314928 + 3 * 23328 + 23328),
    (10, 20, 1950 + 1800 + 363 + 2 * 968, 2662 + 3 * 968),
    (100, 1000, 79500 + 90000 + 30603 + 81608, 2060602 + 4 * 81608),
])
def test_fp64_work_leaves_out_what_runs_beside_it(nsp, nrx, f64, f32):
    assert bench.step_work(mech(nsp, nrx)) == {"f64": f64, "f32": f32}


def test_sizes_of_the_lu_count_it():
    m = mech(200, 2000)
    assert bench.step_work(m)["f64"] == pytest.approx(bench.flops_per_step(m)) and bench.step_work(m)["f32"] == 0
    mixed = bench.step_work(m, 1)
    assert mixed["f64"] + (2 / 3) * 201**3 == pytest.approx(bench.flops_per_step(m)) and mixed["f32"] > 0
