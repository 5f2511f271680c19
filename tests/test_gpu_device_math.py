"""Logarithm and step factor of the integrator over their ranges, in a kernel of their own (needs a GB300)."""
import subprocess

import numpy as np
import pytest

from tests.test_device_headers import compile_cu

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdio>
#include <vector>
#include "integrator_impl.cuh"
__global__ void math_kernel(int n, const double* x, double* out, const double* tab) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[2 * i] = dlb::log_tab(x[i], tab);
  out[2 * i + 1] = dlb::step_factor(x[i]);
}
int main(int argc, char** argv) {   // table, arguments, results
  auto read = [](const char* name) {
    std::vector<double> v;
    double b[512];
    FILE* f = std::fopen(name, "rb");
    for (size_t got; f && (got = std::fread(b, 8, 512, f)) > 0;) v.insert(v.end(), b, b + got);
    if (f) std::fclose(f);
    return v;
  };
  if (argc != 4) return 2;
  const std::vector<double> tab = read(argv[1]), x = read(argv[2]);
  const int n = int(x.size());
  if (tab.size() != 64 || n < 1) return 2;
  std::vector<double> out(2 * size_t(n));
  double *dt = nullptr, *dx = nullptr, *dout = nullptr;
  if (cudaMalloc(&dt, 512) || cudaMalloc(&dx, 8 * size_t(n)) || cudaMalloc(&dout, 16 * size_t(n))) return 3;
  cudaMemcpy(dt, tab.data(), 512, cudaMemcpyHostToDevice);
  cudaMemcpy(dx, x.data(), 8 * size_t(n), cudaMemcpyHostToDevice);
  math_kernel<<<(n + 255) / 256, 256>>>(n, dx, dout, dt);
  if (cudaMemcpy(out.data(), dout, 16 * size_t(n), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  FILE* f = std::fopen(argv[3], "wb");
  const bool ok = f && std::fwrite(out.data(), 8, out.size(), f) == out.size();
  return f && std::fclose(f) == 0 && ok ? 0 : 4;
}
"""


def device_math(tmp_path, x):
    exe = compile_cu(tmp_path, SOURCE)
    tab = np.exp2(np.arange(64, dtype=np.longdouble) / 64).astype(np.float64)
    tab.tofile(tmp_path / "tab")
    np.asarray(x, dtype=np.float64).tofile(tmp_path / "x")
    r = subprocess.run([exe, *(str(tmp_path / k) for k in ("tab", "x", "out"))], capture_output=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return np.fromfile(tmp_path / "out").reshape(-1, 2).T


def test_logarithm(tmp_path):
    """Half an ulp of the result plus 1.7e-16: the table's rounding, 1.1e-16 of a significand near 1,
    and less than half of that for the series. 0.7 ulp between 200 and 4,000 K."""
    rng = np.random.default_rng(2)
    x = np.concatenate([rng.uniform(200.0, 4000.0, 200000), np.exp(rng.uniform(-708.0, 709.0, 100000)),
                        1.0 + rng.uniform(-0.02, 0.02, 50000), np.ldexp(1.0, np.arange(-1022, 1024)),
                        np.nextafter(np.ldexp(1.0, np.arange(-1020, 1024)), 0.0)])
    got = device_math(tmp_path, x)[0]
    want = np.log(x.astype(np.longdouble))
    err = np.abs((got - want).astype(np.float64))
    assert np.all(err <= 0.5 * np.spacing(np.abs(want.astype(np.float64))) + 1.7e-16)
    at = slice(0, 200000)
    assert np.max(err[at] / np.spacing(np.abs(want[at].astype(np.float64)))) <= 0.7


def test_logarithm_of_what_has_none(tmp_path):
    x = np.array([0.0, -0.0, -1.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 2.2e-308])
    got = device_math(tmp_path, x)[0]
    with np.errstate(all="ignore"):
        want = np.log(x)
    np.testing.assert_allclose(got, want, rtol=4e-16)


def test_step_factor(tmp_path):
    """Seven roundings in y^8, an eighth of them in the result, the last sum, the factor 0.9 and its
    product, half an ulp (2^-53 relative) each: 3.5 2^-53. The limits hold outside, NaN among them."""
    rng = np.random.default_rng(3)
    x = np.concatenate([np.exp(rng.uniform(np.log(1.0001e-7), np.log(0.9999e6), 200000)),
                        1.0 + rng.uniform(-1e-3, 1e-3, 50000)])
    got = device_math(tmp_path, x)[1]
    want = np.longdouble(9) / 10 * x.astype(np.longdouble) ** (np.longdouble(-1) / 8)
    assert np.max(np.abs((got - want) / want)) <= 3.5 * 2.0 ** -53
    out = device_math(tmp_path, [0.0, 1e-300, 0.99e-7, 1.01e6, 1e300, np.inf, np.nan])[1]
    assert out.tolist() == [5.0, 5.0, 5.0, 0.2, 0.2, 0.2, 0.2]
