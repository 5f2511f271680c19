"""Properties of the device headers that can be checked on the host: a small translation unit is compiled with nvcc."""
import os
import subprocess

import pytest

from paper_2011_07978_gb300 import build


def compile_cu(tmp_path, source, name="t"):
    src = tmp_path / (name + ".cu")
    src.write_text(source)
    exe = str(tmp_path / name)
    try:
        cc = build.nvcc()
    except RuntimeError as err:
        pytest.skip(str(err))
    r = subprocess.run([cc, *build.ARCH, "-O1", "-std=c++17", "-I", build.CSRC, "-o", exe, str(src)],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.skipif(not os.path.isdir(build.CSRC), reason="no device sources")
def test_a_team_is_not_copied(tmp_path):
    """Which set of slots a team's next reduction writes is state of the team. A function that takes
    the team by value and reduces loses that state on return; the caller's next reduction then writes
    slots that a slower warp still reads. What may be copied is the threads and their barrier."""
    compile_cu(tmp_path, """
#include <type_traits>
#include "integrator_impl.cuh"
template <int W> constexpr bool copied =
    std::is_copy_constructible<dlb::Team<W>>::value || std::is_copy_assignable<dlb::Team<W>>::value;
static_assert(!copied<1> && !copied<2> && !copied<4>, "a copied team reduces through slots that are still read");
int main() { return 0; }
""")


def test_solve_vectors_lie_over_dead_arrays_only(tmp_path):
    """Workspace of the refined solves for every size, chunk and slot count that a mechanism can have:
    what lives across a rate evaluation stays off the arrays that one writes, nothing overlaps, and
    every vector is 16-byte aligned."""
    exe = compile_cu(tmp_path, r"""
#include <cstdio>
#include "dlb_common.cuh"
static int bad(const char* what, int wpc, int N, int DS, int nrx) {
  std::printf("%s: %d warps, %d unknowns, %d slots, %d reactions\n", what, wpc, N, DS, nrx);
  return 1;
}
int main() {
  long checked = 0;
  for (int wpc = 1; wpc <= 4; wpc *= 2)
    for (int N = 2; N <= 32 * wpc; ++N)
      for (int DS = 1; DS <= 12; ++DS)
        for (int nrx = 1; nrx <= 5000; nrx += nrx < 400 ? 1 : 23) {
          const int CH = 32 * wpc;
          const dlb::WsLayout L = dlb::make_layout(N - 1, nrx, CH, N, N + 1, DS, true);
          // start, doubles: weights, right-hand side, first solution, inverse, reciprocals, rows
          const int at[6] = {L.w32, L.v, L.xf, L.xs, L.invs, L.rows};
          const int n[6] = {(N + 1) / 2, CH / 2, (N + 1) / 2,
                            wpc == 1 && N <= dlb::kSharedX ? dlb::kSharedX * N / 2 : 0, 1, CH};
          const bool over = L.w32 < L.scal;
          for (int i = 0; i < 6; ++i) {
            if (at[i] & 1) return bad("not aligned", wpc, N, DS, nrx);
            if (i > 0 && at[i - 1] + n[i - 1] > at[i]) return bad("overlap", wpc, N, DS, nrx);
            const int end = at[i] + n[i];
            if (over && (at[i] < L.dwdT || end > (i < 4 ? L.D : L.scal))) return bad("over a live array", wpc, N, DS, nrx);
            if (!over && (at[i] < L.perm + (N + 1) / 2 + 1 || end > L.total)) return bad("outside", wpc, N, DS, nrx);
          }
          ++checked;
        }
  std::printf("%ld\n", checked);
  return 0;
}
""")
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
