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
