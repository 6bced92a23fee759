"""A launch that the driver refuses while a cycle is being recorded is reported by that
step and by every later one until a recording succeeds: no graph without its coarse levels
is kept.  Host logic alone, on a stand-in of the CUDA runtime (tests/refused_launch.cu)."""
import os
import subprocess

import pytest

from paper_2208_14703_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
ERR_CUDA = -5


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("refused") / "refused_launch")
    cmd = [B.nvcc(), *B.ARCH, "-std=c++17", "-O1", "-cudart=none", "-I", B.CSRC, "-I", B.INCLUDE,
           os.path.join(HERE, "refused_launch.cu"), "-o", exe, "-Xlinker",
           "--unresolved-symbols=ignore-all"]
    p = subprocess.run(cmd, capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    return exe


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("refused", [0, 1, 2])
def test_refused_launch_is_reported_until_recorded(program, precision, refused):
    out = subprocess.run([program, str(precision), str(refused)], capture_output=True, text=True,
                         timeout=60)
    assert out.returncode == 0, (out.returncode, out.stderr)
    *status, graphs, taken = (int(x) for x in out.stdout.split())
    assert [s == ERR_CUDA for s in status] == [k < refused for k in range(3)]
    assert graphs == taken == 1
