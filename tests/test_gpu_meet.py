"""The bounded meeting of the blocks of a launch: all pass while everyone arrives; when a wait
runs out (one arrival more is asked for than there are blocks) every block returns in time,
in that round, with the failure flag set, and the context stays usable."""
import ctypes as C
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1202_2355_gb300 import build
    so = str(tmp_path_factory.mktemp("meet") / "libmeet.so")
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", build.ARCH, "-Xcompiler", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_1202_2355_gb300", "csrc"), "-o", so,
                    os.path.join(ROOT, "tests", "kernels", "meet_check.cu")], check=True)
    return C.CDLL(so)


def _meet(lib, blocks, rounds, miss, limit):
    passed, failed = (C.c_int * blocks)(), C.c_uint(99)
    assert lib.meet_check(blocks, rounds, miss, C.c_uint(limit), passed, C.byref(failed)) == 0
    return list(passed), failed.value


@pytest.mark.parametrize("blocks", [1, 2, 152, 304])
def test_meetings_come_about_or_run_out(lib, blocks):
    assert _meet(lib, blocks, 200, -1, 1 << 22) == ([200] * blocks, 0)
    for miss in (0, 3, 199):
        assert _meet(lib, blocks, 200, miss, 1 << 13) == ([miss] * blocks, 1)
    assert _meet(lib, blocks, 5, -1, 1 << 22) == ([5] * blocks, 0)
