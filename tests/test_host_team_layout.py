"""Where a team keeps its adjoint arrays, for every size of the recomputed
block: one after the other, none over another."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

from paper_2312_02836_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc"))
    if nvcc is None:
        pytest.skip("no nvcc")
    out = str(tmp_path_factory.mktemp("layout") / "liblayout.so")
    subprocess.check_call([nvcc] + build.ARCH + ["-O1", "-std=c++17", "-Xcompiler", "-fPIC",
                           "-shared", "-I", os.path.join(ROOT, "include"),
                           os.path.join(HERE, "host", "team_layout.cu"), "-o", out])
    fn = C.CDLL(out).layout

    def run(*a):
        v = (C.c_longlong * 10)()
        fn(*a, v)
        return list(v)

    return run


@pytest.mark.parametrize("n,R,heat", [(13, 12, 0), (14, 12, 1), (48, 180, 0), (129, 600, 1)])
@pytest.mark.parametrize("K", [1, 64])
@pytest.mark.parametrize("S", [0, 32])
@pytest.mark.parametrize("stride", [1, 16, 2**20, 2**27, 2**31 - 1])
def test_adjoint_arrays_do_not_overlap(layout, n, R, heat, K, S, stride):
    at = layout(n, R, heat, K, stride, S)
    need = [7 * K * n, 7 * K, K * R, K, K * (n if S else 3 * n), n, stride * n, K,
            0 if heat else (1 if S else K) * R]
    for a, size, b in zip(at, need, at[1:]):
        assert a >= 0 and b >= a + size
