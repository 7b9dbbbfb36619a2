"""Kernels in forms that no public call leads to on this GPU (kernel_forms.cu, linked with the library's
objects)."""

import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2411_06563_gb300.hosc")
from paper_2411_06563_gb300 import build  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    objs = [os.path.join(build.BUILD, "hosc_%s.o" % n) for n in ("noalloc", "krylov", "tma", "step")]
    assert all(os.path.exists(o) for o in objs), "the library's objects: build it first"
    out = str(tmp_path_factory.mktemp("forms") / "libforms.so")
    subprocess.run([build.nvcc()] + build.ARCH + ["-std=c++17", "-shared", "-cudart", "static",
                    "-Xcompiler", "-fPIC", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                    os.path.join(HERE, "kernel_forms.cu")] + objs +
                   ["-Xlinker", "-Bsymbolic", "-o", out], check=True, timeout=300)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("N", [5, 12, 70])
@pytest.mark.parametrize("first", [0, 1])
@pytest.mark.parametrize("alpha,omega", [(0.5, 0.25), (1e39, 0.25), (0.5, -1e39), (float("nan"), 1.0),
                                         (1e39, float("nan"))])
def test_flat_xr_leaves_the_walls_zero(forms, N, first, alpha, omega):
    """The stream passes over the i and j walls, which hold zeros that the stencil kernels read in every
    later solve: they stay zero also with scalars beyond float or not finite (a solve that fails)."""
    forms.flat_xr_walls.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_int]
    assert forms.flat_xr_walls(N, alpha, omega, first) == 0
