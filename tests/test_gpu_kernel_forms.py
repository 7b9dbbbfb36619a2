"""Kernels in forms that no public call leads to on this GPU (kernel_forms.cu, linked with the library's
objects)."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2411_06563_gb300.hosc")
torch = pytest.importorskip("torch")
from paper_2411_06563_gb300 import build, inputs  # noqa: E402

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
    lib = ctypes.CDLL(out)
    lib.flat_xr_walls.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_int]
    lib.hosc_bicgstab_noalloc.argtypes = H.lib().hosc_bicgstab_noalloc.argtypes
    return lib


@pytest.mark.parametrize("N", [5, 12, 70])
@pytest.mark.parametrize("first", [0, 1])
@pytest.mark.parametrize("alpha,omega", [(0.5, 0.25), (1e39, 0.25), (0.5, -1e39), (float("nan"), 1.0),
                                         (1e39, float("nan"))])
def test_flat_xr_leaves_the_walls_zero(forms, N, first, alpha, omega):
    """The stream passes over the i and j walls, which hold zeros that the stencil kernels read in every
    later solve: they stay zero also with scalars beyond float or not finite (a solve that fails)."""
    assert forms.flat_xr_walls(N, alpha, omega, first) == 0


FIELDS = (("u", H.HOSC_U), ("v", H.HOSC_V), ("w", H.HOSC_W), ("th", H.HOSC_THETA), ("p", H.HOSC_P))


def _solve(lib, N, w, rhs, fill, tol, max_iter):
    """Status, iterations and increments of lib's allocation-free solve; fill: the walls of rhs."""
    wall = np.ones((N, N, N), bool)
    wall[1:-1, 1:-1, 1:-1] = False
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
           for a in w + [np.where(wall, fill, r) for r in rhs]]
    x = [torch.full((N, N, N), 7.0, dtype=torch.float64, device="cuda") for _ in range(4)]
    torch.cuda.synchronize()
    ptr = lambda ts: (ctypes.c_void_p * len(ts))(*[t.data_ptr() for t in ts])  # noqa: E731
    its = (ctypes.c_int * 4)()
    st = lib.hosc_bicgstab_noalloc(N, ptr(dev[:14]), ptr(dev[14:]), ptr(x), tol, max_iter, its, None)
    torch.cuda.synchronize()
    return st, list(its), [t.cpu().numpy() for t in x]


@pytest.mark.parametrize("N", [5, 16, 21, 37, 41])
def test_allocation_free_solve_kernel_by_kernel(forms, N):
    """Where no shape fits one launch: the solve ends at the residual that it was asked for (the recursion's
    and the true one differ by some roundings of the right-hand side, 1e-14) and within 1e-9 of the one-launch
    form, the parity tolerance of the FP64 solve; twice on the same scratch; it reads no wall of the caller's
    right-hand sides and writes none of x. (Sums grouped by another shape may end some iterations apart.)"""
    st = inputs.cavity_state(N, 1e4, seed=N)
    p = H.hosc_default_params(N, 1e4, 1.0, 0.8)
    p.dt = 0.003
    p.lambda_ = 0.25 / (N - 1) ** 2 / p.dt
    with H.Cavity(p) as cav:
        for name, which in FIELDS:
            cav.set(which, st[name])
        for stage in (H.HOSC_STAGE_VISCOSITY, H.HOSC_STAGE_SOURCES, H.HOSC_STAGE_RHS):
            cav.run_stage(stage)
        w = [cav.get(H.HOSC_A_MOM + q) for q in range(7)] + \
            [cav.get(H.HOSC_A_ENE + q) for q in range(7)]
        rhs = [cav.get(H.HOSC_RHS_U + s) for s in range(4)]
    one = _solve(H.lib(), N, w, rhs, 0.0, 1e-11, 2000)
    apart = _solve(forms, N, w, rhs, 0.0, 1e-11, 2000)
    again = _solve(forms, N, w, rhs, 1e30, 1e-11, 2000)
    assert one[0] == apart[0] == again[0] == H.HOSC_OK
    assert apart[1] == again[1]
    inner = (slice(1, -1),) * 3
    steps = [(0, 0, 0), (0, 0, 1), (0, 0, -1), (0, 1, 0), (0, -1, 0), (1, 0, 0), (-1, 0, 0)]
    for s in range(4):
        o = np.zeros((N, N, N))
        o[inner] = apart[2][s][inner]
        res = rhs[s][inner] - sum(w[q + (7 if s == 3 else 0)][inner] *
                                  np.roll(o, [-d for d in steps[q]], (0, 1, 2))[inner]
                                  for q in range(7))
        assert np.linalg.norm(res) <= (1e-11 + 1e-14) * np.linalg.norm(rhs[s][inner])
    for a, b, c in zip(one[2], apart[2], again[2]):
        assert np.array_equal(b, c)
        assert np.max(np.abs(a[inner] - b[inner])) <= 1e-9 * np.max(np.abs(a[inner]))
        b = b.copy()
        b[inner] = 7.0
        assert np.all(b == 7.0)
    # the limit of iterations is kept, and reported
    st_, its, _ = _solve(forms, N, w, rhs, 0.0, 1e-14, 1)
    assert st_ == H.HOSC_ENOCONV and its == [1, 1, 1, 1]
