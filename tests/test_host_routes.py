"""The host code that chooses, captures and launches the kernels, on a device played on the host
(fake_device.cpp): which kernels a call leads to, and what becomes of a launch that is refused."""

import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2411_06563_gb300 import hosc as H

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2411_06563_gb300", "csrc")
FP64, MIXED = H.HOSC_FP64, H.HOSC_MIXED


@pytest.fixture(scope="module")
def fake_path(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("no C++ compiler or CUDA headers")
    out = str(tmp_path_factory.mktemp("fake") / "libhosc_fake.so")
    subprocess.run(["g++", "-x", "c++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I",
                    "/usr/local/cuda/include", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    os.path.join(CSRC, "hosc_api.cu"), os.path.join(CSRC, "hosc_pool.cu"),
                    os.path.join(ROOT, "tests", "fake_device.cpp"), "-Wl,-Bsymbolic", "-o", out],
                   check=True, timeout=300)
    return out


class Fake:
    def __init__(self, lib):
        self.lib = lib
        lib.fake_log.restype = ctypes.c_char_p
        lib.fake_cost.argtypes = [ctypes.c_char_p, ctypes.c_double]

    def log(self):
        return self.lib.fake_log().decode().split("\n")[:-1]

    def clear(self):
        self.lib.fake_clear()

    def refuse(self, name, launches=-1):
        self.lib.fake_refuse(name.encode(), launches)

    def cost(self, name, ms):
        self.lib.fake_cost(name.encode(), ms)


@pytest.fixture()
def fake(fake_path, monkeypatch):
    monkeypatch.setattr(H, "LIB_PATH", fake_path)
    monkeypatch.setattr(H, "_lib", None)
    H.lib().fake_reset()
    return Fake(H.lib())


def _params(N, precision, **kw):
    p = H.hosc_default_params(N, 1e4, 1.0, 0.75)
    p.precision = precision
    p.use_history = 0
    for k, v in kw.items():
        setattr(p, k, v)
    return p


# ------------------------------------------------------------------ refused launches

# one launch (FP64, mixed, BiCGSTAB(2)), planar and register kernels in the loop
STEPS = [(21, FP64, 0, "arm viscosity sources rhs solve update"),
         (30, MIXED, 0, "arm shadow viscosity sources rhs solve update"),
         (21, FP64, 1, "solve update"),
         (50, FP64, 0, "arm viscosity sources rhs pv st xr loop update"),
         (50, FP64, 1, "b2 loop update"),
         (75, MIXED, 0, "arm shadow viscosity sources rhs pv st xr loop update")]


@pytest.mark.parametrize("N,precision,solver,name",
                         [(N, pr, so, n) for N, pr, so, names in STEPS for n in names.split()])
def test_a_refused_launch_fails_the_step(fake, N, precision, solver, name):
    """No step is reported that ran without one of its launches; the next call, launched kernel by
    kernel where the capture failed, is whole again."""
    with H.Cavity(_params(N, precision, solver=solver)) as cav:
        fake.refuse(name, 1)
        st, info = H.hosc_step(cav.h, 2)
        assert st == H.HOSC_ECUDA and info.steps == 0
        fake.clear()
        st, info = H.hosc_step(cav.h, 2)
        assert st == H.HOSC_OK and info.steps == 2
        ran = [line.split()[0] for line in fake.log()]
        assert "update" in ran
        for q in ("viscosity", "sources", "rhs"):
            assert ran.count(q) == 2
        if precision == MIXED and name in ("arm", "shadow"):
            assert "shadow" in ran   # the float copies that the refused call did not make


@pytest.mark.parametrize("mode", [H.HOSC_POOL_STREAMS, H.HOSC_POOL_GRAPH])
@pytest.mark.parametrize("name", ["arm", "pv", "update"])
def test_a_refused_launch_fails_the_round(fake, mode, name):
    p = _params(30, MIXED)
    st, pool = H.hosc_pool_create(H.hosc_workspace_bytes(p) + 1, 2, mode, 0)
    assert st == 0 and H.hosc_pool_admit(pool, p, 100)[0] == 0
    fake.refuse(name, 1)
    assert H.hosc_pool_run(pool, 1)[0] == H.HOSC_ECUDA
    H.hosc_pool_destroy(pool)


def test_an_older_error_is_not_the_steps(fake):
    """An error that an earlier call left behind does not fail a step that ran."""
    with H.Cavity(_params(21, FP64)) as cav, H.Cavity(_params(21, FP64)) as other:
        fake.refuse("diagnostics", 1)
        fake.refuse("finish", 1)
        assert H.hosc_diagnostics(other.h, 21)[0] == H.HOSC_ECUDA
        assert H.hosc_step(cav.h, 1)[0] == H.HOSC_OK


def test_outcome_of_a_system(tmp_path):
    """A system whose solve did not end is no success (one left open by the host's last iteration of
    the merged form is, as its residual tells)."""
    src = tmp_path / "outcome.cpp"
    src.write_text(r"""
#include <cuda_runtime.h>
#include <stdio.h>
#include <string.h>
#include "hosc.h"
#include "hosc_internal.h"
int main() {
  struct { int done, status; double r0; int merged; } c[] = {
      {1, 0, 1, 0}, {1, 0, 0, 0}, {1, HOSC_ENOCONV, 1, 0}, {1, HOSC_ECUDA, 1, 0}, {0, 0, 0, 0},
      {0, 0, 1, 0}, {0, 0, 1, 1}, {0, 0, 0, 1}};
  for (auto& q : c) {
    hosc::KrylovScalars k;
    memset(&k, 0, sizeof(k));
    k.done = q.done, k.status = q.status, k.r0norm = q.r0;
    printf("%d ", hosc::system_status(k, q.merged));
  }
}
""")
    exe = str(tmp_path / "outcome")
    subprocess.run(["g++", "-std=c++17", "-I", "/usr/local/cuda/include", "-I",
                    os.path.join(ROOT, "include"), "-I", CSRC, str(src), "-o", exe], check=True,
                   timeout=120)
    out = [int(v) for v in subprocess.run([exe], check=True, capture_output=True, text=True,
                                          timeout=60).stdout.split()]
    OK, NO, EC = H.HOSC_OK, H.HOSC_ENOCONV, H.HOSC_ECUDA
    assert out == [OK, OK, NO, EC, EC, EC, OK, EC]


# ------------------------------------------------------------------ launch shapes

def _step_forms(fake, cav):
    """The Krylov form of each launch of one step: 'pv register 384x8', ..."""
    fake.clear()
    assert H.hosc_step(cav.h, 1)[0] == 0
    return sorted({" ".join(line.split()[:2]) for line in fake.log()
                   if line.split()[0] in ("solve", "pv", "init")})


@pytest.mark.parametrize("N", [30, 69, 75, 104])
def test_merged_form_of_a_new_context(fake, N):
    """The merged form is taken at the default shape, whatever that is, and the default is back with
    the three-kernel form."""
    with H.Cavity(_params(N, MIXED)) as cav:
        default = H.hosc_get_tiles(cav.h)
        assert H.hosc_set_krylov_merged(cav.h, 1) == 0 and H.hosc_get_krylov_merged(cav.h) == 1
        assert H.hosc_get_tiles(cav.h)[1] <= 256
        assert _step_forms(fake, cav) == ["init merged", "pv merged"]
        assert H.hosc_set_krylov_merged(cav.h, 0) == 0
        assert H.hosc_get_tiles(cav.h) == default
        assert H.hosc_set_tiles(cav.h, 384, 1) == 0
        assert H.hosc_set_krylov_merged(cav.h, 1) == H.HOSC_EINVAL   # the caller's shape stays
        assert H.hosc_get_tiles(cav.h)[1:] == (384, 1, 0) and H.hosc_get_krylov_merged(cav.h) == 0


# a call of each kind that selects nothing
IDLE = [("hosc_set_xr_form", (0,)), ("hosc_set_stencil_tiles", (0, 0, 0)),
        ("hosc_set_tma_tiles", (0, 0, 3, 3)), ("hosc_set_krylov_merged", (0,))]
# one that selects a form, and the one that undoes it
SELECT = [("hosc_set_xr_form", (1,), (0,)), ("hosc_set_stencil_tiles", (16, 2, 5), (0, 0, 0)),
          ("hosc_set_krylov_merged", (1,), (0,))]


@pytest.mark.parametrize("N,precision,default", [(21, FP64, "solve one_launch"),
                                                 (30, MIXED, "solve one_launch"),
                                                 (75, MIXED, "pv register"),
                                                 (104, MIXED, "pv plane")])
def test_calls_that_select_nothing_keep_the_default_kernels(fake, N, precision, default):
    with H.Cavity(_params(N, precision)) as cav:
        assert _step_forms(fake, cav) == [default]
        for name, args in IDLE:
            assert getattr(H, name)(cav.h, *args) == 0
            assert _step_forms(fake, cav) == [default], name
        assert H.hosc_set_xr_form(cav.h, 2) == H.HOSC_EINVAL
        assert H.hosc_set_tiles(cav.h, 100, 1) == H.HOSC_EINVAL
        assert _step_forms(fake, cav) == [default]
        for name, on, off in SELECT:
            assert getattr(H, name)(cav.h, *on) == 0
            forms = _step_forms(fake, cav)
            if precision == FP64:
                assert forms == [default], name   # FP64 kernels take no setting
            elif name == "hosc_set_xr_form":
                assert forms == [default.replace("solve one_launch", "pv register")]
            else:
                assert default not in forms, name
            assert getattr(H, name)(cav.h, *off) == 0
            assert _step_forms(fake, cav) == [default], name
        _, b, z, narrow = H.hosc_get_tiles(cav.h)
        assert H.hosc_set_tiles(cav.h, b, z, narrow) == 0
        assert _step_forms(fake, cav) == [default if precision == FP64 else "pv register"]


# ------------------------------------------------------------------ shapes in a pool

def _round_forms(fake, pool):
    """p/v lines of one round, with their counts."""
    fake.clear()
    assert H.hosc_pool_run(pool, 1)[0] == 0
    pv = [line for line in fake.log() if line.startswith("pv ")]
    return {q: pv.count(q) for q in pv}


def _pool(N, members, mode, **kw):
    p = _params(N, MIXED, **kw)
    st, pool = H.hosc_pool_create(4 * H.hosc_workspace_bytes(p), 2, mode, 1)
    assert st == 0
    slots = [H.hosc_pool_admit(pool, p, 1000) for _ in range(members)]
    assert all(s[0] == 0 for s in slots)
    return p, pool, [s[1] for s in slots]


@pytest.mark.parametrize("mode", [H.HOSC_POOL_STREAMS, H.HOSC_POOL_GRAPH])
@pytest.mark.parametrize("N,best,flat", [(104, "plane", False), (104, "register", False),
                                         (104, "staged", False), (75, "merged", False),
                                         (75, "register", True), (104, "plane", True),
                                         (30, "staged", False)])
def test_a_tuned_form_reaches_every_member(fake, mode, N, best, flat):
    """The member that a size is tuned on, one that was there and one admitted later run, round after
    round, the form and the tiles that the search found the fastest."""
    for kind in ("pv", "st"):
        fake.cost("%s %s" % (kind, best), 0.125)
    if flat:
        fake.cost("xr_flat", 0.125)
    p, pool, slots = _pool(N, 2, mode)
    _round_forms(fake, pool)
    one = _round_forms(fake, pool)
    assert len(one) == 1, one
    (line, count), = one.items()
    assert line.split()[1] == best and (line.endswith(" flat") == flat), line
    assert H.hosc_pool_admit(pool, p, 1000)[0] == 0
    for _ in range(2):
        more = _round_forms(fake, pool)
        assert list(more) == [line] and more[line] == count * 3 // 2
    H.hosc_pool_destroy(pool)


@pytest.mark.parametrize("merged,plane,expect", [(0.5, 0.125, "plane"), (0.125, 0.5, "merged"),
                                                 (0.75, 2.0, "merged"), (2.0, 2.0, "register")])
def test_the_search_keeps_the_faster_of_merged_form_and_shared_planes(fake, merged, plane, expect):
    for kind in ("pv", "st"):
        fake.cost("%s merged" % kind, merged)
        fake.cost("%s plane" % kind, plane)
        fake.cost("%s staged" % kind, 4.0)
        for z in range(1, 34):   # a block that the merged form takes is the fastest
            fake.cost("%s register 256x%d" % (kind, z), 0.9)
    with H.Cavity(_params(104, MIXED)) as cav:
        assert cav.step(1)["call_status"] == 0
        assert H.hosc_autotune(cav.h, 2)[0] == 0
        assert [q.split()[1] for q in _step_forms(fake, cav) if q.startswith("pv")] == [expect]


def test_a_captured_round_follows_the_form(fake):
    """A form that changes without its tiles makes the pool capture its round again."""
    p, pool, slots = _pool(104, 1, H.HOSC_POOL_GRAPH)
    H.hosc_pool_destroy(pool)
    st, pool = H.hosc_pool_create(4 * H.hosc_workspace_bytes(p), 2, H.HOSC_POOL_GRAPH, 0)
    assert st == 0 and H.hosc_pool_admit(pool, p, 1000)[0] == 0
    ctx = H.hosc_pool_result(pool, 0)[4]
    assert {q.split()[1] for q in _round_forms(fake, pool)} == {"plane"}
    assert H.hosc_set_tiles(ctx, *H.hosc_get_tiles(ctx)[1:]) == 0
    assert {q.split()[1] for q in _round_forms(fake, pool)} == {"register"}
    H.hosc_pool_destroy(pool)
