"""The one-launch solve, whose blocks wait for one another, beside other work on the GPU: a step waits for
blocks that cannot start yet, however long other kernels keep the SMs (a wait's limit counts from when
every block runs), and contexts that step at once do not disturb one another.
"""

import ctypes
import os
import subprocess
import threading
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2411_06563_gb300.hosc")
from paper_2411_06563_gb300 import build, inputs  # noqa: E402

FIELDS = (("u", H.HOSC_U), ("v", H.HOSC_V), ("w", H.HOSC_W), ("th", H.HOSC_THETA), ("p", H.HOSC_P))
FP64, MIXED = H.HOSC_FP64, H.HOSC_MIXED
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def hold(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("hold") / "libhold.so")
    subprocess.run([build.nvcc()] + build.ARCH + ["-shared", "-cudart", "static", "-Xcompiler", "-fPIC",
                    os.path.join(HERE, "hold_sms.cu"), "-o", out], check=True, timeout=300)
    return ctypes.CDLL(out).hold_sms


def _cavity(N, precision, solver):
    p = H.hosc_default_params(N, 1e4, 1.0, 0.75)
    p.dt = 0.002
    p.lambda_ = min(0.25 / (N - 1) ** 2 / p.dt, 0.1)
    p.precision, p.solver, p.auto_defect = precision, solver, 0
    cav = H.Cavity(p)
    st = inputs.cavity_state(N, 1e4, seed=N)
    for name, which in FIELDS:
        cav.set(which, st[name])
    return cav


@pytest.mark.parametrize("N,precision,solver", [(21, FP64, 0), (41, FP64, 0), (34, FP64, 1),
                                                (64, MIXED, 0)])
def test_a_step_waits_for_the_sms(hold, N, precision, solver):
    """3 s with two SMs left (the limit of a wait is 2 s): the step takes them and is the same."""
    out = []
    for ms in (0, 3000):
        cav = _cavity(N, precision, solver)
        assert cav.step(1)["call_status"] == 0   # the captured step is there
        assert cav.step(1)["call_status"] == 0
        t0 = time.perf_counter()
        if ms:
            assert hold(2, ms) == 0
            time.sleep(0.1)
        st, _ = H.hosc_step(cav.h, 1)
        took = time.perf_counter() - t0
        assert st == H.HOSC_OK
        assert took > 2.5 or not ms   # it did need the SMs that were held
        out.append({name: cav.get(which) for name, which in FIELDS})
        cav.close()
    for name, _ in FIELDS:
        assert np.array_equal(out[0][name], out[1][name]), name


def test_contexts_stepped_at_once_by_threads():
    """Eight contexts, one thread and stream each, step as they do alone."""
    kinds = [(21, FP64, 0), (13, MIXED, 0), (41, MIXED, 0), (14, FP64, 1)] * 2
    alone = []
    for k in kinds[:4]:
        cav = _cavity(*k)
        assert cav.step(40)["call_status"] == 0
        alone.append({name: cav.get(which) for name, which in FIELDS})
        cav.close()
    cavs = [_cavity(*k) for k in kinds]
    status = [None] * len(cavs)

    def run(i):
        status[i] = [H.hosc_step(cavs[i].h, 1)[0] for _ in range(20)] + [H.hosc_step(cavs[i].h, 20)[0]]

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(cavs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i, cav in enumerate(cavs):
        assert status[i] == [0] * 21
        for name, which in FIELDS:
            assert np.array_equal(cav.get(which), alone[i % 4][name]), (i, name)
        cav.close()
