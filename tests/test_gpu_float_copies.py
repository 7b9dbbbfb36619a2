"""FP32 sweeps read float copies of the state. A step keeps copies up to date that were valid before
it; copies that were not (a fresh state stepped by FP64 defect sweeps, which do not read them) are
made anew before the first FP32 sweep. Here a state goes through one defect step by each path that a
step can take, then through one step of FP32 sweeps, against a context that takes that last step from
the same state: the same kernels on the same values, so the same bits.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2411_06563_gb300.hosc")
from paper_2411_06563_gb300 import inputs  # noqa: E402
from paper_2411_06563_gb300 import serve as S  # noqa: E402

FIELDS = (("u", H.HOSC_U), ("v", H.HOSC_V), ("w", H.HOSC_W), ("th", H.HOSC_THETA), ("p", H.HOSC_P))
N = 17


def _params(**kw):
    p = H.hosc_default_params(N, 1e4, 1.0, 0.75)
    p.dt = 0.002
    p.lambda_ = 0.1
    p.precision = H.HOSC_MIXED
    p.use_history = 0
    p.auto_defect = 0
    p.tol_steady = 1e-12
    for k, v in kw.items():
        setattr(p, k, v)
    return p


def _state(seed):
    st = inputs.cavity_state(N, 1e4, seed=seed)
    st["th"][:, :, 0], st["th"][:, :, -1] = 0.75, 0.25   # not the walls of the initial state
    return st


def _fields(cav):
    return {name: cav.get(which) for name, which in FIELDS}


def _last_step(p, state):
    with H.Cavity(p) as cav:
        for name, which in FIELDS:
            cav.set(which, state[name])
        assert cav.step(1)["call_status"] == 0
        return _fields(cav)


# tol_div above every divergence: no step corrects the pressure, so that none writes it
@pytest.mark.parametrize("tol_div", [1e-6, 1e9])
@pytest.mark.parametrize("path", ["captured", "staged", "timed", "inner"])
def test_sweeps_after_a_defect_step_of_a_new_state(path, tol_div):
    p = _params(inner_max=1 if path == "inner" else 0, tol_div=tol_div)
    st = _state(11)
    with H.Cavity(p) as cav:
        for name, which in FIELDS:
            cav.set(which, st[name])
        assert H.hosc_set_phase(cav.h, 1) == 0
        if path == "staged":
            for stage in range(5):
                cav.run_stage(stage)
        else:
            H.hosc_profile_enable(cav.h, path == "timed")
            assert cav.step(1)["call_status"] == 0
            H.hosc_profile_enable(cav.h, 0)
        mid = _fields(cav)
        assert H.hosc_set_phase(cav.h, 0) == 0
        assert cav.step(1)["call_status"] == 0
        got = _fields(cav)
    ref = _last_step(p, mid)
    for name, _ in FIELDS:
        assert np.array_equal(got[name], ref[name]), name


@pytest.mark.parametrize("mode", [H.HOSC_POOL_STREAMS, H.HOSC_POOL_GRAPH])
def test_pool_member_back_from_defect_sweeps(mode):
    p = _params()
    st = _state(12)
    G = 2
    with S.Pool(H.hosc_workspace_bytes(p) + 1, G, mode, False) as pool:
        slot = pool.admit(p, 100)
        ctx = H.hosc_pool_result(pool.h, slot)[4]
        for name, which in FIELDS:
            assert H.hosc_set_field(ctx, which, np.ascontiguousarray(st[name])) == 0
        assert H.hosc_set_phase(ctx, 1) == 0
        pool.run(1)
        mid = pool.result(slot, FIELDS)
        assert H.hosc_set_phase(ctx, 0) == 0
        pool.run(1)
        got = pool.result(slot, FIELDS)
    with H.Cavity(p) as cav:
        for name, which in FIELDS:
            cav.set(which, mid[name])
        assert cav.step(G)["call_status"] == 0
        ref = _fields(cav)
    for name, _ in FIELDS:
        assert np.array_equal(got[name], ref[name]), name
