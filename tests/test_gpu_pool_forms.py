"""A pool's members solve kernel by kernel where a context of their size solves in one launch: a block's
partial sums, the order in which the rows are added and every node's operations are the same, so the
fields are the same bits (the smallest grids, each number of planes a block, the last grids in one launch).
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2411_06563_gb300.hosc")
from paper_2411_06563_gb300 import inputs  # noqa: E402
from paper_2411_06563_gb300 import serve as S  # noqa: E402

FIELDS = (("u", H.HOSC_U), ("v", H.HOSC_V), ("w", H.HOSC_W), ("th", H.HOSC_THETA), ("p", H.HOSC_P))
FP64, MIXED = H.HOSC_FP64, H.HOSC_MIXED


@pytest.mark.parametrize("N,precision,solver,Lz", [
    (5, FP64, 0, 1.0), (12, FP64, 0, 1.3), (21, FP64, 0, 1.0), (31, FP64, 0, 1.0), (37, FP64, 0, 0.8),
    (42, FP64, 0, 1.0), (43, FP64, 0, 1.0), (5, FP64, 1, 1.0), (14, FP64, 1, 0.7), (21, FP64, 1, 1.0),
    (34, FP64, 1, 1.4), (42, FP64, 1, 1.0), (5, MIXED, 0, 1.0), (41, MIXED, 0, 1.2),
    (68, MIXED, 0, 1.0)])
def test_member_equals_one_launch_context(N, precision, solver, Lz):
    p = H.hosc_default_params(N, 1e4, 1.0, 0.75)
    p.dt = 0.002
    p.lambda_ = min(0.25 / (N - 1) ** 2 / p.dt, 0.1)
    p.precision, p.solver, p.Lz = precision, solver, Lz
    p.max_lin_iter = 3000
    p.auto_defect = 0
    p.tol_steady = 1e-12
    st = inputs.cavity_state(N, 1e4, seed=N)
    G = 2
    with S.Pool(H.hosc_workspace_bytes(p) + 1, G, H.HOSC_POOL_GRAPH, False) as pool:
        slot = pool.admit(p, 100)
        ctx = H.hosc_pool_result(pool.h, slot)[4]
        for name, which in FIELDS:
            assert H.hosc_set_field(ctx, which, np.ascontiguousarray(st[name])) == 0
        pool.run(1)
        member = pool.result(slot, FIELDS)
    with H.Cavity(p) as cav:
        for name, which in FIELDS:
            cav.set(which, st[name])
        info = cav.step(G)
        assert info["call_status"] == 0
        assert info["last_iters"] == member["info"]["last_iters"]
        for name, which in FIELDS:
            assert np.array_equal(cav.get(which), member[name]), name
