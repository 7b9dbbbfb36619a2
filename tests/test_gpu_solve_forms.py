"""The forms that a step may take for the same arithmetic, and where the choice between them lies.

One launch against one launch a phase (the solve of grids that fit on the chip): a block's partial
sums, the order in which the rows are added and every node's operations are the same, so the fields
are the same bits. The shared-plane p/v and s/t kernels against the register kernels add the rows in
another grouping: the solves stop at a relative residual of 3e-6 either way, and the increments agree
as two FP32 solves do (2e-5 of the increment's size, as against the oracle). Maxima do not depend on
an order: equal. The viscosity is held to the oracle at 1e-13, the parity tolerance.
"""

import numpy as np
import pytest

from oracle import hosc_oracle as O

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2411_06563_gb300.hosc")
torch = pytest.importorskip("torch")
from paper_2411_06563_gb300 import inputs  # noqa: E402

FIELDS = (("u", H.HOSC_U), ("v", H.HOSC_V), ("w", H.HOSC_W), ("th", H.HOSC_THETA), ("p", H.HOSC_P))
FP64, MIXED = H.HOSC_FP64, H.HOSC_MIXED


def _params(N, Ra, n, precision, **kw):
    p = H.hosc_default_params(N, Ra, 1.0, n)
    p.dt = 0.002
    p.lambda_ = min(0.25 / (N - 1) ** 2 / p.dt, 0.1)
    p.precision = precision
    p.max_lin_iter = 3000
    for k, v in kw.items():
        setattr(p, k, v)
    return p


def _run(p, st, steps, chosen):
    """Fields and info after the steps; chosen: the default launch shape set by the caller."""
    with H.Cavity(p) as cav:
        if chosen:
            _, b, z, narrow = H.hosc_get_tiles(cav.h)
            assert H.hosc_set_tiles(cav.h, b, z, narrow) == H.HOSC_OK
        for name, which in FIELDS:
            cav.set(which, st[name])
        info = cav.step(steps)
        assert info["call_status"] == 0
        return {name: cav.get(which) for name, which in FIELDS}, info


# the smallest grids, each number of planes a block, the last grids in one launch and the first beyond
@pytest.mark.parametrize("N,precision,solver,Lz,inner", [
    (5, FP64, 0, 1.0, 1), (12, FP64, 0, 1.3, 1), (21, FP64, 0, 1.0, 3), (31, FP64, 0, 1.0, 1),
    (37, FP64, 0, 0.8, 1), (42, FP64, 0, 1.0, 1), (43, FP64, 0, 1.0, 1),
    (5, FP64, 1, 1.0, 1), (14, FP64, 1, 0.7, 1), (21, FP64, 1, 1.0, 3), (34, FP64, 1, 1.4, 1),
    (42, FP64, 1, 1.0, 1),
    (5, MIXED, 0, 1.0, 1), (12, MIXED, 0, 1.0, 3), (41, MIXED, 0, 1.2, 1), (64, MIXED, 0, 1.0, 1),
    (68, MIXED, 0, 1.0, 1), (70, MIXED, 0, 1.0, 1)])
def test_one_launch_solve_equals_kernel_by_kernel(N, precision, solver, Lz, inner):
    p = _params(N, 1e4, 0.75, precision, solver=solver, Lz=Lz, inner_max=inner)
    st = inputs.cavity_state(N, 1e4, seed=N)
    one, i1 = _run(p, st, 2, False)
    apart, i2 = _run(p, st, 2, True)
    assert i1["last_iters"] == i2["last_iters"] and i1["res"] == i2["res"]
    for name, _ in FIELDS:
        assert np.array_equal(one[name], apart[name]), name


@pytest.mark.parametrize("N,precision,solver", [(9, FP64, 1), (33, FP64, 1), (41, FP64, 0),
                                                (30, MIXED, 0)])
def test_zero_right_hand_sides_in_one_launch(N, precision, solver):
    """Ra = 0 and theta = 1 - x: no system iterates and the increments written are zero."""
    p = _params(N, 0.0, 0.75, precision, solver=solver)
    th = np.broadcast_to(1.0 - np.linspace(0, 1, N), (N, N, N)).copy()
    with H.Cavity(p) as cav:
        cav.set(H.HOSC_THETA, th)
        info = cav.step(2)
        assert info["call_status"] == 0 and info["last_iters"][:3] == [0, 0, 0]
        assert np.max(np.abs(cav.get(H.HOSC_V))) == 0.0
        assert np.max(np.abs(cav.get(H.HOSC_U))) == 0.0


@pytest.mark.parametrize("N", [103, 104, 107])
def test_shared_plane_kernels_against_register_kernels(N):
    """The grids around the line between them (at 103 both runs take the register kernels)."""
    p = _params(N, 1e4, 0.75, MIXED)
    st = inputs.cavity_state(N, 1e4, seed=N)
    plane, _ = _run(p, st, 1, False)
    regs, _ = _run(p, st, 1, True)
    for name, _ in FIELDS[:4]:
        scale = max(np.max(np.abs(regs[name] - st[name])), 1e-12)
        assert np.max(np.abs(plane[name] - regs[name])) <= 2e-5 * scale, name


@pytest.mark.parametrize("N", [50, 52])
def test_maximum_over_the_rows_of_a_launch(N):
    """488 rows of partials (added by one block) and 550 (in two levels): the largest increment and
    the largest change of theta on the adiabatic walls are the step's reported change, exactly."""
    p = _params(N, 1e4, 0.75, FP64)
    st = inputs.cavity_state(N, 1e4, seed=N)
    with H.Cavity(p) as cav:
        for name, which in FIELDS:
            cav.set(which, st[name])
        for stage in (H.HOSC_STAGE_VISCOSITY, H.HOSC_STAGE_SOURCES, H.HOSC_STAGE_RHS,
                      H.HOSC_STAGE_SOLVE):
            cav.run_stage(stage)
        dx = max(np.max(np.abs(cav.get(w)[1:-1, 1:-1, 1:-1])) for w in
                 (H.HOSC_DX_U, H.HOSC_DX_V, H.HOSC_DX_W, H.HOSC_DX_THETA))
        info = cav.run_stage(H.HOSC_STAGE_UPDATE)
        th = np.abs(cav.get(H.HOSC_THETA) - st["th"])
        th[1:-1, 1:-1, 1:-1] = 0.0
        assert info["res"] == max(dx, np.max(th))


@pytest.mark.parametrize("n", [1.5, 0.5, 0.75, 1.25, 0.9, 1.1, 0.8, 0.96875, 0.97, 0.7123, 1.9])
def test_viscosity_root_and_general_exponents(n):
    """2/|n-1| a whole number up to 64 (a root by Newton steps; 0.96875 gives 64) and the others."""
    N = 9
    p = _params(N, 1e4, n, FP64)
    st = inputs.cavity_state(N, 1e4, seed=3)
    op = O.Params(N=N, Ra=1e4, n=n, dt=p.dt, theta_ref=p.theta_ref, I2_eps=p.I2_eps, phi=p.phi)
    ref = O.viscosity(st["u"], st["v"], st["w"], op)[0]
    with H.Cavity(p) as cav:
        for name, which in FIELDS:
            cav.set(which, st[name])
        cav.run_stage(H.HOSC_STAGE_VISCOSITY)
        got = cav.get(H.HOSC_ETA)
    assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))


@pytest.mark.parametrize("N", [5, 16, 37])
def test_noalloc_solve_reads_no_wall_of_the_callers_arrays(N):
    """The right-hand sides' walls may hold anything: the same bits with zeros and with large values."""
    st = inputs.cavity_state(N, 1e4, seed=N)
    with H.Cavity(_params(N, 1e4, 0.8, FP64)) as cav:
        for name, which in FIELDS:
            cav.set(which, st[name])
        for stage in (H.HOSC_STAGE_VISCOSITY, H.HOSC_STAGE_SOURCES, H.HOSC_STAGE_RHS):
            cav.run_stage(stage)
        w = [cav.get(H.HOSC_A_MOM + q) for q in range(7)] + \
            [cav.get(H.HOSC_A_ENE + q) for q in range(7)]
        rhs = [cav.get(H.HOSC_RHS_U + s) for s in range(4)]
    wall = np.ones((N, N, N), bool)
    wall[1:-1, 1:-1, 1:-1] = False
    out = []
    for fill in (0.0, 1e30):
        b = [np.where(wall, fill, r) for r in rhs]
        dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in w + b]
        x = [torch.zeros((N, N, N), dtype=torch.float64, device="cuda") for _ in range(4)]
        torch.cuda.synchronize()
        st_, iters = H.hosc_bicgstab_noalloc(N, [t.data_ptr() for t in dev[:14]],
                                             [t.data_ptr() for t in dev[14:]],
                                             [t.data_ptr() for t in x], 1e-10, 2000)
        torch.cuda.synchronize()
        assert st_ == H.HOSC_OK
        out.append((iters, [t.cpu().numpy() for t in x]))
    assert list(out[0][0]) == list(out[1][0])
    for a, b in zip(out[0][1], out[1][1]):
        assert np.array_equal(a, b)
