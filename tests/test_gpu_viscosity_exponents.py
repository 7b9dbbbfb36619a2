"""The FP64 viscosity eta = x^((n-1)/2), x = I2 + eps, for exponents within rounding of +-1/m (a root by
Newton's method) and others (pow), against 50-digit decimal arithmetic on the very exponent and x.

A uniform shear du/dz on a grid with spacing 1/8 and plane differences that are powers of two makes I2
exact at every node, walls included. Bound: the root is within 0.8 units in the last place, n > 1 takes its
reciprocal and L one product or quotient more: 2 units of 2^-52 for eta, 3 for L.
"""

from decimal import Decimal, getcontext

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2411_06563_gb300.hosc")

N = 9   # h = 1/8


@pytest.mark.parametrize("n", [1 + 2 / 3, 1 - 2 / 3, 1 + 2 / 7, 1 - 2 / 7, 1 + 2 / 13, 1 - 2 / 13, 0.9,
                               1.1, 0.75, 1.25, 0.7123])
@pytest.mark.parametrize("power", [-20, -3, 10, 30, 46])
def test_viscosity_of_a_uniform_shear(n, power):
    getcontext().prec = 50
    p = H.hosc_default_params(N, 1e4, 1.0, n)
    shear = 2.0 ** power
    x = shear * shear + p.I2_eps
    exact = Decimal(x) ** ((Decimal(n) - 1) / 2)
    with H.Cavity(p) as cav:
        for which in (H.HOSC_V, H.HOSC_W, H.HOSC_P):
            cav.set(which, np.zeros((N, N, N)))
        cav.set(H.HOSC_U, np.broadcast_to((np.arange(N) * shear / 8)[:, None, None], (N, N, N)))
        cav.run_stage(H.HOSC_STAGE_VISCOSITY)
        eta, L = cav.get(H.HOSC_ETA), cav.get(H.HOSC_LCOEF)
    assert np.all(eta == eta[4, 4, 4]) and np.all(L == L[4, 4, 4])
    ulp = Decimal(2) ** -52
    assert abs(Decimal(float(eta[4, 4, 4])) / exact - 1) <= 2 * ulp
    assert abs(Decimal(float(L[4, 4, 4])) * exact - 1) <= 3 * ulp
