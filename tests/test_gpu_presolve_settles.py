"""The FP64 pre-solve of a uniform flow comes to rest: the measured change of the density is
exactly 0, at any amplitude of the velocity."""
import numpy as np
import pytest

from paper_1507_02518_gb300 import lb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("nu_pre", [1.0 / 6.0, 0.1])
@pytest.mark.parametrize("amp", [0.03, 1e-4, 1e-6, 1e-8])
def test_change_is_exactly_zero(scheme, nu_pre, amp):
    u0 = amp * np.array([1.0, -2.0 / 3.0, 1.0 / 3.0])
    u = np.broadcast_to(u0.reshape(3, 1, 1, 1), (3, 5, 6, 34)).copy()
    lat = lb.Lattice(34, 6, 5, nu=1e-3, storage="f64", scheme=scheme)
    _, res = lat.presolve(u, nu_pre=nu_pre, max_iters=200, tol=-1.0)
    assert res == 0.0
    rho, v = lat.moments()
    assert np.abs(rho - 1.0).max() <= 27 * 2.0 ** -53 * max(amp, 1.0)
    assert np.abs(v - u).max() <= 1e-12 * amp
