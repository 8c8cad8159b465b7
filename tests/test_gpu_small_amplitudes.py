"""FP64 storage keeps the flow's relative precision at any amplitude."""
import numpy as np
import pytest

from paper_1507_02518_gb300 import lb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("amp", [1e-3, 1e-6, 1e-8, 1e-12, 1e-25])
def test_uniform_flow_keeps_its_momentum(scheme, amp):
    """1000 steps, the last amplitude in FP64 instructions. A step rounds 27 populations, each by
    2^-53 of its size at most; the momentum is several times the largest shift."""
    u0 = amp * np.array([1.0, -0.7, 0.3])
    u = np.broadcast_to(u0.reshape(3, 1, 1, 1), (3, 4, 3, 34)).copy()
    lat = lb.Lattice(34, 3, 4, nu=1e-3, storage="f64", scheme=scheme)
    lat.init_field(None, u)
    lat.step(1000)
    _, v = lat.moments()
    assert np.abs(v / u0.reshape(3, 1, 1, 1) - 1.0).max() <= 1000 * 27 * 2.0 ** -53


@pytest.mark.parametrize("scheme", ["pull", "aa"])
def test_small_shear_wave_is_the_larger_one_scaled(scheme):
    """At u <= 1e-7 the terms of second order are below 1e-7 of the flow: two amplitudes give the
    same decaying wave but for those (0.1 of the flow at most, over 40 steps)."""
    n, out = 32, []
    x = 2 * np.pi * np.arange(n) / n
    for amp in (1e-8, 1e-7):
        u = np.zeros((3, 4, 4, n))
        u[1] = amp * np.sin(x)
        lat = lb.Lattice(n, 4, 4, nu=1e-2, storage="f64", scheme=scheme)
        lat.init_field(None, u)
        lat.step(40)
        out.append(lat.moments()[1][1] / amp)
    assert np.abs(out[0]).max() > 0.9
    assert np.abs(out[0] - out[1]).max() <= 40 * 1e-7
