"""The FP64 pre-solve step (fixed point, and FP64 where a node is outside the format's range)
against the oracle, over relaxations, schemes, odd boxes and velocities in and out of range."""
import numpy as np
import pytest

import oracle
from paper_1507_02518_gb300 import lb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(3, 3, 3), (5, 7, 9), (33, 4, 3), (64, 6, 5)])
@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("nu_pre", [1.0 / 6.0, 0.02, 1.5])
@pytest.mark.parametrize("amp", [0.0, 1e-6, 0.05, 0.3])
def test_presolve_matches_oracle(shape, scheme, nu_pre, amp):
    nx, ny, nz = shape
    rng = np.random.default_rng(3)
    u = amp * rng.uniform(-1, 1, (3, nz, ny, nx))
    lat = lb.Lattice(nx, ny, nz, nu=1e-3, storage="f64", scheme=scheme)
    iters, _ = lat.presolve(u, nu_pre=nu_pre, max_iters=6, tol=-1.0)
    assert iters == 6
    ref = oracle.presolve(u, 1.0 / (6.0 * nu_pre + 1.0), 6, -1.0)[0]
    # six iterations of ~30 rounded FP64 operations on values up to f (0.5 at most here)
    assert np.abs(lat.get_populations() - ref).max() <= 6 * 30 * 2.0 ** -54


@pytest.mark.parametrize("nu_pre", [1.0 / 6.0, 0.1])
def test_fixed_point_has_no_change(nu_pre):
    """A uniform flow is a fixed point of the iteration: the measured change is exactly 0."""
    u = np.broadcast_to(np.array([0.03, -0.02, 0.01]).reshape(3, 1, 1, 1), (3, 5, 6, 34)).copy()
    lat = lb.Lattice(34, 6, 5, nu=1e-3, storage="f64", scheme="aa")
    _, res = lat.presolve(u, nu_pre=nu_pre, max_iters=64, tol=-1.0)
    assert res <= 2.0 ** -52
