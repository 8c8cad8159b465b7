"""Diagnostics of small and odd boxes (fewer nodes than the reduction grid has threads, grids
that end within a block) and of fields with non-finite nodes, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1507_02518_gb300 import lb, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(3, 3, 3), (5, 7, 9), (16, 16, 1 + 16), (33, 17, 15), (64, 48, 54)])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("order", [2, 8])
@pytest.mark.parametrize("nan", [False, True])
def test_diagnostics_match_oracle(shape, storage, order, nan):
    nx, ny, nz = shape
    rng = np.random.default_rng(2)
    u = 0.05 * rng.uniform(-1, 1, (3, nz, ny, nx)) + np.array([0.02, -0.01, 0.03]).reshape(3, 1, 1, 1)
    f = oracle.init_equilibrium(1 + 0.05 * rng.uniform(-1, 1, (nz, ny, nx)), u)
    f *= 1 + 1e-2 * workloads.population_noise(nx, ny, nz, seed=4)
    lat = lb.Lattice(nx, ny, nz, nu=1e-3, storage=storage, scheme="aa")
    lat.set_populations(f)
    lat.step(1)
    lat.set_diag_order(order)
    f1 = lat.get_populations()
    if nan:
        f1[7, nz // 2, ny // 2, nx // 2] = np.nan
        lb.lb_set_time(lat.ctx, 0)
        lat.set_populations(f1)
    d = lat.diagnostics(raise_nonfinite=False)
    rho, uu = oracle.macroscopic(f1)[:2]
    assert d["nonfinite_count"] == int(nan) == int(np.isnan(rho).sum())
    # FP64 sums of P terms; FP32 arithmetic per node and thread: 2^-24 of the summed magnitudes
    eps = 1e-13 if storage == "f64" else 4e-6
    ok = ~np.isnan(rho)
    assert abs(d["mass"] - rho[ok].sum()) <= eps * ok.sum()
    for a in range(3):
        assert abs(d["momentum"][a] - (rho * uu[a])[ok].sum()) <= eps * np.abs(rho * uu[a])[ok].sum()
    k = 0.5 * sum(((uu[a][ok] - uu[a][ok].mean()) ** 2).mean() for a in range(3))
    assert abs(d["kinetic_energy"] - k) <= eps * k
    if nan:
        assert np.isfinite(d["enstrophy"]) and np.isnan(d["gamma_mean"])
        return
    ref = oracle.diagnostics(rho, uu, 1e-3, order)
    for key in ("enstrophy", "dissipation", "dudx2"):
        assert abs(d[key] - ref[key]) <= 4 * eps * ref[key]
    assert abs(d["gamma_mean"] - lat.gamma().astype(np.float64).mean()) <= eps * 2
