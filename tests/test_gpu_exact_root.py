"""The FP64 exact stabilizer: nodes near equilibrium (series), far from it (Newton with
logarithms) and both in one warp, against the oracle's root."""
import numpy as np
import pytest

import oracle
from paper_1507_02518_gb300 import lb, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("noise", [1e-7, 1e-4, 1e-2, 0.05, 0.2, "mixed"])
@pytest.mark.parametrize("variant", ["d", "d+t+q", "cd+ct+cq"])
@pytest.mark.parametrize("nu", [1e-4, 0.05])
def test_root_matches_oracle(noise, variant, nu):
    nx, ny, nz = 33, 5, 4
    rng = np.random.default_rng(1)
    u = rng.uniform(-0.06, 0.06, (3, nz, ny, nx))
    f = oracle.init_equilibrium(1 + rng.uniform(-0.02, 0.02, (nz, ny, nx)), u)
    n = workloads.population_noise(nx, ny, nz, seed=5)
    amp = noise if noise != "mixed" else 10.0 ** rng.uniform(-6, -0.7, (nz, ny, nx))
    f = f * (1 + amp * n)
    lat = lb.Lattice(nx, ny, nz, nu=nu, storage="f64", scheme="pull", variant=variant, gamma="exact")
    lat.set_populations(f)
    gap = lat.stabilizer_gap()
    lat.step(1)
    beta, v = oracle.beta(nu), lb.VARIANT[variant]
    _, g_ex, _ = oracle.collide_field(f, beta, v, oracle.GAMMA_EXACT, want_gamma=True)
    _, g_est, _ = oracle.collide_field(f, beta, v, oracle.GAMMA_ESTIMATE, want_gamma=True)
    ref = oracle.run(f, 1, beta, v, oracle.GAMMA_EXACT)[0]
    assert np.abs(lat.get_populations() - ref).max() <= 1e-14
    # f' is known to ~1e-16, so gamma to that over |dh| (noise W / 10 at least)
    small = float(np.min(amp)) if noise == "mixed" else noise
    tol = 1e-7 + 1e-14 / small
    assert np.abs(lat.gamma() - g_ex).max() <= tol * (1 + np.abs(g_ex).max())
    assert gap["unconverged"] == 0 and gap["skipped"] == 0 and gap["nodes"] == nx * ny * nz
    assert gap["mean_abs"] == pytest.approx(np.abs(g_ex - g_est).mean(), rel=1e-6, abs=1e-14 / small)
