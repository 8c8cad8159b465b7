"""The FP64 step and the FP64 re-collision on the GPU at the edges of the fixed-point format:
nodes inside and outside its range in one warp, and scattered flagged nodes."""
import numpy as np
import pytest

import oracle
from paper_1507_02518_gb300 import lb, workloads

pytestmark = pytest.mark.gpu
SHAPES = [(3, 3, 3), (5, 7, 9), (33, 4, 3), (64, 5, 3)]


def base_state(nx, ny, nz, seed, amp=1e-3):
    rng = np.random.default_rng(seed)
    u = rng.uniform(-0.05, 0.05, (3, nz, ny, nx))
    f = oracle.init_equilibrium(1 + rng.uniform(-0.02, 0.02, (nz, ny, nx)), u)
    return f * (1 + amp * workloads.population_noise(nx, ny, nz, seed=seed + 1))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("variant", ["d", "d+t+q"])
def test_nodes_outside_the_range(shape, scheme, variant):
    nx, ny, nz = shape
    f = base_state(nx, ny, nz, 3)
    n = np.random.default_rng(4).permutation(nx * ny * nz)
    g = f.reshape(27, -1)
    g[:, n[0::5]] *= 2.5     # rho about 2.5, some shifts above 1/4
    g[:, n[1::5]] *= 0.4     # rho about 0.4
    g[14, n[2::5]] += 0.2    # |u| about 0.2
    lat = lb.Lattice(nx, ny, nz, nu=1e-3, storage="f64", scheme=scheme, variant=variant)
    lat.set_populations(f)
    lat.step(2)
    var = {"d": oracle.S_D, "d+t+q": oracle.S_DTQ}[variant]
    ref, gam, _ = oracle.run(f, 2, oracle.beta(1e-3), var, want_gamma=True)
    # f up to 1 here: FP64 rounding of ~50 operations on either side, amplified at most by the
    # ratio of the shear to the higher part in gamma (about 100 for this noise)
    assert np.abs(lat.get_populations() - ref).max() <= 2e-13
    assert np.abs(lat.gamma() - gam).max() <= 1e-5


@pytest.mark.parametrize("scheme", ["pull", "aa"])
def test_a_nan_node_stays_local(scheme):
    f = base_state(9, 4, 5, 7)
    f[5, 2, 1, 3] = np.nan
    lat = lb.Lattice(9, 4, 5, nu=1e-3, storage="f64", scheme=scheme)
    lat.set_populations(f)
    lat.step(1)
    got = lat.get_populations()
    ref, _, _ = oracle.run(f, 1, oracle.beta(1e-3), oracle.S_DTQ)
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.isnan(ref).any()
    assert np.nanmax(np.abs(got - ref)) <= 1e-14


@pytest.mark.parametrize("shape", [(5, 7, 9), (40, 6, 3), (64, 8, 4)])
@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("every", [1, 2, 7, 33])
def test_scattered_fp64_recollision(shape, scheme, every):
    """FP32 storage, every n-th node (and a run of 40) within round-off of equilibrium: those
    are collided again in FP64, the others are not."""
    nx, ny, nz = shape
    f = base_state(nx, ny, nz, 5)
    P = nx * ny * nz
    flat = np.zeros(P, dtype=bool)
    flat[::every] = True
    flat[P // 2:P // 2 + 40] = True
    rho, u = oracle.macroscopic(f)[:2]
    eq = oracle.init_equilibrium(rho, u)
    near = eq * (1 + 1e-7 * workloads.population_noise(nx, ny, nz, seed=6))
    f = np.where(flat.reshape(1, nz, ny, nx), near, f)
    lat = lb.Lattice(nx, ny, nz, nu=1e-3, storage="f32", scheme=scheme)
    lat.set_populations(f)
    fin = lat.get_populations()
    lat.step(1)
    got, gam = lat.get_populations(), lat.gamma().ravel()
    _, want, _ = oracle.run(fin, 1, oracle.beta(1e-3), oracle.S_DTQ, want_gamma=True)
    ref = oracle.run(fin, 1, oracle.beta(1e-3), oracle.S_DTQ)[0]
    assert np.abs(got - ref).max() <= 2e-7            # the bound of an FP32 step
    # gamma of the nodes near equilibrium: the FP64 value, the ratio of products of deviations of
    # ~1e-7 W known to ~1e-17 (the oracle's rounding)
    assert np.abs(gam - want.ravel())[flat].max() <= 1e-6 * np.abs(want).max()
