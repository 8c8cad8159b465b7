"""State transfers (set, get, moments, init) on the GPU against numpy, with values of every kind:
ordinary, tiny, zero, subnormal, infinite, NaN, far from a lattice state."""
import numpy as np
import pytest
import torch

import oracle
from paper_1507_02518_gb300 import lb

pytestmark = pytest.mark.gpu
W = np.array([np.prod([2 / 3 if c == 0 else 1 / 6 for c in (i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1)])
              for i in range(27)]).reshape(27, 1)
V = np.array([(i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1) for i in range(27)])
SHAPES = [(3, 3, 3), (5, 7, 9), (33, 4, 3), (64, 5, 5)]
KINDS = ["plain", "tiny", "rest", "mixed"]


def field(kind, P, storage, seed):
    rng = np.random.default_rng(seed)
    rel = rng.uniform(-0.2, 0.2, (27, P))
    if kind == "tiny":
        rel *= 2.0 ** -rng.integers(10, 40, (27, P))
    elif kind == "rest":
        rel *= rng.integers(0, 2, (1, P))
    f = W * (1 + rel)
    if kind == "mixed":
        n = rng.permutation(P)
        f[:, n[0::6]] *= 40.0
        f[:, n[1::6]] *= 1e-3
        f[3, n[2::6]] = np.nan
        f[20, n[3::6]] = np.inf
        f[8, n[4::6]] = 1e5 if storage == "f16" else 1e200
    return f


def stored(f, storage):
    """The stored value of f as a shift, exactly (extended precision)."""
    if storage == "f64":
        return (f - W).astype(np.longdouble)
    with np.errstate(all="ignore"):
        if storage == "f32":
            return (f - W).astype(np.float32).astype(np.longdouble)
        return W.astype(np.longdouble) * ((f - W) / W).astype(np.float16)


@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("scheme,t", [("pull", 0), ("pull", 1), ("aa", 0), ("aa", 1)])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", SHAPES)
def test_set_get_moments(shape, kind, scheme, t, storage):
    nx, ny, nz = shape
    f = field(kind, nx * ny * nz, storage, 3)
    lat = lb.Lattice(nx, ny, nz, nu=1e-3, storage=storage, scheme=scheme)
    lb.lb_set_time(lat.ctx, t)
    lat.set_populations(f.reshape(27, nz, ny, nx))
    d = stored(f, storage)
    got = lat.get_populations().reshape(27, -1)
    ulp = np.spacing(np.where(np.isfinite(d), np.abs(W + d), 1.0).astype(np.float64))
    with np.errstate(invalid="ignore"):
        # FP16: f = W + W h rounded once or twice, and ties of (f - W)/W may fall either way
        off = np.abs(got - (W + d))
        half = np.maximum(np.abs(d) * 2.0 ** -10, 2.0 ** -24 * W) if storage == "f16" else 0.0
        tie = off > ulp
        assert not (np.isfinite(d) & (off > ulp + half)).any()
        assert (tie & np.isfinite(d)).mean() <= (1e-3 if storage == "f16" else 0.0)
    assert np.array_equal(np.isnan(got), np.isnan(W + d))
    assert np.array_equal(np.isposinf(got), np.isposinf(W + d))
    # a second round trip changes nothing
    lat.set_populations(got.reshape(27, nz, ny, nx))
    assert np.array_equal(lat.get_populations().reshape(27, -1), got, equal_nan=True)

    # moments of the stored shifts, summed in extended precision
    rho, u = lat.moments()
    e = (got - W if storage != "f64" else d).astype(np.longdouble)
    if storage == "f16":
        e = np.where(np.isfinite(got), W.astype(np.longdouble) * ((got - W) / W).astype(np.float16), got)
    elif storage == "f32":
        e = (got - W).astype(np.float32).astype(np.longdouble)
    with np.errstate(all="ignore"):
        s = 1 + e.sum(0)
        m = [(e * V[:, a:a + 1]).sum(0) / s for a in range(3)]
        big = np.abs(e).max(0)
        fin = np.isfinite(big.astype(np.float64))
        # 27 terms rounded at the size of the largest, or of rho; then two roundings of u
        tol = 30 * 2.0 ** -53 * (big + 0) + 2.0 ** -52 * np.abs(s)
        assert (np.abs(rho.ravel() - s)[fin] <= tol[fin]).all()
        for a in range(3):
            ta = 40 * 2.0 ** -53 * big / np.abs(s) + np.abs(m[a]) * (2.0 ** -50 + tol / np.abs(s))
            assert (np.abs(u[a].ravel() - m[a])[fin] <= ta[fin]).all()
    assert not np.isfinite(u[:, ~fin.reshape(nz, ny, nx)]).all(0).any()


@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("amp", [0.0, 1e-9, 1e-5, 0.05, 0.2, 0.5])
@pytest.mark.parametrize("with_rho", [False, True])
@pytest.mark.parametrize("shape", [(3, 3, 3), (33, 4, 3)])
def test_init(shape, with_rho, amp, scheme, storage):
    nx, ny, nz = shape
    rng = np.random.default_rng(1)
    u = amp * rng.uniform(-1, 1, (3, nz, ny, nx))
    rho = 1 + min(4 * amp, 0.6) * rng.uniform(-1, 1, (nz, ny, nx)) if with_rho else None
    want = oracle.init_equilibrium(np.ones((nz, ny, nx)) if rho is None else rho, u)
    ref = want.reshape(27, -1)
    for device in (False, True):
        lat = lb.Lattice(nx, ny, nz, nu=1e-3, storage=storage, scheme=scheme)
        if device:
            lat.init_field(None if rho is None else torch.from_numpy(rho).cuda(),
                           torch.from_numpy(u).cuda())
        else:
            lat.init_field(rho, u)
        got = lat.get_populations().reshape(27, -1)
        # the oracle's f is good to a few 2^-53; then the rounding of the stored shift
        d = np.abs(ref - W)
        tol = 6 * 2.0 ** -53 + {"f64": 0.0, "f32": 2.0 ** -24, "f16": 2.0 ** -11}[storage] * d
        if storage == "f16":
            tol = tol + W * 2.0 ** -25
        assert (np.abs(got - ref) <= tol * 1.01).all()
