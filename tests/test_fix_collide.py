"""The fixed-point FP64 collision (csrc/kbc_fix.cuh), compiled for the host, against the collision
written out in extended precision, and against the same in FP64: it must not be less exact."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1507_02518_gb300", "csrc")
LD = np.longdouble
VEL = [(i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1) for i in range(27)]
V = np.array(VEL)

WRAP = r'''
#define __host__
#define __device__
#define __forceinline__ inline
#include "kbc_fix.cuh"
using namespace kbc;
extern "C" void fix_collide(int n, const double* d, double* o, double* g, int* flags, double beta,
                            int wt, int wq, int mode) {
  const fix::Relax rx = {fix::quarter_beta(beta), fix::two_beta_1(beta), 1.0 / beta,
                         wt, wq, mode};
  for (int k = 0; k < n; ++k) {
    fix::fx v[27];
    uint32_t top = 0;
    for (int i = 0; i < 27; ++i) v[i] = fix::from_f64(d[k * 27 + i], &top);
    int gd = 0;
    bool bad = false;
    g[k] = fix::collide(v, rx, &gd, &bad);
    flags[k] = (top >= fix::kTopF64 || bad ? 2 : 0) | gd;
    for (int i = 0; i < 27; ++i) {
      const int nz = fix::nonzero(i);
      o[k * 27 + i] = nz == 0 ? fix::to_f64<0>(v[i]) : nz == 1 ? fix::to_f64<1>(v[i])
                    : nz == 2 ? fix::to_f64<2>(v[i]) : fix::to_f64<3>(v[i]);
    }
  }
}
extern "C" void fix_equilibrium(int n, const double* in, double* o, float* of, float* odd) {
  uint32_t top = 0;
  for (int k = 0; k < n; ++k) {
    fix::fx v[4], p[27];
    for (int a = 0; a < 4; ++a) v[a] = fix::from_f64(in[4 * k + a], &top);
    fix::equilibrium(v[0], v[1], v[2], v[3], p);
    for (int i = 0; i < 27; ++i) {
      const int nz = fix::nonzero(i), j = k * 27 + i;
      o[j] = nz == 0 ? fix::to_f64<0>(p[i]) : nz == 1 ? fix::to_f64<1>(p[i])
           : nz == 2 ? fix::to_f64<2>(p[i]) : fix::to_f64<3>(p[i]);
      of[j] = nz == 0 ? fix::to_f32<0>(p[i]) : nz == 1 ? fix::to_f32<1>(p[i])
            : nz == 2 ? fix::to_f32<2>(p[i]) : fix::to_f32<3>(p[i]);
      odd[j] = nz == 0 ? fix::to_f32_odd<0>(p[i]) : nz == 1 ? fix::to_f32_odd<1>(p[i])
             : nz == 2 ? fix::to_f32_odd<2>(p[i]) : fix::to_f32_odd<3>(p[i]);
    }
  }
}
extern "C" void fix_round(int n, const double* d, double* o, const float* f, double* of) {
  uint32_t top = 0;
  for (int k = 0; k < n; ++k) {
    o[k] = fix::to_f64<0>(fix::from_f64(d[k], &top));
    of[k] = fix::to_f64<0>(fix::from_f32(f[k], &top));
  }
}
extern "C" void fix_to_f32(int n, const long long* v, float* f, float* odd) {
  for (int k = 0; k < n; ++k) {
    f[k] = fix::to_f32<2>(v[k]);
    odd[k] = fix::to_f32_odd<2>(v[k]);
  }
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fix")
    src = d / "wrap.cpp"
    src.write_text(WRAP)
    so = str(d / "fix.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared",
                    "-I" + CSRC, str(src), "-o", so], check=True)
    return ctypes.CDLL(so)


def weights(T):
    return np.array([np.prod([T(2) / 3 if c == 0 else T(1) / 6 for c in v]) for v in VEL])


def product_equilibrium(rho, u, T):
    ax = []
    for a in range(3):
        R = np.sqrt(1 + 3 * u[a] ** 2)
        ax.append([(2 * R - 1 - 3 * u[a]) / 6, 2 * (2 - R) / 3, (2 * R - 1 + 3 * u[a]) / 6])
    return np.stack([rho * ax[0][v[0] + 1] * ax[1][v[1] + 1] * ax[2][v[2] + 1] for v in VEL], 1)


def reference(delta, beta, wt, wq, mode, T):
    """The collision of the shifts in the type T: (shifts after it, gamma)."""
    d, beta = delta.astype(T), T(beta)
    rho = 1 + d.sum(1)
    u = [(d * V[:, a].astype(T)).sum(1) / rho for a in range(3)]
    eq = product_equilibrium(rho, u, T)
    dev = d + weights(T) - eq

    def m(p, q, r):
        return (dev * (V[:, 0] ** p * V[:, 1] ** q * V[:, 2] ** r).astype(T)).sum(1)
    ks = [(2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1), (0, 1, 1)]
    if wq:
        ks += [(1, 2, 0), (1, 0, 2), (2, 1, 0), (0, 1, 2), (2, 0, 1), (0, 2, 1), (1, 1, 1)]
    M = {k: m(*k) for k in ks}
    if not wt:
        tr = (M[2, 0, 0] + M[0, 2, 0] + M[0, 0, 2]) / 3
        for k in ks[:3]:
            M[k] = M[k] - tr

    def c(v, p):
        return ((1, 0, -1) if v == 0 else (0, v / 2, 0.5))[p]
    ds = np.stack([sum(T(c(v[0], k[0]) * c(v[1], k[1]) * c(v[2], k[2])) * x
                       for k, x in M.items()) for v in VEL], 1)
    dh = dev - ds
    if mode == 0:
        g = 1 / beta - (2 - 1 / beta) * (ds * dh / eq).sum(1) / (dh * dh / eq).sum(1)
    else:
        g = np.full(len(d), T(2) if mode == 1 else 1 / beta)
    return d - beta * (2 * ds + g[:, None] * dh), g


def states(n, shear, higher, umax, seed):
    """Shifts of nodes at velocity up to umax, a non-equilibrium stress and higher moments of
    the given sizes (relative to the weights)."""
    rng = np.random.default_rng(seed)
    rho = (1 + rng.uniform(-0.02, 0.02, n)).astype(LD)
    u = rng.uniform(-umax, umax, (3, n)).astype(LD)
    S = rng.uniform(-1, 1, (n, 3, 3))
    S = (S + S.transpose(0, 2, 1)) / 2
    Q = np.array([np.outer(v, v) - np.eye(3) / 3 for v in VEL])
    neq = shear * np.einsum("iab,nab->ni", Q, S) + higher * rng.uniform(-1, 1, (n, 27))
    return (product_equilibrium(rho, u, LD) + weights(LD) * (neq - 1)).astype(np.float64)


def collide(lib, d, beta, wt, wq, mode):
    n = len(d)
    o, g, fl = np.empty((n, 27)), np.empty(n), np.empty(n, dtype=np.int32)
    p = [a.ctypes.data_as(ctypes.c_void_p) for a in (d, o, g, fl)]
    lib.fix_collide(n, *p, ctypes.c_double(beta), wt, wq, mode)
    return o, g, fl


def rms(a):
    return float(np.sqrt((a.astype(np.float64) ** 2).mean()))


@pytest.mark.parametrize("shear,higher", [(2e-2, 2e-2), (1e-3, 1e-3), (1e-3, 1e-6),
                                          (1e-5, 1e-6), (1e-8, 1e-8), (0.0, 1e-11)])
@pytest.mark.parametrize("wt,wq,mode", [(0, 0, 0), (1, 0, 0), (0, 1, 0), (1, 1, 0), (1, 1, 1),
                                        (0, 1, 2)])
def test_error_is_not_above_that_of_fp64(lib, shear, higher, wt, wq, mode):
    d = states(2000, shear, higher, 0.12, 11)
    beta = 1.0 / (6 * 2e-4 + 1)
    ref, _ = reference(d, beta, wt, wq, mode, LD)
    f64, _ = reference(d, beta, wt, wq, mode, np.float64)
    o, _, fl = collide(lib, d, beta, wt, wq, mode)
    assert not (fl & 2).any()
    assert rms(o - ref) <= rms(f64 - ref)
    # conserved moments: exact but for the rounding of the 27 results (half an ulp of 1/4 each)
    for w in [np.ones(27)] + [V[:, a] for a in range(3)]:
        assert np.abs(((o - d).astype(LD) * w).sum(1)).max() <= 27 * 2.0 ** -55


def test_rest_is_guarded_and_kept(lib):
    o, g, fl = collide(lib, np.zeros((1, 27)), 0.9, 1, 1, 0)
    assert fl[0] == 1 and g[0] == 2.0 and not o.any()


@pytest.mark.parametrize("wt,wq", [(0, 0), (1, 1)])
def test_equilibrium_states_stay(lib, wt, wq):
    """Deviations of a unit or none: gamma is a ratio of nothing, the node must not move."""
    rng = np.random.default_rng(9)
    u = rng.uniform(-0.1, 0.1, (3, 3000)) * rng.integers(0, 2, (3, 3000))
    d = (product_equilibrium(np.ones(3000, dtype=LD), u.astype(LD), LD) - weights(LD))
    d = d.astype(np.float64)
    o, _, fl = collide(lib, d, 0.99, wt, wq, 0)
    ok = (fl & 2) == 0
    assert ok.mean() > 0.9 and (fl & 1).any()
    # |f' - f| is bounded by the deviations (a few units each, 27 of them) whatever gamma is
    assert np.abs(o - d)[ok].max() <= 1000 * 2.0 ** -60


@pytest.mark.parametrize("what", ["nan", "inf", "shift", "rho", "u", "gamma"])
def test_out_of_range_is_reported(lib, what):
    d = states(3, 1e-3, 1e-3, 0.05, 5)
    if what == "nan":
        d[1, 7] = np.nan
    elif what == "inf":
        d[1, 26] = -np.inf
    elif what == "shift":
        d[1, 13] = 0.25
    elif what == "rho":
        d[1] = weights(LD) * -0.55
    elif what == "u":
        d[1] = states(1, 0.0, 0.0, 0.0, 1)[0]
        d[1, 14] += 0.24
        d[1, 17] += 0.1
    else:  # <ds|dh> / <dh|dh> about 10^5
        pxy = np.array([v[0] * v[1] / 4.0 if v[2] == 0 else 0.0 for v in VEL])
        d[1] = states(1, 0.0, 1e-8, 0.0, 3)[0] + 1e-2 * pxy
        x = reference(d[1:2], 0.999, 1, 1, 0, LD)[1]
        assert abs(float(x[0])) > 600
    _, _, fl = collide(lib, d, 0.999, 1, 1, 0)
    assert fl[1] & 2 and not (fl[[0, 2]] & 2).any()


def test_conversions(lib):
    rng = np.random.default_rng(2)
    d = np.concatenate([rng.uniform(-0.25, 0.25, 3000), rng.uniform(-1, 1, 3000) * 2.0 ** -rng.integers(2, 70, 3000),
                        [0.0, -0.0, 2.0 ** -60, 2.0 ** -61, -5e-324, np.nextafter(0.25, 0)]])
    f = d.astype(np.float32)
    f = np.where(np.abs(f) >= 0.25, np.float32(0.1), f)
    o, of = np.empty_like(d), np.empty_like(d)
    p = [a.ctypes.data_as(ctypes.c_void_p) for a in (d, o, f, of)]
    lib.fix_round(len(d), *p)
    unit = 2.0 ** -60
    assert np.array_equal(o, np.trunc(d.astype(LD) / LD(unit)).astype(np.float64) * unit)
    assert np.array_equal(of, np.trunc(f.astype(LD) / LD(unit)).astype(np.float64) * unit)


def test_equilibrium_and_its_roundings(lib):
    """f_eq - W in fixed point, and its roundings to FP32 (to nearest; to odd, after which a
    rounding to half is the rounding of the exact value)."""
    rng = np.random.default_rng(4)
    n = 4000
    x = np.concatenate([rng.uniform(-0.2, 0.2, (n, 4)), np.zeros((1, 4)),
                        rng.uniform(-1e-5, 1e-5, (n, 4))])
    o = np.empty((len(x), 27))
    of, odd = np.empty((len(x), 27), np.float32), np.empty((len(x), 27), np.float32)
    lib.fix_equilibrium(len(x), *[a.ctypes.data_as(ctypes.c_void_p) for a in (x, o, of, odd)])
    ref = product_equilibrium(1 + x[:, 0].astype(LD), x[:, 1:].T.astype(LD), LD) - weights(LD)
    assert np.abs(o - ref).max() <= 16 * 2.0 ** -57  # |u| up to 0.2: e is good to 2^-54
    assert np.abs(o - ref)[n + 1:].max() <= 16 * 2.0 ** -60
    assert not o[n].any() and not of[n].any() and not odd[n].any()
    # o is exact here for |v| < 2^53 units and rounded above; FP32 of either is the same
    assert np.array_equal(of, o.astype(np.float32))
    assert np.array_equal(odd.astype(np.float16), o.astype(np.float16))


@pytest.mark.parametrize("k", range(14, 60))
def test_rounding_of_one_binade(lib, k):
    """FP32 and FP16 of values below 2^k units: ties of FP32 and their neighbours, and the small
    values next to the bound of the short way (2^38). Exact: one rounding, to nearest even."""
    rng = np.random.default_rng(k)
    m = rng.integers(2 ** 24, 2 ** 25, 500)                      # 25 bits: odd ones are ties
    v = np.concatenate([(m << max(k - 25, 0)) >> max(25 - k, 0), 2 ** k - np.arange(1, 40),
                        rng.integers(0, 2 ** k, 500)])
    v = np.concatenate([v - 1, v, v + 1])
    v = np.concatenate([v, -v])
    v = np.ascontiguousarray(v[np.abs(v) < 2 ** 60], dtype=np.int64)
    f, odd = np.empty(len(v), np.float32), np.empty(len(v), np.float32)
    lib.fix_to_f32(len(v), *[a.ctypes.data_as(ctypes.c_void_p) for a in (v, f, odd)])
    x = v.astype(LD) * LD(2.0) ** -62
    assert np.array_equal(f, x.astype(np.float32))
    # FP16, where it is not a tie: the nearest of the exact value
    h = odd.astype(np.float16).astype(LD)
    step = np.maximum(LD(2.0) ** -24, LD(2.0) ** (np.floor(np.log2(np.maximum(np.abs(x), LD(1e-30)))) - 10))
    assert (np.abs(h - x) <= step / 2).all()
