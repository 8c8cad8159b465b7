"""The fixed-point collision and pre-solve (csrc/kbc_fix.cuh), compiled for the host, at every
amplitude of the flow: relative to the node's shifts they must be no less exact than the same in
FP64 instructions, and over many steps mass and momentum must drift no more."""
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
static double value(fix::fx v, int i, uint32_t s) {
  const int nz = fix::nonzero(i);
  return nz == 0 ? fix::to_f64<0>(v, s) : nz == 1 ? fix::to_f64<1>(v, s)
       : nz == 2 ? fix::to_f64<2>(v, s) : fix::to_f64<3>(v, s);
}
// `steps` collisions of each node as FP64 storage takes them; flag 4: the change's conserved
// moments are not exactly 0
extern "C" void collide(int n, int steps, double* d, double* g, int* flags, double beta, int wt,
                        int wq, int mode) {
  const fix::Relax rx = {fix::quarter_beta(beta), fix::two_beta_1(beta), 1.0 / beta,
                         wt, wq, mode};
  for (int k = 0; k < n; ++k) {
    flags[k] = 0;
    for (int t = 0; t < steps; ++t) {
      double* f = d + k * 27;
      fix::fx v[27];
      uint32_t top = 0, s;
      for (int i = 0; i < 27; ++i) top = fix::top_of(f[i]) > top ? fix::top_of(f[i]) : top;
      if (top >= fix::kTopF64 || !fix::scale_of<double>(top, &s)) { flags[k] |= 2; break; }
      for (int i = 0; i < 27; ++i) v[i] = fix::scaled(f[i], s);
      int gd = 0;
      bool bad = false;
      g[k] = fix::collide<true>(v, rx, &gd, &bad, s);
      flags[k] |= (bad ? 2 : 0) | gd;
      if (bad) break;
      fix::fx m[4] = {0, 0, 0, 0};
      for (int i = 0; i < 27; ++i) {
        const fix::fx w = v[i] * (8 >> fix::nonzero(i));
        m[0] += w, m[1] += (i % 3 - 1) * w, m[2] += (i / 3 % 3 - 1) * w, m[3] += (i / 9 - 1) * w;
        f[i] += value(v[i], i, s);
      }
      if (m[0] | m[1] | m[2] | m[3]) flags[k] |= 4;
    }
  }
}
// the same of FP32 shifts, as the re-collision takes them, the results unrounded
extern "C" void collide32(int n, const float* f, double* o, int* flags, double beta) {
  const fix::Relax rx = {fix::quarter_beta(beta), fix::two_beta_1(beta), 1.0 / beta, 1, 1, 0};
  for (int k = 0; k < n; ++k) {
    fix::fx v[27];
    uint32_t top = 0, s;
    for (int i = 0; i < 27; ++i) top = fix::top_of(f[k * 27 + i]) > top ? fix::top_of(f[k * 27 + i]) : top;
    flags[k] = top >= fix::kTopF32 || !fix::scale_of<float>(top, &s) ? 2 : 0;
    if (flags[k]) continue;
    for (int i = 0; i < 27; ++i) v[i] = fix::scaled(f[k * 27 + i], s);
    int gd = 0;
    bool bad = false;
    fix::collide<false>(v, rx, &gd, &bad, s);
    flags[k] = (bad ? 2 : 0) | gd;
    for (int i = 0; i < 27; ++i) o[k * 27 + i] = value(v[i], i, s);
  }
}
// `iters` pre-solve iterations of each node by itself (a uniform flow); rho - 1 of the states
// before the last and after it
extern "C" int presolve(int n, int iters, double* d, const double* u, double* before,
                        double* after, double beta2) {
  int bad = 0;
  for (int k = 0; k < n; ++k) {
    double(&f)[27] = *(double(*)[27])(d + 27 * k);
    for (int t = 0; t < iters; ++t) {
      fix::fx p[27];
      uint32_t s;
      const double* w = u + 3 * k;
      const bool ok = beta2 == 1.0 ? fix::presolve<true>(f, w[0], w[1], w[2], beta2, p, &s, before + k)
                                   : fix::presolve<false>(f, w[0], w[1], w[2], beta2, p, &s, before + k);
      if (!ok) { ++bad; break; }
      for (int i = 0; i < 27; ++i) f[i] = value(p[i], i, s);
    }
    fix::fx v[27], sum;
    uint32_t s, top;
    bool in;
    after[k] = fix::presolve_density(f, v, &sum, &s, &top, &in);
  }
  return bad;
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixamp")
    src = d / "wrap.cpp"
    src.write_text(WRAP)
    so = str(d / "fix.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared",
                    "-I" + CSRC, str(src), "-o", so], check=True)
    return ctypes.CDLL(so)


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def weights(T):
    return np.array([np.prod([T(2) / 3 if c == 0 else T(1) / 6 for c in v]) for v in VEL])


def equilibrium(drho, u, T):
    """f_eq(1 + drho, u) - W, relative to its own size (no W is added and taken away)."""
    g, w = [], weights(T)
    for a in range(3):
        t = 3 * u[a] ** 2
        e = t / (1 + np.sqrt(1 + t))
        g.append([2 * e - 3 * u[a], -e, 2 * e + 3 * u[a]])
    out = []
    for i, v in enumerate(VEL):
        x, y, z = (g[a][v[a] + 1] for a in range(3))
        p = drho + x + drho * x
        p = p + y + p * y
        out.append(w[i] * (p + z + p * z))
    return np.stack(out, 1)


def reference(d, beta, wt, wq, mode, T):
    """One collision of the shifts in the type T, relative to their own size."""
    d, beta = d.astype(T), T(beta)
    drho = d.sum(1)
    u = [(d * V[:, a].astype(T)).sum(1) / (1 + drho) for a in range(3)]
    eqs = equilibrium(drho, u, T)
    eq, dev = weights(T) + eqs, d - eqs

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
        den = (dh * dh / eq).sum(1)
        g = 1 / beta - (2 - 1 / beta) * (ds * dh / eq).sum(1) / np.where(den > 0, den, 1)
        g = np.where(den > 1e-300, g, T(2))
    else:
        g = np.full(len(d), T(2) if mode == 1 else 1 / beta)
    return d - beta * (2 * ds + g[:, None] * dh), g


def states(n, amp, noneq, seed, T=np.float64):
    """Shifts of nodes with velocity and density shift up to amp, a non-equilibrium stress and
    higher moments of the size noneq times amp (relative to the weights)."""
    rng = np.random.default_rng(seed)
    drho = (amp / 4 * rng.uniform(-1, 1, n)).astype(LD)
    u = amp * rng.uniform(-1, 1, (3, n)).astype(LD)
    S = rng.uniform(-1, 1, (n, 3, 3))
    S = (S + S.transpose(0, 2, 1)) / 2
    Q = np.array([np.outer(v, v) - np.eye(3) / 3 for v in VEL])
    neq = noneq * amp * (np.einsum("iab,nab->ni", Q, S) + 0.3 * rng.uniform(-1, 1, (n, 27)))
    return (equilibrium(drho, u, LD) + weights(LD) * neq).astype(T)


def collide(lib, d, beta, wt=1, wq=1, mode=0, steps=1):
    o, g, fl = d.copy(), np.empty(len(d)), np.empty(len(d), dtype=np.int32)
    lib.collide(len(d), steps, ptr(o), ptr(g), ptr(fl), ctypes.c_double(beta), wt, wq, mode)
    return o, g, fl


def rms(a):
    return float(np.sqrt((a ** 2).mean()))


AMPS = [0.12, 1e-2, 1e-3, 1e-4, 1e-6, 1e-8, 1e-12, 1e-17]


@pytest.mark.parametrize("amp", AMPS)
@pytest.mark.parametrize("noneq", [0.3, 1e-2, 1e-5])
@pytest.mark.parametrize("wt,wq,mode", [(0, 0, 0), (1, 1, 0), (1, 1, 1), (0, 1, 2)])
def test_error_is_not_above_that_of_fp64(lib, amp, noneq, wt, wq, mode):
    d = states(2000, amp, noneq, 21)
    beta = 1.0 / (6 * 2e-4 + 1)
    ref, _ = reference(d, beta, wt, wq, mode, LD)
    f64, _ = reference(d, beta, wt, wq, mode, np.float64)
    o, _, fl = collide(lib, d, beta, wt, wq, mode)
    assert not (fl & 6).any()
    size = np.abs(d).max(1, keepdims=True).astype(LD)
    assert rms((o - ref) / size) <= rms((f64 - ref) / size)


@pytest.mark.parametrize("amp", [a for a in AMPS if a > 1e-17])
def test_fp32_shifts_lose_nothing(lib, amp):
    """FP32 storage: what the collision loses lies below the rounding of the stored values."""
    d = states(2000, amp, 1e-6, 22, np.float32)
    beta = 1.0 / (6 * 2e-4 + 1)
    ref, _ = reference(d, beta, 1, 1, 0, LD)
    o, fl = np.empty(d.shape), np.empty(len(d), dtype=np.int32)
    lib.collide32(len(d), ptr(d), ptr(o), ptr(fl), ctypes.c_double(beta))
    assert not (fl & 2).any()
    # 2^-55 of the largest shift per truncated input; a moment of 27 of them, relaxed
    size = np.abs(d).max(1, keepdims=True).astype(LD)
    assert np.abs((o - ref) / size).max() <= 2 * 27 * 2.0 ** -54


STEPS, BETA = 10000, 0.99


@pytest.fixture(scope="module")
def uniform():
    """Uniform flows, 12 of each amplitude, and where 10^4 collisions in FP64 take them."""
    parts = []
    for amp in AMPS:
        rng = np.random.default_rng(5)
        u = amp * rng.uniform(-1, 1, (3, 12)).astype(LD)
        u[1, :4] = u[2, :8] = 0
        parts.append(equilibrium(amp / 8 * rng.uniform(-1, 1, 12).astype(LD), u, LD))
    d = np.concatenate(parts).astype(np.float64)
    f64 = d.copy()
    for _ in range(STEPS):
        f64 = reference(f64, BETA, 1, 1, 0, np.float64)[0]
    return d.reshape(len(AMPS), 12, 27), f64.reshape(len(AMPS), 12, 27)


@pytest.mark.parametrize("k", range(len(AMPS)))
def test_uniform_flow_keeps_mass_and_momentum(lib, uniform, k):
    """10^4 collisions of uniform flows: no drift beyond what FP64 instructions leave."""
    d, f64 = uniform[0][k], uniform[1][k]
    o, _, fl = collide(lib, d, BETA, steps=STEPS)
    assert not (fl & 6).any()
    size = np.abs(d).max(1)
    for w in [np.ones(27)] + [V[:, a] for a in range(3)]:
        ours = np.abs(((o - d).astype(LD) * w).sum(1)) / size
        theirs = np.abs(((f64 - d).astype(LD) * w).sum(1)) / size
        # a settled node is off by the roundings of its 27 populations once
        assert rms(ours) <= max(rms(theirs), 27 * 2.0 ** -54)


def test_edges_of_the_scale(lib):
    """Rest is kept and guarded; shifts below the smallest scale are left to the FP64 collision;
    zeros and subnormal numbers among larger shifts count as nothing."""
    x = states(4, 1e-3, 1e-2, 8)
    d = np.stack([np.zeros(27), x[0] * 2.0 ** -100, x[1] * 2.0 ** -50, x[2], x[3]])
    d[3, ::2] = 0.0
    d[4, ::3] = 5e-324
    beta = 0.9
    o, g, fl = collide(lib, d, beta)
    assert fl.tolist() == [1, 2, 0, 0, 0] and g[0] == 2.0 and not o[0].any()
    assert np.array_equal(o[1], d[1])
    ref, _ = reference(d[2:], beta, 1, 1, 0, LD)
    size = np.abs(d[2:]).max(1, keepdims=True).astype(LD)
    assert np.abs((o[2:] - ref) / size).max() <= 2 * 27 * 2.0 ** -54
    f = d.astype(np.float32)
    f[1] = x[0] * 2.0 ** -60  # below 2^-70
    f[4, ::3] = 1e-45
    o = np.zeros((5, 27))
    lib.collide32(5, ptr(f), ptr(o), ptr(fl), ctypes.c_double(beta))
    assert fl.tolist() == [1, 2, 0, 0, 0] and not o[0].any()
    ref, _ = reference(f[2:], beta, 1, 1, 0, LD)
    assert np.abs((o[2:] - ref) / size).max() <= 2 * 27 * 2.0 ** -54


@pytest.mark.parametrize("amp", [0.03, 1e-2, 1e-4, 1e-6, 1e-8, 1e-12])
@pytest.mark.parametrize("beta2", [1.0, 2 / 1.6, 2 / 1.12, 0.4])
def test_presolve_of_uniform_flow_settles(lib, amp, beta2):
    """The measured change of the density is exactly 0, and the density stays where it was."""
    rng = np.random.default_rng(6)
    n = 40
    u = np.concatenate([np.array([[3.0, -2.0, 1.0]]), rng.uniform(-3, 3, (n - 1, 3))]) * amp
    u[5:10, 1] = 0
    u = np.ascontiguousarray(u)
    drho = np.where(np.arange(n) % 2, amp * rng.uniform(-1, 1, n), 0).astype(LD)
    d = equilibrium(drho, u.T.astype(LD), LD).astype(np.float64)
    before, after = np.empty(n), np.empty(n)
    start = d.copy()
    bad = lib.presolve(n, 200, ptr(d), ptr(u), ptr(before), ptr(after), ctypes.c_double(beta2))
    assert bad == 0
    assert np.array_equal(before, after)
    size = np.abs(start).max(1)
    assert (np.abs((d - start).astype(LD).sum(1)) / size).max() <= 27 * 2.0 ** -53
    assert (np.abs(d - start).max(1) / size).max() <= 27 * 2.0 ** -53


@pytest.mark.parametrize("amp", [0.1, 1e-2, 1e-4, 1e-8])
def test_presolve_error_is_that_of_fp64(lib, amp):
    """One iteration at the default relaxation: f_eq as exact as in FP64 instructions."""
    rng = np.random.default_rng(7)
    n = 2000
    u = np.ascontiguousarray(amp * rng.uniform(-1, 1, (n, 3)))
    d = equilibrium((amp / 4 * rng.uniform(-1, 1, n)).astype(LD), u.T.astype(LD), LD)
    d = d.astype(np.float64)
    ref = equilibrium(d.astype(LD).sum(1), u.T.astype(LD), LD)
    f64 = equilibrium(d.sum(1), u.T, np.float64)
    before, after = np.empty(n), np.empty(n)
    size = np.abs(d).max(1, keepdims=True).astype(LD)
    assert lib.presolve(n, 1, ptr(d), ptr(u), ptr(before), ptr(after), ctypes.c_double(1.0)) == 0
    assert rms((d - ref) / size) <= rms((f64 - ref) / size)
