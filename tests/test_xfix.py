"""The 64-bit block-floating Roe flux of the FP64 path (csrc/xfix.cuh), compiled for the host and
held against the same formulas in long double over the states it can meet: smooth, low Mach,
supersonic, SI units, tiny scales, strong jumps, uniform, wide entropy bands, gamma 3, subnormal
and zero velocities.  The tolerance is the FP64 form's own error bound: its ~60 roundings of 2^-53 on
terms no larger than the sum of the magnitudes of the flux's parts."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_09995_gb300", "csrc")

HARNESS = r"""
#include <algorithm>
#define __host__
#define __device__
#define __forceinline__ inline
#include "xfix.cuh"
extern "C" void roe(int n, const double* L, const double* R, double gamma, double eps, int half, double* F) {
  const gbcfd::XConsts K = gbcfd::xconsts(gamma, eps);
  for (int i = 0; i < n; ++i)
    if (half) gbcfd::xroe<false>(L + 5 * i, R + 5 * i, K, F + 5 * i);
    else gbcfd::xroe<true>(L + 5 * i, R + 5 * i, K, F + 5 * i);
}
extern "C" void roots(int n, const double* v, double* s, double* r) {
  for (int i = 0; i < n; ++i) {
    const gbcfd::XVal a = gbcfd::xrsqrt(gbcfd::xdec_pos<62>(v[i])), b = gbcfd::xrcp(gbcfd::xdec_pos<62>(v[i]));
    s[i] = gbcfd::xenc(a.m, a.e);
    r[i] = gbcfd::xenc(b.m, b.e);
  }
}
"""
_D = ctypes.POINTER(ctypes.c_double)


def _p(a):
    return a.ctypes.data_as(_D)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("xfix")
    src, so = d / "xfix.cpp", d / "xfix.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def reference(L, R, gamma, eps):
    """twice the Roe flux with Harten's fix (Eq. 1's fluxes) in long double, and the sum of the
    magnitudes of its parts"""
    ld = np.longdouble
    l, r = L.astype(ld).T, R.astype(ld).T
    gam = ld(gamma)
    gm1, ggm1 = ld(float(gamma - 1.0)), ld(float(gamma / (gamma - 1.0)))
    h = lambda w: ggm1 * w[4] / w[0] + (w[1] ** 2 + w[2] ** 2 + w[3] ** 2) / 2
    hl, hr, sl, sr = h(l), h(r), np.sqrt(l[0]), np.sqrt(r[0])
    al, ar, rt = sl / (sl + sr), sr / (sl + sr), sl * sr
    u, v, w, ht = (al * a + ar * b for a, b in ((l[1], r[1]), (l[2], r[2]), (l[3], r[3]), (hl, hr)))
    q2 = u * u + v * v + w * w
    c2 = gm1 * (ht - q2 / 2)
    c = np.sqrt(c2)
    d = r - l
    a1, a5, a2 = (d[4] - rt * c * d[1]) / (2 * c2), (d[4] + rt * c * d[1]) / (2 * c2), d[0] - d[4] / c2
    delta = ld(eps) * (abs(u) + c)
    fix = lambda x: np.where(abs(x) < delta, (x * x + delta * delta) / (2 * np.where(delta > 0, delta, 1)), abs(x))
    w1, w2, w5, l2 = fix(u - c) * a1, fix(u) * a2, fix(u + c) * a5, fix(u)
    ml, mr = l[0] * l[1], r[0] * r[1]
    parts = [[ml, mr, -w1, -w2, -w5],
             [ml * l[1], l[4], mr * r[1], r[4], -w1 * (u - c), -w2 * u, -w5 * (u + c)],
             [ml * l[2], mr * r[2], -(w1 + w2 + w5) * v, -l2 * rt * d[2]],
             [ml * l[3], mr * r[3], -(w1 + w2 + w5) * w, -l2 * rt * d[3]],
             [ml * hl, mr * hr, -w1 * (ht - c * u), -w5 * (ht + c * u), -w2 * q2 / 2, -l2 * rt * v * d[2],
              -l2 * rt * w * d[3]]]
    # the strengths' own terms, which FP64 rounds before they cancel
    rho = np.maximum(l[0], r[0])
    noise = [0 * c, 0 * c, 0 * c, 0 * c, 0 * c]
    for k, f in enumerate([1, abs(u) + c, abs(v), abs(w), ht]):
        noise[k] = noise[k] + (abs(d[4]) / c2 + rho * abs(d[1]) / c + abs(d[0])) * (abs(u) + c) * f
    return (np.stack([sum(p) for p in parts]).T,
            np.stack([sum(abs(x) for x in p) + e for p, e in zip(parts, noise)]).T)


def states(kind, n, rng):
    u = lambda a=-1.0, b=1.0, k=n: rng.uniform(a, b, k)
    L = np.stack([1 + 0.1 * u(), 0.5 + 0.1 * u(), 0.3 * u(), 0.2 * u(), (1 + 0.1 * u()) / 1.4], 1)
    R = L * (1 + 1e-2 * rng.uniform(-1, 1, (n, 5)))
    if kind == "low mach":
        L[:, 1:4] *= 1e-4; R[:, 1:4] *= 1e-4
    elif kind == "supersonic":
        L[:, 1] += 3; R[:, 1] += 3
    elif kind == "si":
        for a in (L, R):
            a[:, 0] *= 1.2; a[:, 1:4] *= 340.0; a[:, 4] *= 1.4e5
    elif kind == "tiny":
        for a in (L, R):
            a[:, 0] *= 1e-120; a[:, 4] *= 1e-120
    elif kind == "jumps":
        for a in (L, R):
            a[:, 0] = 10 ** u(); a[:, 4] = 10 ** u(); a[:, 1:4] = rng.uniform(-2, 2, (n, 3))
    elif kind == "uniform":
        R = L.copy()
    elif kind == "cross":  # velocities of very different size, zeros and subnormals among them
        for a in (L, R):
            a[:, 2] *= 10 ** u(-12, 0)
            a[:, 3] = rng.choice([0.0, -0.0, 5e-324, 1e-310, 1e-9], n)
    return np.ascontiguousarray(L), np.ascontiguousarray(R)


@pytest.mark.parametrize("kind,gamma,eps", [
    ("smooth", 1.4, 0.1), ("smooth", 1.4, 0.0), ("smooth", 1.4, 2.0), ("smooth", 3.0, 0.1), ("smooth", 5.0 / 3.0, 1.0),
    ("low mach", 1.4, 0.1), ("supersonic", 1.4, 0.1), ("si", 1.4, 0.1), ("tiny", 1.4, 0.1), ("jumps", 1.4, 0.1),
    ("jumps", 1.1, 0.5), ("uniform", 1.4, 0.1), ("cross", 1.4, 0.1)])
def test_roe_flux(lib, kind, gamma, eps):
    n = 20000
    L, R = states(kind, n, np.random.Generator(np.random.PCG64(7)))
    want, scale = reference(L, R, gamma, eps)
    F = np.empty((n, 5))
    lib.roe(n, _p(L), _p(R), ctypes.c_double(gamma), ctypes.c_double(eps), 0, _p(F))
    err = np.abs(F - want)
    assert np.all(err <= 60 * 2.0 ** -53 * scale + 1e-300)
    # the root mean square error is no larger than one rounding of the result and one of its parts
    rms = np.sqrt(np.mean((err / scale.max(0)).astype(np.float64) ** 2, 0))
    assert np.all(rms <= 2.0 ** -53), rms
    G = np.empty((n, 5))
    lib.roe(n, _p(L), _p(R), ctypes.c_double(gamma), ctypes.c_double(eps), 1, _p(G))
    assert np.array_equal(G * 2.0, F)  # half the flux, bit for bit


def test_uniform_state_has_no_dissipation(lib):
    L, R = states("uniform", 4000, np.random.Generator(np.random.PCG64(3)))
    F = np.empty_like(L)
    lib.roe(len(L), _p(L), _p(R), ctypes.c_double(1.4), ctypes.c_double(0.1), 0, _p(F))
    m = L[:, 0].astype(np.longdouble) * L[:, 1]
    assert np.all(np.abs(F[:, 0] - 2 * m) <= 2.0 ** -52 * np.abs(2 * m))


@pytest.mark.parametrize("where", ["rho_l", "rho_r", "p_both"])
def test_non_physical_states_give_nan(lib, where):
    L, R = states("smooth", 1, np.random.Generator(np.random.PCG64(1)))
    if where == "rho_l":
        L[:, 0] = -0.5
    elif where == "rho_r":
        R[:, 0] = -1e-3
    else:
        L[:, 4] = R[:, 4] = -1.0
    F = np.empty_like(L)
    lib.roe(1, _p(L), _p(R), ctypes.c_double(1.4), ctypes.c_double(0.1), 0, _p(F))
    assert np.all(np.isnan(F))


def test_reciprocal_roots(lib):
    rng = np.random.Generator(np.random.PCG64(5))
    v = np.concatenate([2.0 ** rng.uniform(-300, 300, 200000), [1.0, 2.0, 4.0, 0.5, np.nextafter(1.0, 2), np.nextafter(2.0, 1),
                                                               np.nextafter(4.0, 0)]])
    s, r = np.empty_like(v), np.empty_like(v)
    lib.roots(len(v), _p(v), _p(s), _p(r))
    x = v.astype(np.longdouble)
    # one rounding to double and the iteration's 2^-57
    assert np.all(np.abs(s * np.sqrt(x) - 1) <= 2.0 ** -53 + 2.0 ** -57 + 2.0 ** -62)
    assert np.all(np.abs(r * x - 1) <= 2.0 ** -53 + 2.0 ** -57 + 2.0 ** -62)
