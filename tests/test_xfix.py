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
extern "C" void edges(int n, const double* u, int linear, double* out) {
  const gbcfd::XVal eps = gbcfd::xdec_pos<62>(1e-6);
  for (int i = 0; i < n; ++i) {
    long long m[5];
    short e[5];
    for (int c = 0; c < 5; ++c) gbcfd::xline_value(u[5 * i + c], m + c, e + c);
    const gbcfd::XEdge g = gbcfd::xedges<1>(m, e, linear != 0, eps);
    out[2 * i] = gbcfd::xenc(g.up, g.e);
    out[2 * i + 1] = gbcfd::xenc(g.um, g.e);
  }
}
// the frame flux from doubles, twice or (half) once
static void frame(const double* l, const double* r, const gbcfd::XConsts& K, int half, double* F) {
  gbcfd::XFlux f;
  gbcfd::xroe(gbcfd::xpair(l[0], r[0]), gbcfd::xpair(l[1], r[1]), gbcfd::xpair(l[2], r[2]), gbcfd::xpair(l[3], r[3]),
              gbcfd::xpair(l[4], r[4]), K, f);
  for (int q = 0; q < 5; ++q) F[q] = gbcfd::xflux(f, q, half);
}
extern "C" void roe(int n, const double* L, const double* R, double gamma, double eps, int half, double* F) {
  const gbcfd::XConsts K = gbcfd::xconsts(gamma, eps);
  for (int i = 0; i < n; ++i) frame(L + 5 * i, R + 5 * i, K, half, F + 5 * i);
}
extern "C" void roe_area(int n, const double* L, const double* R, const double* S, double gamma, double eps, double* F) {
  const gbcfd::XConsts K = gbcfd::xconsts(gamma, eps);
  for (int i = 0; i < n; ++i) {
    const double *l = L + 5 * i, *r = R + 5 * i, *s = S + 3 * i;
    gbcfd::XFlux f;
    gbcfd::xroe_area(gbcfd::xpair(l[0], r[0]), gbcfd::xpair(l[1], r[1]), gbcfd::xpair(l[2], r[2]), gbcfd::xpair(l[3], r[3]),
                     gbcfd::xpair(l[4], r[4]), s[0], s[1], s[2], K, f);
    for (int q = 0; q < 5; ++q) F[5 * i + q] = gbcfd::xflux(f, q, 0);
  }
}
extern "C" void prims(int n, const double* q, double gamma, double* W, int* ok) {
  const gbcfd::XConsts K = gbcfd::xconsts(gamma, 0.1);
  for (int i = 0; i < n; ++i) {
    gbcfd::XPrim w;
    ok[i] = gbcfd::xprim(q + 5 * i, K, w);
    const gbcfd::XVal c = gbcfd::xsound(w, K.gam), v[6] = {w.r, w.u[0], w.u[1], w.u[2], w.p, c};
    for (int k = 0; k < 6; ++k) W[6 * i + k] = gbcfd::xenc(v[k].m, v[k].e);
  }
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
ULP = 2.0 ** -53


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


@pytest.mark.parametrize("kind", ["smooth", "uniform", "jumps", "aligned"])
def test_roe_flux_through_an_area_vector(lib, kind):
    """the curvilinear form, x, y, z momentum, against the frame form in long double"""
    n, rng = 8000, np.random.Generator(np.random.PCG64(9))
    L, R = states("smooth" if kind == "aligned" else kind, n, rng)
    S = rng.uniform(-1, 1, (n, 3)) * 10.0 ** rng.uniform(-6, 0, (n, 1))
    if kind == "aligned":  # axis-aligned and nearly aligned faces
        S = np.eye(3)[rng.integers(0, 3, n)] * 1e-3 + rng.choice([0.0, 1e-9, 1e-20], (n, 3))
    S = np.ascontiguousarray(S)
    ld = np.longdouble
    s = S.astype(ld)
    area = np.sqrt((s * s).sum(1))
    nrm = s / area[:, None]
    a = np.abs(S).argmin(1)
    e = np.eye(3)[a].astype(ld)
    t1 = e - (nrm * e).sum(1)[:, None] * nrm
    t1 /= np.sqrt((t1 * t1).sum(1))[:, None]
    t2 = np.cross(nrm, t1)
    frame = lambda w: np.concatenate([w[:, :1].astype(ld)] + [(w[:, 1:4].astype(ld) * v).sum(1)[:, None] for v in (nrm, t1, t2)]
                                     + [w[:, 4:].astype(ld)], 1)
    f, sc = reference(frame(L), frame(R), 1.4, 0.1)
    want = np.concatenate([f[:, :1], f[:, 1:2] * nrm + f[:, 2:3] * t1 + f[:, 3:4] * t2, f[:, 4:]], 1) * (area / 2)[:, None]
    # the normal velocity is a sum of products of the size of |u|: what the flux carries of it is
    # rounded relative to |u|, however small u . n is (rho, rho |u| + rho c, rho H per unit of it)
    speed = np.maximum(np.abs(L[:, 1:4]).sum(1), np.abs(R[:, 1:4]).sum(1))
    rho, p = np.maximum(L[:, 0], R[:, 0]), np.maximum(L[:, 4], R[:, 4])
    h = np.maximum(3.5 * L[:, 4] / L[:, 0], 3.5 * R[:, 4] / R[:, 0]) + 0.5 * speed ** 2
    mom = (sc[:, 1:4].sum(1) + rho * speed * (speed + np.sqrt(h)))[:, None]
    scale = np.concatenate([sc[:, :1] + (rho * speed)[:, None], mom, mom, mom, sc[:, 4:] + (rho * h * speed)[:, None]],
                           1) * (area / 2)[:, None]
    F = np.empty((n, 5))
    lib.roe_area(n, _p(L), _p(R), _p(S), ctypes.c_double(1.4), ctypes.c_double(0.1), _p(F))
    # the FP64 form's bound, with the rotations' roundings (about 20 more)
    assert np.all(np.abs(F - want) <= 80 * ULP * scale)


def test_primitives(lib):
    n, rng = 50000, np.random.Generator(np.random.PCG64(11))
    r, p = 10.0 ** rng.uniform(-2, 2, n), 10.0 ** rng.uniform(-2, 2, n)
    v = rng.uniform(-2, 2, (3, n)) * 10.0 ** rng.uniform(-9, 0, (3, n))
    v[2, ::3] = 0.0
    q = np.ascontiguousarray(np.stack([r, r * v[0], r * v[1], r * v[2], p / 0.4 + 0.5 * r * (v * v).sum(0)], 1))
    W, ok = np.empty((n, 6)), np.zeros(n, dtype=np.int32)
    lib.prims(n, _p(q), ctypes.c_double(1.4), _p(W), ok.ctypes.data_as(ctypes.c_void_p))
    assert ok.all()
    Q = q.astype(np.longdouble)
    u = Q[:, 1:4] / Q[:, :1]
    P = np.longdouble(1.4 - 1.0) * (Q[:, 4] - 0.5 * (Q[:, 1:4] * u).sum(1))
    assert np.array_equal(W[:, 0], q[:, 0])
    assert np.all(np.abs(W[:, 1:4] - u) <= (ULP + 2.0 ** -56) * np.abs(u))  # zero stays zero
    # the kinetic part's products and the difference: 2^-57 of the energy each, then one rounding
    assert np.all(np.abs(W[:, 4] - P) <= ULP * np.abs(P) + 8 * 2.0 ** -57 * Q[:, 4])
    c = np.sqrt(np.longdouble(1.4) * W[:, 4].astype(np.longdouble) / Q[:, 0])
    assert np.all(np.abs(W[:, 5] - c) <= 3 * ULP * c)


@pytest.mark.parametrize("q", [(-1, 0, 0, 0, 1), (0, 0, 0, 0, 1), (1, 0, 0, 0, -1), (1, 10, 0, 0, 1), (np.nan, 0, 0, 0, 1),
                               (np.inf, 0, 0, 0, 1), (1, np.inf, 0, 0, 1), (1, 0, np.nan, 0, 1), (1, 0, 0, -np.inf, 1),
                               (1, 0, 0, 0, np.inf), (1, 0, 0, 0, np.nan)])
def test_non_physical_primitives_are_refused(lib, q):
    a, W, ok = np.array(q, dtype=np.float64), np.empty(6), np.ones(1, dtype=np.int32)
    lib.prims(1, _p(a), ctypes.c_double(1.4), _p(W), ok.ctypes.data_as(ctypes.c_void_p))
    assert not ok[0]


@pytest.mark.parametrize("kind", ["smooth", "rough", "step", "flat", "tiny", "offset", "zero", "mixed sizes"])
@pytest.mark.parametrize("linear", [0, 1])
def test_weighted_interpolation(lib, kind, linear):
    """both edge values of the WCNS-E-5 interpolation against the definition in long double.  The FP64
    form rounds the candidates and the sum relative to the stencil's largest value; its weights'
    roundings (about 20) act on the candidates' distances."""
    n, rng = 20000, np.random.Generator(np.random.PCG64(21))
    x = np.arange(5) * 0.1
    u = {"smooth": lambda: np.sin(x + rng.uniform(0, 6.3, (n, 1))) + 2.0,
         "rough": lambda: rng.uniform(-1, 1, (n, 5)),
         "step": lambda: np.where(np.arange(5) < rng.integers(0, 6, (n, 1)), 1.0, 0.125) + 1e-4 * rng.uniform(-1, 1, (n, 5)),
         "flat": lambda: np.repeat(rng.uniform(-1, 1, (n, 1)), 5, 1),
         "tiny": lambda: 1e-200 * rng.uniform(-1, 1, (n, 5)),
         "offset": lambda: 1e5 + rng.uniform(-1, 1, (n, 5)),
         "zero": lambda: np.zeros((n, 5)),
         "mixed sizes": lambda: rng.uniform(-1, 1, (n, 5)) * 10.0 ** rng.uniform(-8, 2, (n, 5))}[kind]()
    u = np.ascontiguousarray(u)
    out = np.empty((n, 2))
    lib.edges(n, _p(u), linear, _p(out))
    w = u.astype(np.longdouble).T

    def edge(a):
        g = [(a[0] - 4 * a[1] + 3 * a[2]) / 2, (a[3] - a[1]) / 2, (-3 * a[2] + 4 * a[3] - a[4]) / 2]
        s = [a[0] - 2 * a[1] + a[2], a[1] - 2 * a[2] + a[3], a[2] - 2 * a[3] + a[4]]
        al = [c if linear else c / (np.longdouble(1e-6) + gk * gk + sk * sk) ** 2
              for c, gk, sk in zip((np.longdouble(1), 10, 5), g, s)]
        return a[2] + sum(k * (gk / 2 + sk / 8) for k, gk, sk in zip(al, g, s)) / sum(al)

    want = np.stack([edge(w), edge(w[::-1])], 1)
    big, span = np.abs(u).max(1, keepdims=True), (u.max(1) - u.min(1))[:, None]
    assert np.all(np.abs(out - want) <= 4 * ULP * big + 20 * ULP * span)
    if kind in ("flat", "zero"):
        assert np.array_equal(out, u[:, 2:3].repeat(2, 1))


def test_staged_values_that_are_not_finite_stay_so(lib):
    u = np.ones((3, 5))
    u[0, 0], u[1, 2], u[2, 4] = np.nan, np.inf, -np.inf
    out = np.empty((3, 2))
    lib.edges(3, _p(u), 0, _p(out))
    assert not np.isfinite(out).any()
