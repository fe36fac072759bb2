"""The block-floating arithmetic of the FP64 path (csrc/xfix.cuh) where values of very different size meet,
compiled for the host.  The bar is the FP64 form's own error: the same formulas evaluated in doubles here, against
long double, on the same inputs.  A component's root mean square error may be no larger than that
form's and one rounding of the result to a double."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_09995_gb300", "csrc")
ULP = 2.0 ** -53
F64, LD = np.float64, np.longdouble
_D = ctypes.POINTER(ctypes.c_double)
_d = ctypes.c_double

HARNESS = r"""
#include <algorithm>
#define __host__
#define __device__
#define __forceinline__ inline
#include "xfix.cuh"
using namespace gbcfd;
"""


def _p(a):
    return a.ctypes.data_as(_D)


def compiled(tmp_path_factory, name, code):
    d = tmp_path_factory.mktemp(name)
    src, so = d / "x.cpp", d / "x.so"
    src.write_text(HARNESS + code)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


def held(got, form, want):
    """per component: the root mean square error against that of the FP64 form"""
    got, form, want = (np.atleast_2d(x.T).T for x in (got, form, want))
    for q in range(want.shape[1]):
        rms = lambda x: float(np.sqrt(np.mean((x[:, q] / np.max(np.abs(want[:, q]) + LD(1e-300))) ** 2)))
        a, b = rms(got.astype(LD) - want), rms(form.astype(LD) - want)
        assert a <= b + ULP * rms(want), (q, a, b)


def roe(L, R, gamma, eps, t):
    """twice the Roe flux with Harten's fix in the face frame, columns (rho, un, ut1, ut2, p), evaluated in type t"""
    l, r = L.astype(t).T, R.astype(t).T
    gm1, ggm1 = t(float(gamma - 1.0)), t(float(gamma / (gamma - 1.0)))
    h = lambda w: ggm1 * w[4] / w[0] + t(0.5) * (w[1] ** 2 + w[2] ** 2 + w[3] ** 2)
    hl, hr, sl, sr = h(l), h(r), np.sqrt(l[0]), np.sqrt(r[0])
    al, ar, rt = sl / (sl + sr), sr / (sl + sr), sl * sr
    u, v, w, ht = (al * a + ar * b for a, b in ((l[1], r[1]), (l[2], r[2]), (l[3], r[3]), (hl, hr)))
    q2 = u * u + v * v + w * w
    c2 = gm1 * (ht - t(0.5) * q2)
    c = np.sqrt(c2)
    d = r - l
    a1, a5 = (d[4] - rt * c * d[1]) / (2 * c2), (d[4] + rt * c * d[1]) / (2 * c2)
    a2 = d[0] - d[4] / c2
    delta = t(eps) * (abs(u) + c)
    fix = lambda x: np.where(abs(x) < delta, (x * x + delta * delta) / (2 * np.where(delta > 0, delta, 1)), abs(x))
    w1, w2, w5, l2 = fix(u - c) * a1, fix(u) * a2, fix(u + c) * a5, fix(u)
    ml, mr, ws = l[0] * l[1], r[0] * r[1], w1 + w2 + w5
    return np.stack([ml + mr - ws,
                     (ml * l[1] + l[4]) + (mr * r[1] + r[4]) - (w1 * (u - c) + w2 * u + w5 * (u + c)),
                     ml * l[2] + mr * r[2] - (ws * v + l2 * rt * d[2]),
                     ml * l[3] + mr * r[3] - (ws * w + l2 * rt * d[3]),
                     ml * hl + mr * hr - (w1 * (ht - c * u) + w5 * (ht + c * u) + w2 * t(0.5) * q2
                                          + l2 * rt * (v * d[2] + w * d[3]))]).T


def smooth(n, g, size=(1.0, 1.0, 1.0), jump=1e-2):
    """both sides' (rho, u, v, w, p), velocities about `size`"""
    u = lambda a=-1.0, b=1.0: g.uniform(a, b, n)
    L = np.stack([1 + 0.1 * u(), size[0] * (0.5 + 0.1 * u()), size[1] * u(0.2, 0.4), size[2] * u(0.1, 0.3),
                  (1 + 0.1 * u()) / 1.4], 1)
    return np.ascontiguousarray(L), np.ascontiguousarray(L * (1 + jump * g.uniform(-1, 1, (n, 5))))


# ---- faces with an area vector --------------------------------------------------------------------

def roe_area(L, R, S, gamma, eps, t):
    """the flux through S, x, y, z momentum: rotated into the face frame and back, as the FP64 form"""
    s = S.astype(t)
    area = np.sqrt((s * s).sum(1))
    n = s / area[:, None]
    a = np.abs(n).argmin(1)
    e = np.eye(3)[a].astype(t)
    na = np.take_along_axis(n, a[:, None], 1)
    t1 = (e - na * n) / np.sqrt(1 - na * na)
    t2 = np.cross(n, t1)
    frame = lambda w: np.concatenate([w[:, :1].astype(t)] + [(w[:, 1:4].astype(t) * v).sum(1)[:, None] for v in (n, t1, t2)]
                                     + [w[:, 4:].astype(t)], 1)
    f = roe(frame(L), frame(R), gamma, eps, t)
    m = f[:, 1:2] * n + f[:, 2:3] * t1 + f[:, 3:4] * t2
    return np.concatenate([f[:, :1], m, f[:, 4:]], 1) * (t(0.5) * area)[:, None]


@pytest.fixture(scope="module")
def area_lib(tmp_path_factory):
    return compiled(tmp_path_factory, "area", r"""
extern "C" void flux(int n, const double* L, const double* R, const double* S, double gamma, double eps, double* F) {
  const XConsts K = xconsts(gamma, eps);
  for (int i = 0; i < n; ++i) {
    const double *l = L + 5 * i, *r = R + 5 * i, *s = S + 3 * i;
    XFlux f;
    xroe_area(xpair(l[0], r[0]), xpair(l[1], r[1]), xpair(l[2], r[2]), xpair(l[3], r[3]), xpair(l[4], r[4]), s[0], s[1],
              s[2], K, f);
    for (int q = 0; q < 5; ++q) F[5 * i + q] = xflux(f, q, 0);
  }
}
""")


@pytest.mark.parametrize("size", [1.0, 1e-3, 1e-6, 1e-9])
@pytest.mark.parametrize("faces", ["extruded", "aligned", "nearly aligned", "any"])
def test_area_flux_of_small_components(area_lib, faces, size):
    """one velocity component `size` times the others, on faces to which it is tangential (a grid extruded
    in z, axis-aligned ones), nearly so, and on any"""
    n, g = 6000, rng(3)
    L, R = smooth(n, g, (1.0, 1.0, size))
    S = g.uniform(0.2, 1.0, (n, 3)) * g.choice([-1.0, 1.0], (n, 3)) * 1e-3
    if faces == "extruded":
        S[:, 2] = 0.0
    elif faces != "any":
        off = ~np.eye(3, dtype=bool)[g.integers(0, 2, n)]
        S[off] *= 0.0 if faces == "aligned" else 1e-9
    F = np.empty((n, 5))
    area_lib.flux(n, _p(L), _p(R), _p(np.ascontiguousarray(S)), _d(1.4), _d(0.1), _p(F))
    held(F, roe_area(L, R, S, 1.4, 0.1, F64), roe_area(L, R, S, 1.4, 0.1, LD))


def test_area_flux_of_no_velocity_along_z_is_zero_there(area_lib):
    n, g = 500, rng(4)
    L, R = smooth(n, g, (1.0, 1.0, 0.0))
    S = np.stack([g.uniform(0.2, 1.0, n), g.uniform(0.2, 1.0, n), np.zeros(n)], 1)
    F = np.empty((n, 5))
    area_lib.flux(n, _p(L), _p(R), _p(S), _d(1.4), _d(0.1), _p(F))
    assert np.all(F[:, 3] == 0.0)


# ---- the flux in the face frame -------------------------------------------------------------------

@pytest.fixture(scope="module")
def roe_lib(tmp_path_factory):
    return compiled(tmp_path_factory, "roe", r"""
extern "C" void flux(int n, const double* L, const double* R, double gamma, double eps, double* F) {
  const XConsts K = xconsts(gamma, eps);
  for (int i = 0; i < n; ++i) {
    const double *l = L + 5 * i, *r = R + 5 * i;
    XFlux f;
    xroe(xpair(l[0], r[0]), xpair(l[1], r[1]), xpair(l[2], r[2]), xpair(l[3], r[3]), xpair(l[4], r[4]), K, f);
    for (int q = 0; q < 5; ++q) F[5 * i + q] = xflux(f, q, 0);
  }
}
""")


@pytest.mark.parametrize("eps", [0.1, 0.0])
@pytest.mark.parametrize("mach", [1.0, 1e-3, 1e-6])
@pytest.mark.parametrize("ratio", [1.01, 2.0, 10.0, 30.0])
def test_contact(roe_lib, ratio, mach, eps):
    """a jump of the density alone: the entropy wave's kinetic energy is far below the enthalpies, its speed
    below the sound speed"""
    n, g = 6000, rng(5)
    L, _ = smooth(n, g, (mach, mach, mach))
    R = L.copy()
    R[:, 0] *= np.where(g.random(n) < 0.5, ratio, 1 / ratio)
    F = np.empty((n, 5))
    roe_lib.flux(n, _p(L), _p(R), _d(1.4), _d(eps), _p(F))
    held(F, roe(L, R, 1.4, eps, F64), roe(L, R, 1.4, eps, LD))


# ---- states beside jumps --------------------------------------------------------------------------

@pytest.fixture(scope="module")
def muscl_lib(tmp_path_factory):
    return compiled(tmp_path_factory, "muscl", r"""
static XPair states(const double* w, int lim) {
  long long m[4];
  int e[4];
  for (int c = 0; c < 4; ++c) {
    const XVal v = xdec_zero(w[c]);
    m[c] = v.m >> 1;
    e[c] = v.e + 1;
  }
  return xmuscl(m, e, lim).s;
}
extern "C" void muscl(int n, const double* w, int lim, double* LR) {
  for (int i = 0; i < n; ++i) {
    const XPair s = states(w + 4 * i, lim);
    LR[2 * i] = xenc(s.l, s.e);
    LR[2 * i + 1] = xenc(s.r, s.e);
  }
}
extern "C" void flux(int n, const double* w, int lim, double* F, int* far) {  // w[i][variable][cell]
  const XConsts K = xconsts(1.4, 0.1);
  for (int i = 0; i < n; ++i) {
    const double* a = w + 20 * i;
    const XPos r = states(a, lim), p = states(a + 16, lim);
    far[i] = xfar(r, p);
    XFlux f;
    xroe(r, states(a + 4, lim), states(a + 8, lim), states(a + 12, lim), p, K, f);
    for (int q = 0; q < 5; ++q) F[5 * i + q] = xflux(f, q, 0);
  }
}
""")


def muscl(w, lim, t):
    w = w.astype(t)
    d01, d12, d23 = (w[..., i + 1] - w[..., i] for i in range(3))
    if lim:
        return w[..., 1] + t(0.25) * (d01 + d12), w[..., 2] - t(0.25) * (d12 + d23)
    mm = lambda a, b: np.where((a > 0) == (b > 0), np.where(abs(a) < abs(b), a, b), t(0)) * ((a != 0) & (b != 0))
    return w[..., 1] + t(0.5) * mm(d01, d12), w[..., 2] - t(0.5) * mm(d12, d23)


@pytest.mark.parametrize("lim", [0, 1])
@pytest.mark.parametrize("outer", [1.0, 3.0, 1e2, 1e6, 1e12, 0.0])
def test_states_beside_a_jump(muscl_lib, outer, lim):
    """cells 1 and 2 about 1, cell 0 or 3 (or both) `outer` times that, of either sign; with the central slope a state
    takes the jump in, and only then may its error be relative to that"""
    n, g = 8000, rng(7)
    w = 1.0 + 0.1 * g.uniform(-1, 1, (n, 4))
    for c in (0, 3):
        w[g.random(n) < 0.7, c] *= outer * g.choice([-1.0, 1.0])
    w = np.ascontiguousarray(w)
    out = np.empty((n, 2))
    muscl_lib.muscl(n, _p(w), lim, _p(out))
    L, R = muscl(w, lim, LD)
    want = np.stack([L, R], 1)
    size = np.abs(w[:, 1:3]).max(1, keepdims=True) if not lim else np.abs(w).max(1, keepdims=True)
    # the value and half a slope are rounded once each (FP64 form); the pair shares a class
    assert np.all(np.abs(out - want) <= 2 * ULP * (np.abs(want) + size))


@pytest.mark.parametrize("where", [0, 3])
@pytest.mark.parametrize("jump", [10.0, 1e3, 1e6])
def test_flux_beside_a_jump(muscl_lib, jump, where):
    """the face's own cells are smooth, the cell beyond is `jump` times them in every variable"""
    n, g = 6000, rng(8)
    L, _ = smooth(n, g)
    w = np.stack([L * (1 + 1e-2 * g.uniform(-1, 1, (n, 5))) for _ in range(4)], 2)
    w[:, :, where] *= jump
    w = np.ascontiguousarray(w)
    F, far = np.empty((n, 5)), np.zeros(n, dtype=np.int32)
    muscl_lib.flux(n, _p(w), 0, _p(F), far.ctypes.data_as(ctypes.c_void_p))
    assert not far.any()
    sides = lambda t: muscl(w, 0, t)
    held(F, roe(*sides(F64), 1.4, 0.1, F64), roe(*sides(LD), 1.4, 0.1, LD))


@pytest.mark.parametrize("v", [0, 4])
def test_faces_far_apart_are_told(muscl_lib, v):
    """a density or pressure jump of 2^7 and more at the face itself is left to FP64, one below 2^4 is not"""
    n, g = 2000, rng(9)
    for ratio, far_wanted in ((8.0, False), (128.0, True), (1e6, True)):
        L, _ = smooth(n, g)
        w = np.repeat(L[:, :, None], 4, 2)
        w[:, v, 2:] *= np.where(g.random(n) < 0.5, ratio, 1 / ratio)[:, None]
        F, far = np.empty((n, 5)), np.zeros(n, dtype=np.int32)
        muscl_lib.flux(n, _p(np.ascontiguousarray(w)), 0, _p(F), far.ctypes.data_as(ctypes.c_void_p))
        assert np.all(far == far_wanted), ratio


@pytest.mark.parametrize("ratio", [2.0, 16.0])
@pytest.mark.parametrize("vel", [1.0, 1e2])
def test_flux_across_a_jump(muscl_lib, vel, ratio):
    """jumps at the face that are not left to FP64: densities and pressures by `ratio`, velocities by `vel`, either way"""
    n, g = 6000, rng(10)
    L, _ = smooth(n, g)
    w = np.repeat(L[:, :, None], 4, 2) * (1 + 1e-2 * g.uniform(-1, 1, (n, 5, 4)))
    for v, k in ((0, ratio), (4, ratio)):
        w[:, v, 2:] *= np.where(g.random(n) < 0.5, k, 1 / k)[:, None]
    w[:, 1:4, 2:] *= np.where(g.random(n) < 0.5, vel, 1 / vel)[:, None, None]
    w = np.ascontiguousarray(w)
    F, far = np.empty((n, 5)), np.zeros(n, dtype=np.int32)
    muscl_lib.flux(n, _p(w), 0, _p(F), far.ctypes.data_as(ctypes.c_void_p))
    sides = lambda t: muscl(w, 0, t)
    held(F, roe(*sides(F64), 1.4, 0.1, F64), roe(*sides(LD), 1.4, 0.1, LD))


# ---- the viscous flux on uniform grids ------------------------------------------------------------

@pytest.fixture(scope="module")
def visc_lib(tmp_path_factory):
    return compiled(tmp_path_factory, "visc", r"""
// w[i][variable u_n, u_t1, u_t2, theta][cell]: cells L, R and the neighbours + and - of L, then of R, along t1, then t2
extern "C" void viscous(int n, const double* w, const double* h, double mu, double kappa, double* F) {
  XBlk X;
  for (int t = 0; t < 3; ++t) {
    const double ih = 1.0 / h[t], m2 = mu + mu;
    X.a[t] = xdec_pos<62>(m2 * ih);
    X.a43[t] = xdec_pos<62>((4.0 / 3.0) * m2 * ih);
    X.b[t] = xdec_pos<62>(m2 * (0.25 * ih));
    X.b23[t] = xdec_pos<62>((2.0 / 3.0) * m2 * (0.25 * ih));
    X.k[t] = xdec_pos<62>(4.0 * kappa * ih);
  }
  for (int i = 0; i < n; ++i) {
    long long m[4][10];
    int e[4][10];
    for (int v = 0; v < 4; ++v)
      for (int c = 0; c < 10; ++c) {
        const XVal a = xdec_zero(w[(i * 4 + v) * 10 + c]);
        m[v][c] = a.m >> 1;
        e[v][c] = a.e + 1;
      }
    XVal dn[4];
    long long us[3];
    int eu[3];
    for (int v = 0; v < 4; ++v) {
      const int E = xmax(e[v][0], e[v][1]);
      const long long l = xshr(m[v][0], E - e[v][0]), r = xshr(m[v][1], E - e[v][1]);
      dn[v] = xquick0(r - l, E);
      if (v < 3) {
        us[v] = l + r;
        eu[v] = E;
      }
    }
    auto tang = [&](int v, int at) {
      long long a[4];
      int b[4];
      for (int c = 0; c < 4; ++c) {
        a[c] = m[v][at + c];
        b[c] = e[v][at + c];
      }
      return xtang(a, b, 0);
    };
    XFlux f;
    for (int q = 0; q < 5; ++q) {
      f.m[q] = 0;
      f.e[q] = XZERO;
    }
    xviscous(0, 1, 2, X, dn, us, eu, tang(0, 2), tang(0, 6), tang(1, 2), tang(2, 6), f);
    for (int q = 0; q < 4; ++q) F[4 * i + q] = xflux(f, 1 + q, 0);
  }
}
""")


def viscous(w, h, mu, kappa, t):
    w = w.astype(t)
    ih = [t(1.0 / x) for x in h]
    tang = lambda v, at, d: ((w[:, v, at] - w[:, v, at + 1]) + (w[:, v, at + 2] - w[:, v, at + 3])) * (t(0.25) * ih[d])
    gn = [(w[:, v, 1] - w[:, v, 0]) * ih[0] for v in range(4)]
    div = gn[0] + tang(1, 2, 1) + tang(2, 6, 2)
    tau = [t(2 * mu) * (2 * gn[0] - t(2.0 / 3.0) * div), t(2 * mu) * (gn[1] + tang(0, 2, 1)), t(2 * mu) * (gn[2] + tang(0, 6, 2))]
    e = sum((w[:, v, 0] + w[:, v, 1]) * tau[v] for v in range(3)) + t(4 * kappa) * gn[3]
    return np.stack([-tau[0], -tau[1], -tau[2], t(-0.5) * e], 1)


@pytest.mark.parametrize("size", [1.0, 1e-3, 1e-6, 1e-9])
@pytest.mark.parametrize("small", [0, 1, 2])
@pytest.mark.parametrize("still", ["none", "u_n along t1", "u_t1", "all but the small one"])
def test_viscous_flux_of_small_components(visc_lib, still, small, size):
    """one velocity component `size` times the others, which vary everywhere, or not along a tangent, or not
    at all: no stress takes bits from another, nor a term from one that is zero"""
    n, g = 3000, rng(11)
    w = 1.0 + 0.05 * g.uniform(-1, 1, (n, 4, 10))
    if still == "u_n along t1":
        w[:, 0, 2:6] = w[:, 0, :1]
    elif still == "u_t1":
        w[:, 1] = w[:, 1, :1]
    elif still != "none":
        for v in {0, 1, 2} - {small}:
            w[:, v] = w[:, v, :1]
    w[:, small] *= size
    w = np.ascontiguousarray(w)
    h, F = np.array([1 / 64, 1 / 48, 1e-3]), np.empty((n, 4))
    visc_lib.viscous(n, _p(w), _p(h), _d(1e-4), _d(4.9e-4), _p(F))
    held(F, viscous(w, h, 1e-4, 4.9e-4, F64), viscous(w, h, 1e-4, 4.9e-4, LD))


# ---- WCNS-E-5 edges beside jumps ------------------------------------------------------------------

@pytest.fixture(scope="module")
def edge_lib(tmp_path_factory):
    return compiled(tmp_path_factory, "edges", r"""
extern "C" void edges(int n, const double* u, int linear, double* out) {
  const XVal eps = xdec_pos<62>(1e-6);
  for (int i = 0; i < n; ++i) {
    long long m[5];
    short e[5];
    for (int c = 0; c < 5; ++c) xline_value(u[5 * i + c], m + c, e + c);
    const XEdge g = xedge_values<1>(m, e, linear != 0, eps);
    out[2 * i] = xenc(g.up, g.e);
    out[2 * i + 1] = xenc(g.um, g.e);
  }
}
""")


def edges(u, linear, t):
    w = u.astype(t).T

    def edge(a):
        g = [t(0.5) * (a[0] - 4 * a[1] + 3 * a[2]), t(0.5) * (a[3] - a[1]), t(0.5) * (4 * a[3] - 3 * a[2] - a[4])]
        s = [a[0] - 2 * a[1] + a[2], a[1] - 2 * a[2] + a[3], a[2] - 2 * a[3] + a[4]]
        al = [t(c) if linear else t(c) / (t(1e-6) + (gk * gk + sk * sk)) ** 2 for c, gk, sk in zip((1, 10, 5), g, s)]
        return a[2] + sum(k * (t(0.5) * gk + t(0.125) * sk) for k, gk, sk in zip(al, g, s)) / sum(al)

    return np.stack([edge(w), edge(w[::-1])], 1)


@pytest.mark.parametrize("linear", [0, 1])
@pytest.mark.parametrize("low", [0.5, 0.1, 1e-2, 1e-4, 1e-8])
@pytest.mark.parametrize("side,at", [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (1, 4)])
def test_edges_beside_a_jump(edge_lib, side, at, low, linear):
    """cells on one side of the jump are 1, on the other `low`: the weights keep the jump out of the values on either
    side.  Errors relative to the cell's value and its distance from the edge's (what the FP64 form rounds)."""
    n, g = 3000, rng(13)
    hi = (np.arange(5) >= at) if side else (np.arange(5) < at)
    u = np.ascontiguousarray(np.where(hi, 1.0, low) * (1 + 0.05 * g.uniform(-1, 1, (n, 5))))
    out = np.empty((n, 2))
    edge_lib.edges(n, _p(u), linear, _p(out))
    want, form = edges(u, linear, LD), edges(u, linear, F64)
    size = np.maximum(np.abs(u[:, 2:3]), np.abs(want - u[:, 2:3]))
    rms = lambda x: float(np.sqrt(np.mean((x / size) ** 2)))
    assert rms(out - want) <= rms(form - want) + ULP


@pytest.mark.parametrize("u", [(0.0,) * 5, (1.0,) * 5, (1e-30,) * 5])
def test_edges_of_a_constant_are_that_constant(edge_lib, u):
    a, out = np.array(u), np.empty(2)
    for linear in (0, 1):
        edge_lib.edges(1, _p(a), linear, _p(out))
        assert np.all(out == u[2])


def test_edges_that_are_not_finite_stay_so(edge_lib):
    for c in range(5):
        for bad in (np.nan, np.inf, -np.inf):
            a, out = np.array([1e-9] * 5), np.empty(2)
            a[c] = bad
            edge_lib.edges(1, _p(a), 0, _p(out))
            assert not np.isfinite(out).any()


# ---- below the normal range -----------------------------------------------------------------------

@pytest.fixture(scope="module")
def tiny_lib(tmp_path_factory):
    return compiled(tmp_path_factory, "tiny", r"""
extern "C" void again(int n, const double* a, double* b, double* c, double* d) {  // through a value, a line's, and scaled
  for (int i = 0; i < n; ++i) {
    const XVal v = xdec_zero(a[i]);
    b[i] = xenc(v.m, v.e);
    long long m;
    short e;
    xline_value(a[i], &m, &e);
    c[i] = xenc(m, e - XW_BIAS);
    d[i] = xenc(v.m, v.e - 30);
  }
}
extern "C" void velocity(int n, const double* q, double* u) {
  const XConsts K = xconsts(1.4, 0.1);
  for (int i = 0; i < n; ++i) {
    XPrim W;
    xprim(q + 5 * i, K, W);
    for (int x = 0; x < 3; ++x) u[3 * i + x] = xenc(W.u[x].m, W.u[x].e);
  }
}
""")


def test_doubles_below_the_normal_range(tiny_lib):
    """every double survives; scaled down it is rounded to the nearest multiple of 2^-1074"""
    g = rng(17)
    a = np.concatenate([g.uniform(-1, 1, 4000) * 2.0 ** -1021, g.integers(-2 ** 20, 2 ** 20, 4000) * 2.0 ** -1074,
                        [0.0, 2.0 ** -1074, -2.0 ** -1074, 2.0 ** -1022, np.nextafter(2.0 ** -1022, 0)]])
    b, c, d = (np.empty_like(a) for _ in range(3))
    tiny_lib.again(len(a), _p(a), _p(b), _p(c), _p(d))
    assert np.array_equal(a, b) and np.array_equal(a, c)
    assert np.all(np.abs(d.astype(LD) - a.astype(LD) * LD(2) ** -30) <= LD(2) ** -1075)


def test_velocities_below_the_normal_range(tiny_lib):
    n, g = 2000, rng(18)
    q = np.ones((n, 5))
    q[:, 0] = g.uniform(0.5, 2, n)
    q[:, 1:4] = g.uniform(-1, 1, (n, 3)) * 10.0 ** g.uniform(-315, -306, (n, 3))
    u = np.empty((n, 3))
    tiny_lib.velocity(n, _p(q), _p(u))
    want = q[:, 1:4].astype(LD) / q[:, :1].astype(LD)
    assert np.all(np.abs(u - want) <= LD(2) ** -1074 + ULP * np.abs(want))
