"""FP64 residuals where values of very different size meet, each component by its own size: a spanwise velocity far
below the others on extruded states, and cells beside a strong jump.  The reference is the schemes in long double (the
FP64 oracle's own rounding of the large components reaches the small one)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1710_09995_gb300 import cases  # noqa: E402

LD = np.longdouble
G, PR, EPS = LD(1.4), LD(0.72), LD(0.1)


@pytest.fixture(scope="module")
def gb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09995_gb300 import gbcfd
    gbcfd.lib()
    return gbcfd


# ---- periodic blocks in long double: arrays [...][z][y][x], d = 0 along x --------------------------

def at(a, d, s):
    """the value s cells further along d"""
    return np.roll(a, -s, a.ndim - 1 - d)


def prim(q):
    u = q[1:4] / q[0]
    return np.concatenate([q[:1], u, ((G - 1) * (q[4] - q[0] * (u * u).sum(0) / 2))[None]])


def roe(l, r, S):
    """the Roe flux with Harten's fix through area vectors S"""
    area = np.sqrt((S * S).sum(0))
    n = S / area
    ul, ur = (l[1:4] * n).sum(0), (r[1:4] * n).sum(0)
    h = lambda w: G / (G - 1) * w[4] / w[0] + (w[1:4] * w[1:4]).sum(0) / 2
    hl, hr, sl, sr = h(l), h(r), np.sqrt(l[0]), np.sqrt(r[0])
    al, ar, rt = sl / (sl + sr), sr / (sl + sr), sl * sr
    v, ht = al * l[1:4] + ar * r[1:4], al * hl + ar * hr
    q2 = (v * v).sum(0)
    c2 = (G - 1) * (ht - q2 / 2)
    c, un = np.sqrt(c2), (v * n).sum(0)
    dr, dp, dn = r[0] - l[0], r[4] - l[4], ur - ul
    a1, a5, a2 = (dp - rt * c * dn) / (2 * c2), (dp + rt * c * dn) / (2 * c2), dr - dp / c2
    sh = rt * (r[1:4] - l[1:4] - dn * n)
    de = EPS * (abs(un) + c)
    fix = lambda x: np.where(abs(x) < de, (x * x + de * de) / (2 * de), abs(x))
    w1, w2, w5, l2 = fix(un - c) * a1, fix(un) * a2, fix(un + c) * a5, fix(un)
    side = lambda w, un_, h_: np.concatenate([(w[0] * un_)[None], w[0] * un_ * w[1:4] + w[4] * n, (w[0] * un_ * h_)[None]])
    F = side(l, ul, hl) + side(r, ur, hr)
    F[0] -= w1 + w2 + w5
    F[1:4] -= w1 * (v - c * n) + w2 * v + l2 * sh + w5 * (v + c * n)
    F[4] -= w1 * (ht - c * un) + w2 * q2 / 2 + l2 * (v * sh).sum(0) + w5 * (ht + c * un)
    return F * area / 2


def cartesian(c):
    S = np.zeros((3, 3, c.nz, c.ny, c.nx), LD)
    h = [LD(x) for x in c.spacing]
    for d in range(3):
        S[d, d] = h[(d + 1) % 3] * h[(d + 2) % 3]
    return S, np.full((c.nz, c.ny, c.nx), h[0] * h[1] * h[2])


def plane_metrics(nodes):
    """lower-face area vectors and volumes of a grid extruded in z"""
    X = nodes.astype(LD)
    x, y, dz = X[0, 0], X[1, 0], X[2, 1, 0, 0] - X[2, 0, 0, 0]
    nz = X.shape[1] - 1
    dx, dy = lambda a: a[:, 1:] - a[:, :-1], lambda a: a[1:] - a[:-1]
    A = ((x[1:, 1:] - x[:-1, :-1]) * (y[1:, :-1] - y[:-1, 1:]) - (y[1:, 1:] - y[:-1, :-1]) * (x[1:, :-1] - x[:-1, 1:])) / -2
    S = np.zeros((3, 3) + A.shape, LD)
    S[0, 0], S[0, 1] = dy(y)[:, :-1] * dz, -dy(x)[:, :-1] * dz
    S[1, 0], S[1, 1] = -dx(y)[:-1] * dz, dx(x)[:-1] * dz
    S[2, 2] = abs(A)
    return np.repeat(S[:, :, None], nz, 2), np.repeat(abs(A)[None] * dz, nz, 0)


def fv_residual(c, S, V):
    w = prim(c.state.astype(LD))
    R = np.zeros_like(w)
    mm = lambda a, b: np.where((a > 0) == (b > 0), np.where(abs(a) < abs(b), a, b), LD(0))
    phi, kap = np.concatenate([w[1:4], (w[4] / w[0])[None]]), LD(c.mu) * G / ((G - 1) * PR)
    for d in range(3):
        s = [at(w, d, o) for o in (-2, -1, 0, 1)]
        F = roe(s[1] + mm(s[1] - s[0], s[2] - s[1]) / 2, s[2] - mm(s[2] - s[1], s[3] - s[2]) / 2, S[d])
        if c.viscous:  # uniform grids
            h, L = [LD(x) for x in c.spacing], at(phi, d, -1)
            g = [sum(at(a, t, 1) - at(a, t, -1) for a in (L, phi)) / (4 * h[t]) if t != d else (phi - L) / h[d] for t in range(3)]
            div = g[0][0] + g[1][1] + g[2][2]
            tau = [LD(c.mu) * (g[d][a] + g[a][d]) - (LD(2) / 3 * LD(c.mu) * div if a == d else 0) for a in range(3)]
            F[1:] -= np.stack(tau + [sum((L[a] + phi[a]) / 2 * tau[a] for a in range(3)) + kap * g[d][3]]) * S[d, d]
        R += at(F, d, 1) - F
    return R / V


def wcns_residual(c):
    w, h = prim(c.state.astype(LD)), [LD(x) for x in c.spacing]
    R = np.zeros_like(w)

    def edge(u):
        g = [(u[0] - 4 * u[1] + 3 * u[2]) / 2, (u[3] - u[1]) / 2, (-3 * u[2] + 4 * u[3] - u[4]) / 2]
        s = [u[0] - 2 * u[1] + u[2], u[1] - 2 * u[2] + u[3], u[2] - 2 * u[3] + u[4]]
        a = [k / (LD(1e-6) + x * x + y * y) ** 2 for k, x, y in zip((1, 10, 5), g, s)]
        return u[2] + sum(k * (x / 2 + y / 8) for k, x, y in zip(a, g, s)) / sum(a)

    for d in range(3):
        n = np.zeros((3,) + w.shape[1:], LD)
        n[d] = 1
        F = roe(edge([at(w, d, o) for o in (-2, -1, 0, 1, 2)]), edge([at(w, d, o) for o in (3, 2, 1, 0, -1)]), n)
        for k, o in ((LD(75) / 64, 0), (-LD(25) / 384, 1), (LD(3) / 640, 2)):
            R += (at(F, d, o) - at(F, d, -1 - o)) * (k / h[d])
    if c.viscous:
        d4 = lambda a, d: (at(a, d, -2) - 8 * at(a, d, -1) + 8 * at(a, d, 1) - at(a, d, 2)) / (12 * h[d])
        phi, mu = np.concatenate([w[1:4], (w[4] / w[0])[None]]), LD(c.mu)
        g = [d4(phi, d) for d in range(3)]
        div, kap = g[0][0] + g[1][1] + g[2][2], mu * G / ((G - 1) * PR)
        for d in range(3):
            tau = [mu * (g[d][a] + g[a][d]) - (LD(2) / 3 * mu * div if a == d else 0) for a in range(3)]
            R[1:] -= d4(np.stack(tau + [sum(w[1 + a] * tau[a] for a in range(3)) + kap * g[d][3]]), d)
    return R


# ---- extruded states ------------------------------------------------------------------------------

def extruded(size, viscous, n=(40, 24, 8), seed=5):
    """a smooth state that does not vary along z, w about `size`"""
    nx, ny, nz = n
    g = np.random.Generator(np.random.PCG64(seed))
    X, Y = np.meshgrid((np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny, indexing="xy")
    f = lambda: sum(g.uniform(0.3, 1) * np.sin(2 * np.pi * (i * X + j * Y) + g.uniform(0, 6.3)) for i, j in ((1, 0), (0, 1), (1, 2)))
    r, u, v, w, p = 1 + 0.05 * f(), 0.5 + 0.1 * f(), 0.2 + 0.1 * f(), size * (1 + 0.2 * f()), (1 + 0.05 * f()) / 1.4
    q = np.ascontiguousarray(np.repeat(cases.conserved(r, u, v, w, p)[:, None], nz, 1))
    return cases.Case("extruded", nx, ny, nz, q, None, (1 / nx, 1 / ny, 1 / nz), mu=2e-3 if viscous else 0.0, viscous=viscous)


def curved_in_the_plane(nx, ny, nz):
    """grid points of a grid curved in x and y and extruded in z, multiples of 2^-14 (the area vectors, differences of
    products of theirs, are then exact: x- and y-faces have none along z)"""
    x, y, z = (np.arange(m + 1) / m for m in (nx, ny, nz))
    Z, Y, X = np.meshgrid(z, y, x, indexing="ij")
    q = lambda a: np.round(a * 2.0 ** 14) / 2.0 ** 14
    return np.ascontiguousarray(np.stack([q(X + 0.05 * np.sin(2 * np.pi * Y)), q(Y + 0.05 * np.sin(2 * np.pi * X)), Z]))


# the FP64 form rounds each flux of a component some 100 times at 1.1e-16 of it, and a difference of fluxes is
# some 10 times smaller than they are: 1e-13
COMPONENT = 1e-13


def by_component(R, ref):
    return [float(np.linalg.norm((R[m] - ref[m]).astype(np.float64)) / np.linalg.norm(ref[m].astype(np.float64))) for m in range(5)]


def gpu_residual(block):
    return block.compute_residual().cpu().numpy()


@pytest.mark.parametrize("size", [1.0, 1e-3, 1e-6, 1e-9])
def test_spanwise_momentum_on_an_extruded_grid(gb, size):
    c = extruded(size, False)
    c.nodes = curved_in_the_plane(c.nx, c.ny, c.nz)
    err = by_component(gpu_residual(gb.block_for_case(c, precision=gb.FP64)), fv_residual(c, *plane_metrics(c.nodes)))
    assert max(err) <= COMPONENT, err


# ---- a strong jump --------------------------------------------------------------------------------

def halves(n=(48, 8, 8), seed=9):
    """a smooth slow state with density and pressure 1 for x < 1/2, 1e-4 and 1e-7 beyond (and the jump back at the
    periodic boundary); the size of a residual's components in each cell, from the cell's own state"""
    nx, ny, nz = n
    c = cases.smooth_random(nx, ny, nz, seed=seed, amp=0.1)
    w = np.stack([c.state[0], *(c.state[1:4] / c.state[0]), 0.4 * (c.state[4] - 0.5 * (c.state[1:4] ** 2).sum(0) / c.state[0])])
    w[1:4] *= 1e-2
    w[0, :, :, nx // 2:] *= 1e-4
    w[4, :, :, nx // 2:] *= 1e-7
    c.state = cases.conserved(*w)
    s = np.abs(w[1:4]).sum(0) + np.sqrt(1.4 * w[4] / w[0])
    return c, np.stack([w[0] * s, w[0] * s * s, w[0] * s * s, w[0] * s * s, w[0] * s ** 3]) / min(c.spacing)


@pytest.mark.parametrize("curved,viscous", [(False, False), (False, True), (True, False)])
def test_cells_beside_a_jump(gb, curved, viscous):
    """every face at the jump, and those whose stencil it enters from beyond; in cells of the low side that have no face at
    it errors stay relative to that side (some 100 roundings of 1.1e-16)"""
    c, size = halves()
    c.viscous, c.mu = viscous, 1e-7 if viscous else 0.0  # stresses about the size of the low side's fluxes
    if curved:
        c.nodes = curved_in_the_plane(c.nx, c.ny, c.nz)
    ref = fv_residual(c, *(plane_metrics(c.nodes) if curved else cartesian(c)))
    R = gpu_residual(gb.block_for_case(c, precision=gb.FP64))
    assert max(by_component(R, ref)) <= COMPONENT
    low = slice(c.nx // 2 + 1, c.nx - 1)
    assert np.all(np.abs(R - ref)[..., low] <= COMPONENT * size[..., low])


@pytest.mark.parametrize("viscous", [False, True])
@pytest.mark.parametrize("size", [1.0, 1e-3, 1e-6, 1e-9])
def test_spanwise_momentum_on_a_uniform_grid(gb, size, viscous):
    c = extruded(size, viscous)
    err = by_component(gpu_residual(gb.block_for_case(c, precision=gb.FP64)), fv_residual(c, *cartesian(c)))
    assert max(err) <= COMPONENT, err


@pytest.mark.parametrize("viscous", [False, True])
@pytest.mark.parametrize("size", [1.0, 1e-3, 1e-6, 1e-9])
def test_spanwise_momentum_wcns(gb, size, viscous):
    """the viscous part alone too, as the difference of the residuals with and without viscosity (the inviscid
    parts subtracted are some 10 times as large)"""
    c = extruded(size, viscous)
    R, ref = gpu_residual(gb.wcns_block_for_case(c, precision=gb.FP64)), wcns_residual(c)
    err = by_component(R, ref)
    assert max(err) <= COMPONENT, err
    if viscous:
        c.viscous = False
        R = R - gpu_residual(gb.wcns_block_for_case(c, precision=gb.FP64))
        ref = ref - wcns_residual(c)
        err = [float(np.linalg.norm(R[m] - ref[m]) / np.linalg.norm(ref[m])) for m in (1, 2, 3)]
        assert max(err) <= 10 * COMPONENT, err


def test_cells_beside_a_jump_wcns(gb):
    """the same for WCNS-E-5, in cells of the low side with no edge of Eq. 2 at the jump; the weights there are some
    10^12 apart and carry 20 roundings to what they let in"""
    c, size = halves()
    ref = wcns_residual(c)
    R = gpu_residual(gb.wcns_block_for_case(c, precision=gb.FP64))
    assert max(by_component(R, ref)) <= COMPONENT
    low = slice(c.nx // 2 + 4, c.nx - 4)
    assert np.all(np.abs(R - ref)[..., low] <= COMPONENT * size[..., low])
