"""The central screen of the fast policy's 1D Euler tiles (wt_central.cuh).

A field of an interface is decided in FP32 only where that proves, on both sides, that the
reconstruction is restricted (Eq. (be_res)) and either theta (Eq. (tau_we6)) or that |Delta^5 v| / 60 is at
most 2^-53 rho (|u| + c), where theta does not matter; an interface takes the central flux C f
where all fields have theta = 0 so.  ``screen`` restates that proof in numpy float32, step by step
as the kernels take it; the CPU test holds every decided field against the decisions in
extended precision.  The GPU tests hold the kernels against the oracle, and every launch
path against the others bit for bit, on data at the screen's edges."""
import numpy as np
import pytest

from paper_1504_00731_gb300 import workloads as W

f4 = np.float32
GM1 = 0.4


def _trunc(x):
    """The leading 24 bits of x as a float, truncated."""
    m, e = np.frexp(np.asarray(x, dtype=np.float64))
    return f4(np.ldexp(np.trunc(np.ldexp(m, 24)), e - 24))


def _pair(x):
    h = _trunc(x)
    return h, _trunc(x - h.astype(np.float64))


def _sub(a, b):
    s = a[0] - b[0]
    bb = s - a[0]
    e = (a[0] - (s - bb)) - (b[0] + bb)
    return s, (a[1] - b[1]) + e


def _high(d):
    s = [_sub(d[k + 1], d[k]) for k in range(4)]
    t = [_sub(s[k + 1], s[k]) for k in range(3)]
    v = [_sub(t[k + 1], t[k]) for k in range(2)]
    w = (v[1][0] - v[0][0]) + (v[1][1] - v[0][1])
    return [t[1][0] + t[1][1], v[0][0] + v[0][1], v[1][0] + v[1][1], w]


def screen(f, U, vel, H, al, eps, aR):
    """Verdicts [field][interface] (0: left to FP64; else 1, + 2 if the + side has theta = 1, + 4 if the - side
    has) from six-cell windows f, U [3][6][n] (float64), and the two centre cells'
    velocity and enthalpy."""
    with np.errstate(all="ignore"):
        r0, r1 = _trunc(U[0, 2]), _trunc(U[0, 3])
        ua, ub, Ha, Hb = _trunc(vel[0]), _trunc(vel[1]), _trunc(H[0]), _trunc(H[1])
        sa, sb = r0 * (f4(1) / np.sqrt(r0)), r1 * (f4(1) / np.sqrt(r1))
        hw = f4(0.5) * (sa - sb) * (f4(1) / (sa + sb))
        du = ua - ub
        u = hw * du + f4(0.5) * (ua + ub)
        Hm = hw * (Ha - Hb) + f4(0.5) * (Ha + Hb)
        Um = np.maximum(np.abs(ua), np.abs(ub))
        he = f4(-0.5) * u * u + Hm
        big = Um * Um + np.maximum(np.abs(Ha), np.abs(Hb))
        c2 = f4(GM1) * he
        ic = f4(1) / np.sqrt(c2)
        b1 = f4(GM1) * (ic * ic)
        rel = f4(2.0**-19) * (big * b1) + f4(2.0**-20)
        q = f4(2.0**-20) * (np.abs(du) / (Um + f4(1e-30))) + f4(1.5 * 2.0**-21)
        thr = f4(60 * 2.0**-53) * np.minimum(r0, r1) * (c2 * ic + np.abs(u))
        ok = (he * f4(32) >= big) & (r0 > 2.0**-60) & (r1 > 2.0**-60) & (r0 < 2.0**60) & (r1 < 2.0**60)
        ok &= (big < 2.0**60) & (big > 2.0**-60)

        def project(x):
            w1 = -u * x[0] + x[1]
            return ic * w1, b1 * (f4(-0.5) * u * (x[1] + w1) + x[2])

        def bound(x):
            n1 = Um * np.abs(x[0]) + np.abs(x[1])
            return ic * n1, b1 * (Um * n1 + np.abs(x[2]))

        parts = []
        for X in (f, U):
            D = [[_pair(X[c, k + 1] - X[c, k]) for k in range(5)] for c in range(3)]
            hi = [_high(D[c]) for c in range(3)]
            vecs = [[D[c][k][0] for c in range(3)] for k in range(5)] + [[hi[c][v] for c in range(3)] for v in range(4)]
            jk = [project(x) for x in vecs]
            mx = [np.max([np.abs(D[c][k][0]) for k in range(5)], axis=0) for c in range(3)]
            nb = [bound(mx)] + [bound(vecs[5 + v]) for v in range(4)]
            jm = np.max([np.abs(jk[k][0]) for k in range(5)], axis=0)
            km = np.max([np.abs(jk[k][1]) for k in range(5)], axis=0)
            parts.append((vecs, jk, nb, jm, km, mx[0]))
        out = []
        for s in range(3):
            A, E = [], []
            for vecs, jk, nb, jm, km, xm in parts:
                A.append([vecs[k][0] - jk[k][1] if s == 1 else jk[k][1] + (-jk[k][0] if s == 0 else jk[k][0])
                          for k in range(9)])

                def err(b, aj, ak, ax):
                    if s == 1:
                        return rel * ak + (q * b[1] + f4(2.0**-22) * ax)
                    return rel * (aj + ak) + q * (b[0] + b[1])

                pe = f4(2.0**-40) * ((xm + nb[0][1]) if s == 1 else (nb[0][0] + nb[0][1]))
                E.append([err(nb[0], jm, km, xm)] + [
                    pe + err(nb[1 + v], np.abs(jk[5 + v][0]), np.abs(jk[5 + v][1]), np.abs(vecs[5 + v][0]))
                    for v in range(4)])
            kap = f4(2 if s == 1 else 4)
            epsk, a = f4(eps) * kap * kap, f4(al[s])
            bm = np.max([np.abs(A[1][k]) for k in range(5)], axis=0)
            eta = a * (f4(2.0**-21) * bm + E[1][0]) + E[0][0]
            eh = [a * (f4(2.0**-21) * np.abs(A[1][5 + v]) + E[1][1 + v]) + E[0][1 + v] for v in range(4)]
            good, verdict = ok.copy(), np.ones(ok.shape, dtype=int)
            C, C3 = f4(13 / 12), f4(13 / 48)
            for side in range(2):
                sa_ = -a if side else a
                d = [sa_ * A[1][4 - k if side else k] + A[0][4 - k if side else k] for k in range(5)]
                s0, s1, s2, s3 = (d[k + 1] - d[k] for k in range(4))
                e0, g3, e3, dd = s0 + d[1], f4(3) * s2 - s3, s3 - d[3], d[2] * d[2]
                B = [C * s0 * s0 + e0 * e0, C * s1 * s1 + dd, C * s2 * s2 + dd, C3 * g3 * g3 + e3 * e3]
                S = np.max(np.abs(d), axis=0)
                dl = f4(54) * S * eta + (f4(27) * eta * eta + f4(2.0**-16) * S * S)
                bx, bn = np.max(B, axis=0), np.min(B, axis=0)
                restricted = bx + dl < f4(aR) * (epsk + (bn - dl)) * f4(1 - 2.0**-18)
                y, z = (7, 6) if side else (6, 7)
                t3 = np.abs(sa_ * A[1][5] + A[0][5])
                ty, tz = sa_ * A[1][y] + A[0][y], sa_ * A[1][z] + A[0][z]
                a5, a6, e6 = np.abs(sa_ * A[1][8] + A[0][8]), np.abs(ty + tz), eh[1] + eh[2]
                t5, lo5 = a5 + eh[3], np.maximum(a5 - eh[3], 0)
                hi3, hi4, lo6 = t3 + eh[0], np.abs(ty) + eh[y - 5], np.maximum(a6 - e6, 0)
                lo3, lo4 = np.maximum(t3 - eh[0], 0), np.maximum(np.abs(ty) - eh[y - 5], 0)
                hi6 = a6 + e6
                t5lo = C * lo4 * lo4 + lo3 * lo3
                t6hi = C * t5 * t5 + f4(0.25) * (hi6 * hi6)
                theta0 = (t6hi * f4(1 + 2.0**-18) < t5lo) & (t5lo > f4(2.0**-100))
                t5hi = C * hi4 * hi4 + hi3 * hi3
                t6lo = C * lo5 * lo5 + f4(0.25) * (lo6 * lo6)
                theta1 = (t5hi * f4(1 + 2.0**-18) < t6lo) & (t6lo > f4(2.0**-100))
                zero = theta0 | (t5 <= thr * kap)
                good &= restricted & (zero | theta1)
                verdict[~zero] |= 4 if side else 2
            out.append(np.where(good, verdict, 0))
        return np.array(out)


def _decide(f, U, vel, H, al, eps, aR):
    """(restricted, tau6 - tau5, |Delta^5 v|, rho (|u| + c)) per field, side and interface in extended
    precision, from the same windows."""
    L = np.longdouble
    f, U, vel, H = f.astype(L), U.astype(L), vel.astype(L), H.astype(L)
    sa, sb = np.sqrt(U[0, 2]), np.sqrt(U[0, 3])
    u, Hm = (sa * vel[0] + sb * vel[1]) / (sa + sb), (sa * H[0] + sb * H[1]) / (sa + sb)
    c = np.sqrt(L(GM1) * (Hm - u * u / 2))
    b1 = L(GM1) / (c * c)
    b2 = u * u * b1 / 2
    rows = [[(b2 + u / c) / 2, -(b1 * u + 1 / c) / 2, b1 / 2], [1 - b2, b1 * u, -b1],
            [(b2 - u / c) / 2, -(b1 * u - 1 / c) / 2, b1 / 2]]
    res = []
    for s in range(3):
        for side in range(2):
            sg = -1 if side else 1
            v = [sum(rows[s][e] * (f[e, k] + sg * L(al[s]) * U[e, k]) for e in range(3)) / 2 for k in range(6)]
            x = v[::-1] if side else v
            b = [L(13) / 12 * (x[0] - 2 * x[1] + x[2])**2 + (x[0] - 3 * x[1] + 2 * x[2])**2,
                 L(13) / 12 * (x[1] - 2 * x[2] + x[3])**2 + (x[3] - x[2])**2,
                 L(13) / 12 * (x[2] - 2 * x[3] + x[4])**2 + (x[3] - x[2])**2,
                 L(13) / 48 * (3 * x[2] - 7 * x[3] + 5 * x[4] - x[5])**2 + (2 * x[3] - 3 * x[4] + x[5])**2]
            t5 = L(13) / 12 * (x[0] - 4 * x[1] + 6 * x[2] - 4 * x[3] + x[4])**2 + (-x[1] + 3 * x[2] - 3 * x[3] + x[4])**2
            d5 = -x[0] + 5 * x[1] - 10 * x[2] + 10 * x[3] - 5 * x[4] + x[5]
            t6 = L(13) / 12 * d5**2 + (x[0] - 3 * x[1] + 2 * x[2] + 2 * x[3] - 3 * x[4] + x[5])**2 / 4
            res.append((np.max(b, axis=0) <= L(aR) * (L(eps) + np.min(b, axis=0)), t6 - t5, np.abs(d5)))
    return res, np.minimum(U[0, 2], U[0, 3]) * (np.abs(u) + c)


def _fields(U):
    rho, m, E = U
    u = m / rho
    p = GM1 * (E - 0.5 * m * u)
    return np.stack([m, m * u + p, (E + p) * u]), u, (E + p) / rho, np.sqrt(1.4 * p / rho)


def _states():
    rng = np.random.default_rng(7)
    for n, kind in [(300, 0), (1200, 0), (5000, 0), (30000, 0), (400, 1), (6000, 1), (800, 2), (4000, 3), (2000, 4)]:
        if kind == 0:  # two states and an entropy wave
            yield W.euler_riemann(n, W.riemann_params(int(rng.integers(1 << 20))))[0]
        elif kind == 1:  # smooth waves in every field, over scales from 1 down to 1e-9
            x = np.linspace(0, 2 * np.pi, n, endpoint=False)
            a = 10.0 ** -np.linspace(0.5, 9, n)
            yield W.cons_1d(1 + a * np.sin(5 * x), 0.7 + a * np.cos(3 * x), 1 + a * np.sin(2 * x + 1))
        elif kind == 2:  # rough data
            yield W.cons_1d(rng.uniform(0.1, 1, n), rng.uniform(-2, 2, n), rng.uniform(0.1, 1, n))
        elif kind == 3:  # high Mach number and a strong pressure jump
            x = np.linspace(-1, 1, n)
            yield W.cons_1d(1 + 0.2 * np.sin(9 * x), 20 + np.sin(4 * x), np.where(x < 0, 1000.0, 0.01))
        else:  # rounding noise on a constant state
            yield W.ulp_perturbed(W.cons_1d(np.full(n, 0.7), np.full(n, 0.3), np.full(n, 0.9)), 3)


@pytest.mark.parametrize("aR", [1.0, 10.0, 50.0])
def test_every_decided_field_is_as_decided(aR):
    eps, central, upwind = 1e-10, 0, 0
    for U in _states():
        f, u, H, c = _fields(U)
        n = U.shape[1] - 5
        idx = np.arange(6)[:, None] + np.arange(n)
        w = (f[:, idx], U[:, idx], np.stack([u[2:n + 2], u[3:n + 3]]), np.stack([H[2:n + 2], H[3:n + 3]]))
        al = [np.abs(u - c).max(), np.abs(u).max(), np.abs(u + c).max()]
        ok = screen(*w, al, eps, aR)
        res, scale = _decide(*w, al, eps, aR)
        for s in range(3):
            for side in range(2):
                restricted, gap, d5 = res[2 * s + side]
                decided, one = ok[s] != 0, (ok[s] & (4 if side else 2)) != 0
                assert np.all(restricted[decided])
                free = d5 <= 60 * np.longdouble(2.0)**-53 * scale
                assert np.all(((gap < 0) | free)[decided & ~one])
                assert np.all((gap > 0)[one])
                upwind += int(one.sum())
        central += int((ok == 1).all(axis=0).sum())
    assert central > 20000 and upwind > 0  # the screen decides most of the smooth data, both ways


torch = pytest.importorskip("torch")


def _edge_state(kind, n):
    x, _ = W.grid_1d(n, -5.0, 5.0, periodic=False)
    wave = 1 + 0.2 * np.sin(5 * x)
    if kind == "shock in a wave":
        return W.cons_1d(np.where(x < 0.3, 3.8, wave), np.where(x < 0.3, 2.6, 0.0), np.where(x < 0.3, 10.3, 1.0))
    if kind == "noise":
        return W.ulp_perturbed(W.cons_1d(np.full(n, 0.7), np.full(n, 0.3), np.full(n, 0.9)), 3)
    if kind == "large values":  # beyond the screen's range
        return W.cons_1d(wave * 2.0**62, 0.4 + 0.1 * np.cos(x), wave * 2.0**62)
    if kind == "small values":
        return W.cons_1d(wave * 2.0**-70, 0.4 + 0.1 * np.cos(x), wave * 2.0**-70)
    if kind == "high Mach":
        return W.cons_1d(wave, 300 + np.cos(x), np.full(n, 0.5))
    return W.cons_1d(wave, 1e-12 * np.sin(2 * x), np.full(n, 1.0))  # a contact at rest: fields 0, 2 cancel


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["shock in a wave", "noise", "large values", "small values", "high Mach", "contact"])
@pytest.mark.parametrize("n", [3, 31, 32, 127, 128, 700, 1369, 2737, 5000])
def test_screened_paths_match_the_oracle_and_each_other(wtlib, oracle, kind, n, monkeypatch):
    """RHS within 1e-13 of the largest |L| per component, or ten times the oracle's own spread over data moved
    by at most one ulp where rounding alone moves L further (cancelling fluxes, high Mach numbers:
    the criterion of the other fast-mode tests); three steps bit for bit the same through the
    persistent kernels, the stage kernels and the batched tiles with one and with several items
    per thread."""
    b, O = wtlib, oracle
    U = _edge_state(kind, n)
    dx = 10.0 / n
    P = O.problem(O.FLUX_EULER1D, bc=O.BC_OUTFLOW, alpha_R=10.0)
    ref = O.rhs(P, U, dx)
    g = b.grid_1d(n, -5.0, 5.0)
    prob = b.problem(b.WT_FLUX_EULER1D, bc=b.WT_BC_OUTFLOW, alpha_R=10.0)
    ws = b.alloc_workspace(b.workspace_bytes(prob, g))
    u0 = torch.from_numpy(U).cuda()
    L = torch.empty_like(u0)
    b.weno_theta_rhs(prob, g, u0, L, ws)
    spread = np.max([np.abs(O.rhs(P, W.ulp_perturbed(U, s), dx) - ref).max(axis=1) for s in range(3)], axis=0)
    tol = np.maximum(1e-13 * np.abs(ref).max(axis=1), 10 * spread)
    assert np.all(np.abs(L.cpu().numpy() - ref).max(axis=1) <= tol)
    runs = []
    for launch in (b.WT_LAUNCH_AUTO, b.WT_LAUNCH_STAGES):
        pl = b.problem(b.WT_FLUX_EULER1D, bc=b.WT_BC_OUTFLOW, alpha_R=10.0, launch=launch)
        u = u0.clone()
        b.weno_theta_step(pl, g, u, 0.5, ws, max_steps=3)
        runs.append(u.cpu().numpy())
    s = b.WtSegment()
    s.offset, s.n, s.lo, s.hi, s.bc_lo, s.bc_hi = 0, n, -5.0, 5.0, b.WT_BC_OUTFLOW, b.WT_BC_OUTFLOW
    wb = b.alloc_workspace(b.workspace_bytes(prob, None, n, 1))
    for code in (31, 2127):
        monkeypatch.setenv("WT_BATCHED_TILE", str(code))
        u = u0.clone()
        b.weno_theta_step_batched(prob, [s], u, n, 0.5, 3, wb)
        runs.append(u.cpu().numpy())
    for r in runs[1:]:
        assert np.array_equal(r, runs[0])


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["front", "smooth", "noise", "large values"])
@pytest.mark.parametrize("nx,ny", [(3, 3), (7, 16), (15, 8), (16, 7), (17, 15), (33, 6), (64, 29), (224, 1260)])
def test_screened_2d_matches_the_oracle(wtlib, oracle, kind, nx, ny):
    """Edges of the 16 x 7 tiles, and a grid of 32 x 7 ones: RHS as above, and one step's maxima (the next
    step's dt) equal to those of the speeds of every cell."""
    b, O = wtlib, oracle
    x, y = np.meshgrid((np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny)
    wave = 1 + 0.2 * np.sin(2 * np.pi * (x + 2 * y))
    one = np.ones((ny, nx))
    scale = 2.0**62 if kind == "large values" else 1.0
    if kind == "front":
        U = W.cons_2d(np.where(x + y > 0.8, 1.0, 0.125), 0.3 * wave, 0.1 * one, np.where(x + y > 0.8, 1.0, 0.1))
    elif kind == "noise":
        U = W.ulp_perturbed(W.cons_2d(0.7 * one, 0.3 * one, 0.2 * one, 0.9 * one), 5)
    else:
        U = W.cons_2d(wave * scale, 0.4 + 0.1 * np.cos(2 * np.pi * y), 0.2 * wave, wave * scale)
    dx, dy = 1.0 / nx, 1.0 / ny
    P = O.problem(O.FLUX_EULER2D, bc=0, alpha_R=10.0)
    ref = O.rhs(P, U, dx, dy)
    spread = np.max([np.abs(O.rhs(P, W.ulp_perturbed(U, s), dx, dy) - ref).max(axis=(1, 2)) for s in range(3)], axis=0)
    tol = np.maximum(1e-13 * np.abs(ref).max(axis=(1, 2)), 10 * spread)
    g = b.grid_2d(nx, ny)
    prob = b.problem(b.WT_FLUX_EULER2D, alpha_R=10.0)
    ws = b.alloc_workspace(b.workspace_bytes(prob, g))
    u = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    L = torch.empty_like(u)
    b.weno_theta_rhs(prob, g, u, L, ws)
    assert np.all(np.abs(L.cpu().numpy() - ref).max(axis=(1, 2)) <= tol)
    # two steps in one call, and in two: the second call takes the speeds of every cell (alpha2d)
    v, w = u.clone(), u.clone()
    t2, _ = b.weno_theta_step(prob, g, v, 0.4, ws, max_steps=2)
    ta, _ = b.weno_theta_step(prob, g, w, 0.4, ws, max_steps=1)
    tb, _ = b.weno_theta_step(prob, g, w, 0.4, ws, max_steps=1)
    assert torch.equal(v, w) and t2 == ta + tb
