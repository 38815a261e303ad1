"""FP64 2D bounds, every lower and upper bound relative to itself, against sums in extended precision
(numpy long double): small lower sums count as much as large ones here.

Worst-case tolerance.  A node's Maxwellian is the product of two table entries of 2^-48 each, its
envelope value takes three FP32 roundings of a rest of 2^-23 or less, 2^-47 at most each, and the rest
of the sums are FP64: 2^-45 covers them.  The FP64 roundings of the state, of 2^-53 each, move the
exponent z^2 / 2 = (u - U)^2 / (2 theta), in the FP64 kernel as in the pairs: three in theta and three
more amplified by the cancellation E / (E - K) of its pressure, z^2 / 2 (3 + 3 E / (E - K)); three in
u - U, z 3 (|u| + |U|) / sqrt(theta).  Their sum at its largest over the states."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
L = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_20966_gb300 import build
    build.build()


def _cons(rho, u, v, th, gamma=1.4):
    return np.stack([rho, rho * u, rho * v, rho * th / (gamma - 1.0) + 0.5 * rho * (u * u + v * v)], -1)


def _reference(S, nu, k, quad, gamma=1.4):
    """Bounds [2][4], the sums of the terms' magnitudes [2][4], the worst-case tolerance, the largest
    exponent argument |u - U| sqrt(log2(e) / (2 theta)) and the scaled lower density sum."""
    from paper_2407_20966_gb300 import kbl
    S = S.astype(L)
    rho, U = S[:, 0], S[:, 1:3] / S[:, :1]
    K = L(0.5) * (S[:, 1] ** 2 + S[:, 2] ** 2) / rho
    P = (L(gamma) - L(1)) * (S[:, 3] - K)
    th = P / rho
    s = L(k) * np.sqrt(th)
    lo, hi = (U - s[:, None]).min(0), (U + s[:, None]).max(0)
    h = (hi - lo) / (nu - 1)
    u = [lo[d] + np.arange(nu).astype(L) * h[d] for d in (0, 1)]
    q = kbl.velocity_weights(nu, quad).astype(L)
    z = [(u[d][None] - U[:, d:d + 1]) / np.sqrt(th)[:, None] for d in (0, 1)]
    A = rho / (8 * np.arctan(L(1)) * th)
    ex, ey = A[:, None] * np.exp(-z[0] ** 2 / 2), np.exp(-z[1] ** 2 / 2)
    C = (L(1) / (L(gamma) - L(1)) - L(1)) * th
    T = [np.full((nu, nu), np.inf, L), np.zeros((nu, nu), L)]
    I = [T[0].copy(), T[1].copy()]
    for i in range(len(S)):
        g = ex[i][:, None] * ey[i][None]
        T = [np.minimum(T[0], g), np.maximum(T[1], g)]
        I = [np.minimum(I[0], C[i] * g), np.maximum(I[1], C[i] * g)]
    M = (q * h[0])[:, None] * (q * h[1])[None]
    ke = L(0.5) * (u[0][:, None] ** 2 + u[1][None] ** 2)
    out, mag = np.zeros((2, 4), L), np.zeros((2, 4), L)
    for b in (0, 1):
        out[b, 0] = (M * T[b]).sum()
        out[b, 3] = (M * (T[b] * ke + I[b])).sum()
        for d in (0, 1):
            ud = u[0][:, None] if d == 0 else u[1][None]
            t = M * ud * np.where(ud < 0, T[1 - b], T[b])
            out[b, 1 + d], mag[b, 1 + d] = t.sum(), np.abs(t).sum()
    mag[:, [0, 3]] = out[:, [0, 3]]
    zm = max(float(np.abs(a).max()) for a in z)
    speed = float((np.abs(np.stack([lo, hi])).max() + np.abs(U).max()) / np.sqrt(th.min()))
    cond = zm * 3 * speed + zm * zm / 2 * (3 + 3 * float((S[:, 3] / (S[:, 3] - K)).max()))
    e = int(np.floor(np.log2(float((rho / th).max()))))
    return out, mag, 2.0 ** -45 + 2.0 ** -53 * cond, 0.8493218002880191 * zm, float(out[0, 0] / (h[0] * h[1])) * 2.0 ** -e


def _bounds(S, nu, k, quad):
    import torch
    from paper_2407_20966_gb300 import kbl
    ctx = kbl.Context(dim=2, p=3, nu=(nu, nu), precision=kbl.FP64, k=k, quadrature=quad, r_fac=0.0, rho_floor=0.0)
    bnd = torch.zeros((2, 4, len(S)), dtype=torch.float64, device="cuda")
    ctx.bounds_stencil(torch.from_numpy(np.ascontiguousarray(S)).cuda(), bnd)
    ctx.check()
    return bnd.cpu().numpy()


def _streams(sep, angle, th, ratio, n, E=4):
    """Half of each stencil `sep` thermal speeds from the other half along `angle`, `ratio` times as dense."""
    rng = np.random.default_rng([int(10 * sep), n])
    g = np.where(np.arange(n) % 2 == 0, -0.5, 0.5)[None] * sep * np.sqrt(th)
    r = np.where(np.arange(n) % 2 == 0, ratio, 1.0)[None] * (1 + 0.1 * rng.uniform(-1, 1, (E, n)))
    d = 0.02 * np.sqrt(th) * rng.uniform(-1, 1, (2, E, n))
    return _cons(r, g * np.cos(angle) + d[0], g * np.sin(angle) + d[1], th * (1 + 0.02 * rng.uniform(-1, 1, (E, n))))


GRIDS = [(31, 4.0, 0), (32, 4.0, 0), (33, 4.0, 1), (33, 4.0, 0), (36, 4.0, 0), (40, 4.0, 0), (41, 4.0, 1),
         (48, 4.0, 0), (49, 4.0, 0), (64, 8.0, 0)]


@pytest.mark.parametrize("nu,k,quad", GRIDS)
@pytest.mark.parametrize("sep,angle,th,ratio,n", [
    (11.0, 0.0, 0.25, 1.0, 2), (12.0, 0.0, 1.0, 1.0, 2), (8.0, 0.0, 1.0, 1e-4, 24), (9.0, 1.57, 0.3, 1.0, 17),
    (7.0, 0.7, 1.0, 1.0, 48), (14.4, 0.785, 1.0, 1.0, 24), (3.0, 0.0, 1.0, 1e-8, 24), (3.0, 0.4, 0.5, 1e-3, 41)])
def test_small_lower_sums(sep, angle, th, ratio, n, nu, k, quad):
    """Lower sums from 2^-39 to 1e-3 of the upper ones, on grids that fill their tile and grids that
    do not.  With 8 thermal units each side the wider ones leave the pairs' range; the tolerance is
    the same there."""
    S = _streams(sep, angle, th, ratio, n)
    got = _bounds(S, nu, k, quad)
    for e in range(len(S)):
        ref, mag, tol, z, s = _reference(S[e], nu, k, quad)
        if k == 4.0:   # on the pairs: the range test of the kernel
            assert z < 15.3 and s >= 2.0 ** -40, (z, s)
        err = (np.abs(got[:, :, e].astype(L) - ref) / mag).astype(float)
        assert err.max() < tol, (e, err, tol)


@pytest.mark.parametrize("nu,k", [(64, 4.0), (513, 8.0)])
def test_line_states_equal_to_rounding(nu, k):
    """1D stencils whose states differ by 1e-15 of themselves: the envelopes still take the smallest and
    the largest Maxwellian.  The roundings of a bound have no sign of their own: over 256 elements the
    mean error of the upper densities less that of the lower ones stays below 2^-53 (winners picked to
    2^-48 leave 2^-51)."""
    import torch
    from paper_2407_20966_gb300 import kbl
    E, n = 256, 9
    rng = np.random.default_rng(11)
    r, u, th = rng.uniform(0.5, 2, (E, 1)), rng.uniform(-1, 1, (E, 1)), rng.uniform(0.5, 2, (E, 1))
    S = np.stack([r, r * u, 2.5 * r * th + 0.5 * r * u * u], -1) * (1 + 1e-15 * rng.uniform(-1, 1, (E, n, 3)))
    ctx = kbl.Context(dim=1, p=4, nu=(nu,), precision=kbl.FP64, k=k, r_fac=0.0, rho_floor=0.0)
    nbr = np.array([[-(2 * e + 1), -(2 * e + 2)] for e in range(E)], dtype=np.int32)
    ctx.mesh_upload(nbr, np.ones((E, 1)), S[:, 7:].reshape(2 * E, 3))
    w, wf = (torch.from_numpy(np.ascontiguousarray(x.transpose(2, 0, 1))).cuda() for x in (S[:, :5], S[:, 5:7]))
    bnd = torch.zeros((2, 3, E), dtype=torch.float64, device="cuda")
    ctx.bounds(w, wf, bnd)
    ctx.check()
    got = bnd.cpu().numpy()
    q = kbl.velocity_weights(nu, 0).astype(L)
    err = np.zeros((2, E))
    for e in range(E):
        s = S[e].astype(L)
        U = s[:, 1] / s[:, 0]
        t = (L(1.4) - L(1)) * (s[:, 2] - s[:, 1] ** 2 / (2 * s[:, 0])) / s[:, 0]
        lo, hi = (U - k * np.sqrt(t)).min(), (U + k * np.sqrt(t)).max()
        h = (hi - lo) / (nu - 1)
        v = lo + np.arange(nu).astype(L) * h
        g = (s[:, 0] / np.sqrt(8 * np.arctan(L(1)) * t))[:, None] * np.exp(-(v[None] - U[:, None]) ** 2 / (2 * t[:, None]))
        for b, f in enumerate((g.min(0), g.max(0))):
            ref = (q * f).sum() * h
            err[b, e] = float((L(got[b, 0, e]) - ref) / ref)
    assert abs(err[1].mean() - err[0].mean()) < 2.0 ** -53, err.mean(1)


def _rms_sets():
    rng = np.random.default_rng(21)
    E, n = 24, 33
    u = lambda a, b, s=(E, n): rng.uniform(a, b, s)
    x, y = u(-1, 1), u(-1, 1)
    g = u(-0.1, 0.1, (8, E, 1))
    smooth = _cons(1 + g[0] * x + g[1] * y, 0.3 + g[2] * x + g[3] * y, -0.2 + g[4] * x + g[5] * y, 1 + g[6] * x + g[7] * y)
    r, t = u(0.5, 1.5, (E, 1)), u(0.5, 1.5, (E, 1))
    nodes = _cons(r * u(0.8, 1.2), u(-1, 1, (E, 1)) + u(-0.2, 0.2), u(-1, 1, (E, 1)) + u(-0.2, 0.2), t * u(0.8, 1.2))
    factors = _cons(u(0.1, 2.0), u(-1, 1), u(-1, 1), u(0.5, 2.0))
    return {"smooth": (smooth, 3e-16), "nodes": (nodes, 3e-16), "factors": (factors, 4.5e-16)}


@pytest.mark.parametrize("nu,k,quad", [(32, 4.0, 0), (33, 4.0, 1), (40, 4.0, 0), (48, 4.0, 0), (64, 8.0, 0)])
@pytest.mark.parametrize("which", ["smooth", "nodes", "factors"])
def test_stated_errors(which, nu, k, quad):
    """The rms errors that include/kbl.h states for the pairs: below 3e-16 for smooth and moderately
    scattered states over all bounds and over the lower ones of density and energy; below 4.5e-16 where
    the states of a stencil differ by factors."""
    S, stated = _rms_sets()[which]
    got = _bounds(S, nu, k, quad)
    err = np.zeros(got.shape)
    for e in range(len(S)):
        ref, mag, _, _, _ = _reference(S[e], nu, k, quad)
        err[:, :, e] = (np.abs(got[:, :, e].astype(L) - ref) / mag).astype(float)
    rms, low = np.sqrt((err ** 2).mean()), np.sqrt((err[0, [0, 3]] ** 2).mean())
    assert rms < stated and low < stated, (rms, low)
