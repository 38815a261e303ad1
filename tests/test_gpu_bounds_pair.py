"""FP64 bounds on float pairs (grids of 3.75 or more velocity nodes per thermal unit): against the
checker at the edges of the velocity tiles and stencil capacities, on both sides of the rule that
selects the pairs, and on stencils that leave the pairs' range and run on the FP64 pipe.

Tolerance: a node's envelope is valued to 2^-47 and the checker's sums to about 1e-15 of the sums'
magnitudes, so 1e-13 of each component's scale leaves a factor of ten."""
import numpy as np
import pytest

from paper_2407_20966_gb300 import inputs
from tests.gpu_helpers import bounds_error, to_dev, zeros_dev

pytestmark = pytest.mark.gpu
TOL = 1e-13


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_20966_gb300 import build
    build.build()


def _check(orc, S, nu, tol=TOL, **kw):
    from paper_2407_20966_gb300 import kbl
    E = len(S)
    ctx = kbl.Context(dim=2, p=3, nu=(nu, nu), precision=kbl.FP64, **kw)
    bnd = zeros_dev(2, 4, E)
    ctx.bounds_stencil(to_dev(S), bnd)
    ctx.check()
    cfg = orc.Config(dim=2, p=3, nu=(nu, nu), **kw)
    ref = np.zeros((2, 4, E))
    for e in range(E):
        ref[0, :, e], ref[1, :, e] = orc.bounds_stencil(cfg, S[e])
    got = bnd.cpu().numpy()
    assert np.isfinite(got).all()
    with np.errstate(invalid="ignore"):   # equal values (0 and 0 where the checker underflows) have no error
        err = np.where(got == ref, 0.0, bounds_error(got, ref)).max()
    assert err < tol, err


def _states(seed, E, n, spread=0.3):
    rng = np.random.default_rng(seed)
    base = inputs.random_states(rng, E, 2)
    S = np.repeat(base[:, None, :], n, axis=1) * (1.0 + spread * rng.uniform(-1.0, 1.0, (E, n, 4)))
    ke = 0.5 * (S[..., 1] ** 2 + S[..., 2] ** 2) / S[..., 0]
    S[..., 3] = np.maximum(S[..., 3], 1.05 * ke + 1e-3)
    return S


@pytest.mark.parametrize("n,nu,kw", [
    (1, 32, {}), (17, 31, {}), (48, 30, {}), (48, 33, dict(quadrature=1)), (24, 40, {}), (41, 41, {}),
    (64, 48, {}), (33, 49, {}), (16, 61, dict(k=8.0)), (16, 60, dict(k=8.0)), (64, 64, {}), (7, 25, dict(k=3.0)),
    (20, 65 - 1, dict(k=8.0, r_fac=0.0)), (15, 24, {}), (15, 48, dict(k=8.0)), (12, 32, dict(gamma=2.0))])
def test_tiles_and_rule(orc, n, nu, kw):
    _check(orc, _states(n + nu, 11, n), nu, **kw)


@pytest.mark.parametrize("scale,speed", [(1e-30, 1.0), (1e60, 1e25), (1.0, 1e-20), (1e-200, 1e90)])
def test_scaled_states(orc, scale, speed):
    """Densities and velocities scaled over and beyond the FP32 range."""
    S = _states(5, 9, 24) * scale
    S[..., 1:3] *= speed
    S[..., 3] *= speed * speed
    _check(orc, S, 32, rho_floor=0.0)


@pytest.mark.parametrize("ratio", [3.0, 10.0, 30.0, 1e3, 1e6])
def test_strong_jumps(orc, ratio):
    """Half of each stencil `ratio` times hotter: from 30 on its cold Maxwellians underflow the
    pairs inside the box and the element runs on the FP64 pipe."""
    S = _states(6, 9, 24, spread=0.02)
    S[:, 12:, 3] += (ratio - 1) * (S[:, 12:, 3] - 0.5 * (S[:, 12:, 1] ** 2 + S[:, 12:, 2] ** 2) / S[:, 12:, 0])
    _check(orc, S, 32)
    _check(orc, S, 40)


def test_fast_streams(orc):
    """Two cold streams through each other: tiny lower sums, far from the largest state's."""
    for v in (4.0, 12.0, 40.0):
        S = _states(7, 5, 20, spread=0.02)
        S[:, :10, 3] += v * (S[:, :10, 1] + 0.5 * v * S[:, :10, 0])   # the boost's kinetic energy
        S[:, :10, 1] += v * S[:, :10, 0]
        _check(orc, S, 32)
    S = inputs.random_states(np.random.default_rng(8), 40, 2, vel=(50.0, 60.0)).reshape(5, 8, 4)
    _check(orc, S, 32)


def _line(orc, w, mesh, p, nu, tol=TOL, **kw):
    from paper_2407_20966_gb300 import kbl
    E = mesh.n_elem
    ctx = kbl.Context(dim=1, p=p, nu=(nu,), precision=kbl.FP64, **kw)
    ctx.mesh_upload(mesh.nbr, mesh.h, mesh.bc)
    cfg = orc.Config(dim=1, p=p, nu=(nu,), **kw)
    wf, bnd = zeros_dev(3, E, 2), zeros_dev(2, 3, E)
    wd = to_dev(w)
    ctx.traces(wd, wf)
    ctx.bounds(wd, wf, bnd)
    ctx.check()
    om = orc.Mesh(mesh.nbr, mesh.h, mesh.bc)
    ref = orc.bounds(cfg, om, w, wf.cpu().numpy())
    got = bnd.cpu().numpy()
    with np.errstate(invalid="ignore"):
        err = np.where(got == ref, 0.0, bounds_error(got, ref)).max()
    assert err < tol, err


def _line_field(p, n=23, seed=0):
    mesh = inputs.mesh_1d(n, 0.0, 1.0, periodic=True)
    xi = np.polynomial.legendre.leggauss(p + 1)[0]
    return mesh, inputs.random_discontinuous_field(np.random.default_rng(seed), mesh, xi)


@pytest.mark.parametrize("p,nu,kw", [
    (1, 2, {}), (2, 3, {}), (3, 5, {}), (4, 63, {}), (3, 64, {}), (5, 65, dict(quadrature=1)), (3, 255, {}),
    (2, 257, dict(quadrature=1, k=8.0)), (4, 2048, dict(k=8.0, r_fac=0.0)), (1, 4096, {}),
    (3, 64, dict(stencil=1)), (5, 100, dict(stencil=1)), (3, 64, dict(gamma=3.0))])
def test_line_nodes_and_stencils(orc, p, nu, kw):
    """1D: node counts around the block sizes, both stencils, delta = 0."""
    mesh, w = _line_field(p)
    _line(orc, w, mesh, p, nu, **kw)


@pytest.mark.parametrize("ratio", [3.0, 30.0, 1e5])
def test_line_jumps_and_scales(orc, ratio):
    """1D jumps that leave the floats' range inside the box, and scaled states."""
    mesh, ic = inputs.riemann_1d(12, (1.0, 0.3, ratio), (0.5, -0.2, 1.0), 0.0, 1.0, 0.5)
    w = inputs.nodal_field(mesh, np.polynomial.legendre.leggauss(4)[0], ic)
    _line(orc, w, mesh, 3, 64)
    s = np.array([1e-40, 1e-40 * 1e30, 1e-40 * 1e60])
    mesh.bc = mesh.bc * s
    _line(orc, w * s[:, None, None], mesh, 3, 100, rho_floor=0.0)
