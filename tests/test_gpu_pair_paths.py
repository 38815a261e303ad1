"""FP64 paths on the default 32-node grid that run other kernels than the 16-node tests reach: triangle
bounds and steps on float pairs, the FP64 triangle residual of meshes beyond two blocks per SM, quads
of every order on pairs, and pair bounds in the branched step graph.  Tolerances are the FP64 ones of
the tests of the same calls on 16 nodes."""
import numpy as np
import pytest

from paper_2407_20966_gb300 import inputs
from tests.gpu_helpers import TOL_FP64, both, bounds_error, mesh_and_field, to_dev, upload, zeros_dev
from tests.test_gpu_triangles import _elem_scale, _residual_scale, _smooth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_20966_gb300 import build
    build.build()


def _tri(orc, p, nx, ny, curved, flux=1, nu=32):
    from paper_2407_20966_gb300 import kbl
    make = inputs.tri_curved_mesh if curved else inputs.tri_mesh_2d
    m = make(nx, ny, 0.0, 1.0, 0.0, 0.9, jitter=0.1 if curved else 0.2, seed=7)
    om = orc.TriMesh(m.xy, m.nbr, m.nbr_edge, m.bc, xy6=m.xy6)
    cfg = orc.Config(dim=2, p=p, nu=(nu, nu), flux=flux)
    tm = kbl.TriMesh(p, m.xy, m.nbr, m.nbr_edge, m.bc, xy6=m.xy6, flux=flux, nu=(nu, nu))
    rs, _ = orc.tri_points(p)
    w = inputs.tri_nodal_field(m, rs, _smooth)
    w = np.ascontiguousarray(w * (1 + 0.02 * np.random.default_rng(7).uniform(-1, 1, w.shape)))
    return m, om, cfg, tm, w


@pytest.mark.parametrize("p,curved,nu", [(1, False, 32), (2, False, 33), (1, True, 40), (2, True, 32)])
def test_triangle_bounds_and_step_on_pairs(orc, p, curved, nu):
    m, om, cfg, tm, w = _tri(orc, p, 9, 7, curved, nu=nu)
    E = m.n_elem
    wf = orc.tri_traces(cfg, om, w)
    bnd = zeros_dev(2, 4, E)
    tm.bounds(to_dev(w), to_dev(wf), bnd)
    ref = np.zeros((2, 4, E))
    for e in range(E):
        ref[0, :, e], ref[1, :, e] = orc.bounds_stencil(cfg, orc.tri_gather_stencil(cfg, om, w, wf, e))
    assert bounds_error(bnd.cpu().numpy(), ref).max() < TOL_FP64
    wd, dt, out = to_dev(w), orc.tri_dt(cfg, om, w, 0.2), w
    for _ in range(2):
        tm.step(wd, dt)
        out, _ = orc.tri_ssprk3_step(cfg, om, out, dt)
    tm.check()
    assert (np.abs(wd.cpu().numpy() - out) / _elem_scale(out)).max() < TOL_FP64


@pytest.mark.parametrize("p,curved,flux", [(1, False, 0), (2, False, 2), (1, True, 1), (2, True, 0)])
def test_triangle_residual_of_a_large_mesh(orc, p, curved, flux):
    """5,096 elements: blocks of 16, the last one half full (152 SMs)."""
    m, om, cfg, tm, w = _tri(orc, p, 52, 49, curved, flux=flux, nu=8)
    assert m.n_elem % 16 == 8
    wf = orc.tri_traces(cfg, om, w)
    wd, wfd = to_dev(w), to_dev(wf)
    R, S = zeros_dev(*w.shape), zeros_dev(m.n_elem, tm.nstencil, 4)
    tm.residual(wd, wfd, R)
    tm.gather_stencil(wd, wfd, S)
    tm.check()
    ref = orc.tri_rhs(cfg, om, w, wf)
    err = np.abs(R.cpu().numpy() - ref) / np.maximum(np.abs(ref), _residual_scale(m, w, S.cpu().numpy()))
    assert err.max() < TOL_FP64, err.max()


@pytest.mark.parametrize("p,nu", [(1, 32), (2, 32), (3, 32), (4, 36), (5, 32), (5, 48)])
def test_quad_bounds_on_pairs(orc, p, nu):
    """20 to 84 states."""
    ctx, cfg = both(orc, 2, p, (nu, nu))
    mesh, w = mesh_and_field(orc, 2, p, (5, 4), seed=31 + p, kind="disc", periodic=True)
    om = upload(ctx, orc, mesh)
    wf = orc.traces(cfg, om, w)
    bnd = zeros_dev(2, 4, mesh.n_elem)
    ctx.bounds(to_dev(w), to_dev(wf), bnd)
    ctx.check()
    assert bounds_error(bnd.cpu().numpy(), orc.bounds(cfg, om, w, wf)).max() < TOL_FP64


@pytest.mark.parametrize("p,nu,quad", [(1, 32, 0), (3, 32, 0), (4, 33, 1), (2, 48, 0)])
def test_branched_step_graph_on_pairs_is_bitwise_serial(orc, p, nu, quad):
    from paper_2407_20966_gb300 import kbl
    ctx, _ = both(orc, 2, p, (nu, nu), quadrature=quad)
    mesh, w = mesh_and_field(orc, 2, p, (13, 11), seed=23, kind="disc", periodic=True)
    upload(ctx, orc, mesh)
    out = []
    for ov in (1, 0):
        ctx.set_tuning(kbl.TUNE_RHS_OVERLAP, ov)
        wd = to_dev(w)
        ctx.set_time(0.0)
        for _ in range(3):
            ctx.step(wd, 0.05)
        ctx.check()
        out.append((wd.cpu().numpy(), ctx.time()))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1] > 0.0
