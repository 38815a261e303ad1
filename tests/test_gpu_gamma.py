"""Ratios of specific heats above (d + 2) / d, where the internal weight delta / 2 of Eq. 44 is negative:
its envelopes against the checker, and the bounds' vector-Jacobian product against differences."""
import numpy as np
import pytest

from paper_2407_20966_gb300 import inputs
from tests.gpu_helpers import TOL_FP32, TOL_FP64, bounds_error, mesh_and_field, to_dev, zeros_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_20966_gb300 import build
    build.build()


def _case(orc, dim, p, nu, gamma, precision, seed=5):
    from paper_2407_20966_gb300 import kbl
    mesh, _ = mesh_and_field(orc, dim, p, (5, 4) if dim == 2 else 11, seed=seed, periodic=True)
    rng = np.random.default_rng(seed)
    E, ns = mesh.n_elem, (p + 1) ** dim
    w = inputs.random_states(rng, E * ns, dim, gamma=gamma).T.reshape(dim + 2, E, ns).copy()
    ctx = kbl.Context(dim=dim, p=p, nu=(nu,) * dim, precision=precision, gamma=gamma)
    ctx.mesh_upload(mesh.nbr, mesh.h, mesh.bc)
    # face values: states of their own, physical whatever the polynomial does at the ends
    wf = inputs.random_states(rng, E * ctx.nfp, dim, gamma=gamma).T.reshape(dim + 2, E, ctx.nfp).copy()
    return ctx, mesh, w, wf


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("dim,p,nu,gamma", [(2, 3, 16, 2.5), (2, 2, 32, 2.2), (2, 1, 48, 3.0), (1, 3, 64, 3.5), (1, 4, 300, 4.0)])
def test_bounds_with_negative_internal_weight(orc, dim, p, nu, gamma, precision):
    ctx, mesh, w, wf = _case(orc, dim, p, nu, gamma, precision)
    bnd = zeros_dev(2, dim + 2, mesh.n_elem)
    ctx.bounds(to_dev(w), to_dev(wf), bnd)
    ctx.check()
    cfg = orc.Config(dim=dim, p=p, nu=(nu,) * dim, gamma=gamma)
    ref = orc.bounds(cfg, orc.Mesh(mesh.nbr, mesh.h, mesh.bc), w, wf)
    assert bounds_error(bnd.cpu().numpy(), ref).max() < (TOL_FP32 if precision else TOL_FP64)


@pytest.mark.parametrize("p,nu,gamma", [(2, 16, 2.5), (3, 32, 3.0)])
def test_bounds_vjp_with_negative_internal_weight(orc, p, nu, gamma):
    ctx, mesh, w, wf = _case(orc, 2, p, nu, gamma, 0)
    rng = np.random.default_rng(1)
    E, nfp = mesh.n_elem, ctx.nfp
    bnd = zeros_dev(2, 4, E)
    ctx.bounds(to_dev(w), to_dev(wf), bnd)
    bb = np.zeros((2, 4, E))
    bb[:, 3] = rng.standard_normal((2, E))   # the energy bounds carry the internal envelopes
    wb, wfb, wfbx = zeros_dev(*w.shape), zeros_dev(4, E, nfp), zeros_dev(4, E, nfp)
    ctx.bounds_vjp(to_dev(w), to_dev(wf), bnd, to_dev(bb), wb, wfb, wfbx)
    ctx.check()
    vw, vf = rng.standard_normal(w.shape), rng.standard_normal(wf.shape)
    h = 1e-7

    def B(s):
        out = zeros_dev(2, 4, E)
        ctx.bounds(to_dev(w + s * h * vw), to_dev(wf + s * h * vf), out)
        return out.cpu().numpy()
    fd = float((bb * (B(1) - B(-1))).sum()) / (2 * h)
    terms = [wb.cpu().numpy() * vw, (wfb.cpu().numpy() + wfbx.cpu().numpy()) * vf]
    ad, mag = sum(float(t.sum()) for t in terms), sum(float(np.abs(t).sum()) for t in terms)
    assert abs(fd - ad) <= 1e-6 * mag, (fd, ad, mag)
