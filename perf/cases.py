"""Performance cases of the kinetic-bounds limiter: the calls that programs make, from the smallest
meshes to the largest, through the public Python binding.

``listed()`` gives the fixed cases, ``draw(rng)`` one more of the same ranges.  ``prepare`` builds a
case's inputs from a seed (mesh, initial state on the device, context), ``run`` makes one pass,
``work`` counts what the method itself needs, and ``exact`` evaluates the same pass in FP64 with
plain torch and numpy, from the equations of the method.

Families:
  step1d  limited SSP-RK3 steps on a line mesh (the 1D experiments)
  step2d  limited SSP-RK3 steps on a quad mesh (the 2D runs)
  batch   one step of many independent quad problems of mixed sizes and orders
  tri     limited SSP-RK3 steps on triangles, affine or curved
  grad    the gradient of the integrated entropy through limited steps (reverse mode)
  nodes   bounds of explicit stencils and the limiter on explicit node sets, as a solver on another
          element family calls them
"""
import math

import numpy as np
import torch

from paper_2407_20966_gb300 import adjoint, inputs, kbl

GAMMA = 1.4


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _case(family, name=None, **kw):
    c = {"family": family, "f64": True, "p": 3, "nu": 32, "steps": 1, "flux": 0, "romberg": False, "k": 4.0,
         "r_fac": 1e-3, "uncoupled": False, "ic": "waves"}
    c.update(kw)
    return {"name": name, **c} if name else c


def listed():
    return [
        # Sod shock tube at the library's default precision: the smallest run, all latency
        _case("step1d", "sod200_p3_f64", n=200, nu=64, ic="tube", steps=10),
        # the paper's own 1D resolution: k = 8 and 2048 velocity points, HLLC, convected pulse
        _case("step1d", "pulse300_p4_nu2048_f64", n=300, p=4, nu=2048, k=8.0, flux=1, ic="pulse", steps=2),
        # a small 2D run in the fast mode (a study on a laptop-sized mesh): launches and latency
        _case("step2d", "vortex16_p3_mixed", nx=16, ny=16, f64=False, ic="vortex", steps=10),
        # the benchmark workload: isentropic vortex, 128^2 P3, fast mode
        _case("step2d", "vortex128_p3_mixed", nx=128, ny=128, f64=False, ic="vortex", steps=4),
        # the same run at full precision (the library's default)
        _case("step2d", "vortex128_p3_f64", nx=128, ny=128, ic="vortex"),
        # a large blast in the fast mode, HLL as for Sedov's problem
        _case("step2d", "blast512_p2_hll_mixed", nx=512, ny=512, p=2, f64=False, flux=2, ic="blast"),
        # a ragged high-order mesh at full precision with Romberg quadrature, HLLC, uncoupled limiting
        _case("step2d", "waves46x27_p4_romberg33_f64", nx=46, ny=27, p=4, nu=33, romberg=True, flux=1,
              uncoupled=True),
        # many independent Riemann problems of uneven size and order (P1-P4) advanced together
        _case("batch", "batch96_mixed", problems=96, n_lo=16, n_hi=64, f64=False, ic="quadrants"),
        # unstructured-looking triangles, fast mode, HLLC
        _case("tri", "tri96_p2_hllc_mixed", n=96, p=2, f64=False, flux=1, ic="blast", curved=False, steps=2),
        # curved triangles at full precision
        _case("tri", "tricurved24_p2_f64", n=24, p=2, flux=1, ic="waves", curved=True),
        # sensitivities: gradient through limited steps of a shock-vortex interaction, checkpointed
        _case("grad", "grad48_p3_f64", n=48, steps=6, every=3, ic="shockvortex"),
        # bounds and limiter on caller-assembled stencils and node sets (another element family)
        _case("nodes", "nodes5000_41_f64", n=5000, states=41, ns=10, nf=15),
    ]


def _envelope_evals(c):
    """(stencil state, velocity node) pairs of one pass, and element-stages."""
    f, p = c["family"], c["p"]
    n1 = p + 1
    if f == "step1d":
        es, st, nodes = 3 * c["steps"] * c["n"], n1 + 4, c["nu"]
    elif f == "step2d":
        es, st, nodes = 3 * c["steps"] * c["nx"] * c["ny"], n1 * n1 + 8 * n1, c["nu"] ** 2
    elif f == "tri":
        es, st, nodes = 3 * c["steps"] * 2 * c["n"] ** 2, n1 * (n1 + 1) // 2 + 6 * n1, c["nu"] ** 2
    elif f == "grad":
        es, st, nodes = 3 * c["steps"] * c["n"] ** 2, n1 * n1 + 8 * n1, c["nu"] ** 2
    elif f == "nodes":
        es, st, nodes = c["n"], c["states"], c["nu"] ** 2
    else:   # batch: mean stencil of P1..P4
        es = 3 * c["problems"] * ((c["n_lo"] + c["n_hi"]) / 2) ** 2
        st, nodes = sum((q + 1) ** 2 + 8 * (q + 1) for q in (1, 2, 3, 4)) / 4, 1024
    return es * st * nodes, es


# A drawn case costs no more than the largest listed one.  Full precision runs on a pipe about 1/40
# of the fast mode's.
def _cost(c):
    ev, es = _envelope_evals(c)
    return (ev + 2000 * es) * (40 if c["f64"] else 1)


_COST_MAX = 40 * (3 * 128 * 128 * (48 * 1024 + 2000))


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        f = rng.choice(["step1d", "step2d", "step2d", "step2d", "batch", "tri", "tri", "grad", "nodes"])
        f64 = rng.random() < 0.5
        kw = {"f64": f64, "r_fac": rng.choice([1e-3, 1e-3, 0.0]), "uncoupled": rng.random() < 0.2,
              "flux": rng.choice([0, 1, 2])}
        if f == "step1d":
            nu, rom = rng.choice([(64, False), (100, False), (129, True), (513, True), (2048, False)])
            kw.update(n=_logint(rng, 50, 2000), p=rng.randint(1, 5), nu=nu, romberg=rom,
                      k=8.0 if nu > 500 else 4.0, ic=rng.choice(["tube", "pulse"]), steps=rng.randint(1, 8))
        elif f == "step2d":
            nu, rom = rng.choice([(32, False)] * 4 + [(16, False), (24, False), (33, True), (17, True), (48, False)])
            kw.update(nx=_logint(rng, 5, 512), ny=_logint(rng, 5, 512), p=rng.choice([1, 2, 3, 3, 4, 5]), nu=nu,
                      romberg=rom, ic=rng.choice(["vortex", "blast", "waves"]), steps=rng.randint(1, 4))
        elif f == "batch":
            n_lo = rng.randint(8, 40)
            kw.update(problems=_logint(rng, 2, 96), n_lo=n_lo, n_hi=n_lo + rng.randint(4, 40), f64=False,
                      ic="quadrants", r_fac=1e-3)
        elif f == "tri":
            nu = rng.choice([32, 32, 16, 20])
            kw.update(n=_logint(rng, 5, 110), p=rng.choice([1, 2, 2]), nu=nu, ic=rng.choice(["blast", "waves"]),
                      curved=rng.random() < 0.3, uncoupled=False, steps=rng.randint(1, 3))
        elif f == "grad":
            kw.update(n=4 * rng.randint(2, 14), p=rng.randint(1, 4), nu=rng.choice([16, 32]), flux=0, f64=True,
                      uncoupled=False, r_fac=1e-3, steps=rng.randint(2, 8), every=rng.randint(1, 4),
                      ic="shockvortex")
        else:
            kw.update(n=_logint(rng, 50, 40000), states=rng.randint(5, 64), ns=rng.randint(3, 16),
                      nf=rng.randint(0, 24), nu=rng.choice([32, 32, 16, 24]), flux=0)
        c = _case(f, **kw)
        if _cost(c) <= _COST_MAX:
            return c


# ---------------------------------------------------------------------------
# inputs (host arrays)
# ---------------------------------------------------------------------------
def _cons(rho, u, v, P):
    return np.stack([rho, rho * u, rho * v, P / (GAMMA - 1) + 0.5 * rho * (u * u + v * v)])


def _field2d(ic, rng, lo, hi, n):
    """A conservative state (x, y) -> (4, ...) of one of the 2D set-ups, with seeded parameters; n is
    the number of elements along the shorter side."""
    L = [hi[0] - lo[0], hi[1] - lo[1]]
    if ic == "vortex":     # isentropic vortex on the periodic box
        xc, yc = [lo[k] + L[k] * rng.uniform(0.4, 0.6) for k in (0, 1)]
        beta, u0, v0, R = rng.uniform(3, 5), rng.uniform(0.5, 1.5), rng.uniform(0.5, 1.5), 0.1 * min(L)

        def f(x, y):
            dx = ((x - xc) / L[0] - np.round((x - xc) / L[0])) * L[0] / R
            dy = ((y - yc) / L[1] - np.round((y - yc) / L[1])) * L[1] / R
            a = beta / (2 * math.pi) * np.exp(0.5 * (1 - dx * dx - dy * dy))
            T = 1 - (GAMMA - 1) / (2 * GAMMA) * a * a
            rho = T ** (1 / (GAMMA - 1))
            return _cons(rho, u0 - a * dy, v0 + a * dx, rho ** GAMMA)
        return f
    if ic == "blast":      # circular blast, a tanh front, uniform ambient at rest in a weak shear
        xc, yc = [lo[k] + L[k] * rng.uniform(0.45, 0.55) for k in (0, 1)]
        r0, wd, p_in = 0.25 * min(L), max(0.008, 1.5 / n) * min(L), rng.uniform(1.0, 10.0)

        def f(x, y):
            s = 0.5 * (1 - np.tanh((np.hypot(x - xc, y - yc) - r0) / wd))
            return _cons(0.125 + 0.875 * s, 0.2 * np.sin(2 * np.pi * (y - lo[1]) / L[1]),
                         -0.2 * np.sin(2 * np.pi * (x - lo[0]) / L[0]), 0.1 + (p_in - 0.1) * s)
        return f
    modes = rng.uniform(0, 2 * math.pi, (4, 3)), rng.integers(1, 4, (4, 3, 2)), rng.uniform(-1, 1, (4, 3))

    def f(x, y):           # a few periodic Fourier modes in every primitive variable
        q = []
        for i, (base, amp) in enumerate(((1.0, 0.12), (0.3, 0.2), (-0.2, 0.2), (1.0, 0.12))):
            g = np.full(np.shape(x), base)
            for m in range(3):
                kx, ky = modes[1][i, m]
                g = g + amp * modes[2][i, m] * np.sin(modes[0][i, m] + 2 * math.pi * (
                    kx * (x - lo[0]) / L[0] + ky * (y - lo[1]) / L[1]))
            q.append(g)
        return _cons(*q)
    return f


def _problem(c, seed):
    """Mesh and initial state of a mesh case (host): (mesh, w0)."""
    rng = np.random.default_rng(seed)
    f = c["family"]
    if f == "tri":
        make = inputs.tri_curved_mesh if c["curved"] else inputs.tri_mesh_2d
        m = make(c["n"], c["n"], 0.0, 1.0, 0.0, 1.0, jitter=0.1 if c["curved"] else 0.2, seed=seed)
        rs, _ = _tri_points(c["p"])
        return m, inputs.tri_nodal_field(m, rs, _field2d(c["ic"], rng, (0.0, 0.0), (1.0, 1.0), c["n"]))
    xi = np.polynomial.legendre.leggauss(c["p"] + 1)[0]
    if f == "step1d":
        if c["ic"] == "tube":
            l = (1.0 * rng.uniform(0.9, 1.1), rng.uniform(-0.1, 0.1), 1.0 * rng.uniform(0.9, 1.1))
            r = (0.125 * rng.uniform(0.9, 1.1), rng.uniform(-0.1, 0.1), 0.1 * rng.uniform(0.9, 1.1))
            mesh, ic = inputs.riemann_1d(c["n"], l, r, 0.0, 1.0, 0.5)
        else:
            mesh = inputs.mesh_1d(c["n"], -0.5, 0.5, periodic=True)
            sg, u0, x0 = rng.uniform(150, 250), rng.uniform(0.8, 1.2), rng.uniform(-0.2, 0.2)

            def ic(x):
                return inputs.conservative(1 + np.exp(-sg * (x - x0) ** 2), [u0 + 0 * x], np.ones_like(x))
        return mesh, inputs.nodal_field(mesh, xi, ic)
    if f == "grad":
        mesh, ic = inputs.shock_vortex(c["n"], centre=(rng.uniform(0.2, 0.3), rng.uniform(0.4, 0.6)))
        w = inputs.nodal_field(mesh, xi, ic)
        return mesh, w * (1 + 1e-2 * rng.uniform(-1, 1, w.shape))
    per = c["ic"] != "blast"
    hi = (10.0 * c["nx"] / max(c["nx"], c["ny"]), 10.0 * c["ny"] / max(c["nx"], c["ny"]))
    mesh = inputs.mesh_2d(c["nx"], c["ny"], 0.0, hi[0], 0.0, hi[1], periodic=(per, per))
    mesh.bc = np.array([[0.125, 0.0, 0.0, 0.25]])
    return mesh, inputs.nodal_field(mesh, xi, _field2d(c["ic"], rng, (0.0, 0.0), hi, min(c["nx"], c["ny"])))


def _batch_problems(c, seed):
    """(p, mesh, ic) of four-quadrant Riemann problems: sizes and orders from the case, states seeded."""
    shape = np.random.default_rng([c["problems"], c["n_lo"], c["n_hi"]])
    rng, out = np.random.default_rng(seed), []
    for _ in range(c["problems"]):
        n, p = 2 * int(shape.integers(c["n_lo"] // 2, c["n_hi"] // 2 + 1)), int(shape.integers(1, 5))
        mesh, ic = inputs.four_quadrant(n, inputs.four_quadrant_states(rng))
        out.append((p, mesh, ic))
    return out


def _max_dt(mesh, w, cfl):
    """cfl * min h / (|U| + c) of a quad state (host)."""
    u = np.abs(w[1:-1] / w[0])
    P = (GAMMA - 1) * (w[-1] - 0.5 * (w[1:-1] ** 2).sum(0) / w[0])
    a = np.sqrt(GAMMA * P / w[0])
    return cfl * float(min((mesh.h[:, k, None] / (u[k] + a)).min() for k in range(len(u))))


def _node_sets(c, seed):
    """Explicit stencils S[E][n][4] and node sets U, F with weights W (host): states scattered about a
    smooth state per element, a tenth of the elements across a jump."""
    rng = np.random.default_rng(seed)
    E, n, ns, nf = c["n"], c["states"], c["ns"], c["nf"]
    amp = np.where(rng.random((E, 1)) < 0.1, 0.4, 0.03)
    base = np.stack([rng.uniform(0.5, 1.5, E), rng.uniform(-1, 1, E), rng.uniform(-1, 1, E), rng.uniform(0.5, 1.5, E)])

    def scatter(m):
        d = rng.uniform(-1, 1, (4, E, m)) * amp
        q = _cons(base[0][:, None] * (1 + d[0]), base[1][:, None] + d[1], base[2][:, None] + d[2],
                  base[3][:, None] * (1 + d[3]))
        return np.ascontiguousarray(np.moveaxis(q, 0, -1))
    return scatter(n), rng.uniform(0.5, 1.5, ns), scatter(ns), scatter(nf)


def _cfl(c):
    return 0.1 if c["family"] == "step1d" else 0.05


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def _options(c):
    return dict(flux=c["flux"], quadrature=int(c["romberg"]), k=c["k"], r_fac=c["r_fac"],
                uncoupled=int(c["uncoupled"]))


def prepare(case, seed):
    c, f = case, case["family"]
    prec = kbl.FP64 if c["f64"] else kbl.FP32_MIXED
    s = {"case": c}
    if f == "nodes":
        s["ctx"] = kbl.Context(dim=2, p=3, nu=(c["nu"], c["nu"]), precision=prec, r_fac=c["r_fac"],
                               uncoupled=int(c["uncoupled"]))
        S, W, U, F = _node_sets(c, seed)
        s["S"], s["U0"], s["F"] = (torch.from_numpy(a).cuda() for a in (S, U, F))
        s["U"] = torch.empty_like(s["U0"])
        s["W"] = W
        s["bnd"] = torch.empty(2, 4, c["n"], dtype=torch.float64, device="cuda")
        s["alpha"] = torch.empty(2, c["n"], dtype=torch.float64, device="cuda")
        return s
    if f == "batch":
        probs = _batch_problems(c, seed)
        s["b"] = b = kbl.Batch([(p, m.nbr, m.h, m.bc) for p, m, _ in probs], flux=c["flux"],
                               uncoupled=int(c["uncoupled"]))
        nodes = {q: np.polynomial.legendre.leggauss(q + 1)[0] for q in (1, 2, 3, 4)}
        w0 = inputs.batch_state(probs, lambda q: nodes[q], b.state_offsets)
    elif f == "tri":
        m, w0 = _problem(c, seed)
        s["t"] = kbl.TriMesh(c["p"], m.xy, m.nbr, m.nbr_edge, m.bc, precision=prec, xy6=m.xy6,
                             nu=(c["nu"], c["nu"]), flux=c["flux"], r_fac=c["r_fac"])
        s["dt"] = 0.05 * 0.25 / (c["n"] * 6.0)
    else:
        mesh, w0 = _problem(c, seed)
        dim = 1 if f == "step1d" else 2
        opt = dict(eps_rule=1) if f == "grad" else _options(c)
        s["ctx"] = ctx = kbl.Context(dim=dim, p=c["p"], nu=(c["nu"],) * dim, precision=prec, **opt)
        ctx.mesh_upload(mesh.nbr, mesh.h, mesh.bc)
        ctx.set_time(0.0)
        if f == "grad":
            s["dts"] = [_max_dt(mesh, w0, 0.05)] * c["steps"]
    s["w0"] = torch.from_numpy(np.ascontiguousarray(w0)).cuda()
    s["w"] = torch.empty_like(s["w0"])
    return s


def run(state):
    s, c = state, state["case"]
    f = c["family"]
    if f == "nodes":
        ctx = s["ctx"]
        ctx.bounds_stencil(s["S"], s["bnd"])
        s["U"].copy_(s["U0"])
        ctx.limit_nodes(s["W"], s["U"], s["F"], s["bnd"], s["alpha"])
        return {"bnd": s["bnd"], "U": s["U"], "alpha": s["alpha"]}
    if f == "grad":
        x = s["w0"].clone().requires_grad_(True)
        w = adjoint.trajectory(x, s["ctx"], s["dts"], checkpoint_every=c["every"])
        J = adjoint.entropy(w, s["ctx"])
        J.backward()
        return {"J": J.detach(), "grad": x.grad}
    w = s["w"]
    w.copy_(s["w0"])            # every pass is the run from the initial condition
    for _ in range(c["steps"]):
        if f == "batch":
            s["b"].step(w, 0.05)
        elif f == "tri":
            s["t"].step(w, s["dt"])
        else:
            s["ctx"].step(w, _cfl(c))
    return w


def work(case):
    """The envelopes (2 products and 4 comparisons per stencil state and velocity node) and, per
    stage, the state and the bounds read and written once."""
    ev, es = _envelope_evals(case)
    n1, f = case["p"] + 1, case["family"]
    if f == "nodes":
        return {"bytes": 8.0 * case["n"] * (4 * (case["states"] + 2 * case["ns"] + case["nf"]) + 10), "flops": 6.0 * ev}
    vals = {"step1d": 3 * n1, "tri": 2 * n1 * (n1 + 1), "batch": 4 * 13.5}.get(f, 4 * n1 * n1)
    return {"bytes": 8.0 * es * 2 * vals * (3 if f == "grad" else 1), "flops": 6.0 * ev * (2 if f == "grad" else 1)}


# ---------------------------------------------------------------------------
# the same pass in FP64 with torch
# ---------------------------------------------------------------------------
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=_dev())


def _lagrange(x, y):
    """l_j(y) and l_j'(y) of the nodes x: two [len(y)][len(x)] arrays."""
    n = len(x)
    l, d = np.ones((len(y), n)), np.zeros((len(y), n))
    for j in range(n):
        for m in range(n):
            if m == j:
                continue
            term = np.ones(len(y))
            for q in range(n):
                if q not in (j, m):
                    term = term * (y - x[q]) / (x[j] - x[q])
            d[:, j] += term / (x[j] - x[m])
            l[:, j] *= (y - x[m]) / (x[j] - x[m])
    return l, d


def _pressure(q):       # q[component first]
    return (GAMMA - 1) * (q[-1] - 0.5 * (q[1:-1] ** 2).sum(0) / q[0])


def _flux(q, d):
    P, u = _pressure(q), q[1 + d] / q[0]
    F = [q[1 + d]] + [q[k] * u + (P if k == 1 + d else 0) for k in range(1, len(q) - 1)] + [(q[-1] + P) * u]
    return torch.stack(F)


def _common_flux(kind, ql, qr, d):
    """Rusanov (0), HLLC (1) or HLL (2), Davis wave speeds, ql on the minus side of axis d."""
    Fl, Fr = _flux(ql, d), _flux(qr, d)
    Pl, Pr = _pressure(ql), _pressure(qr)
    ul, ur = ql[1 + d] / ql[0], qr[1 + d] / qr[0]
    cl, cr = (GAMMA * Pl / ql[0]).sqrt(), (GAMMA * Pr / qr[0]).sqrt()
    if kind == 0:
        return 0.5 * (Fl + Fr) - 0.5 * torch.maximum(ul.abs() + cl, ur.abs() + cr) * (qr - ql)
    Sl, Sr = torch.minimum(ul - cl, ur - cr), torch.maximum(ul + cl, ur + cr)
    if kind == 2:
        mid = (Sr * Fl - Sl * Fr + Sl * Sr * (qr - ql)) / (Sr - Sl)
    else:
        ml, mr = ql[0] * (Sl - ul), qr[0] * (Sr - ur)
        Ss = (Pr - Pl + ml * ul - mr * ur) / (ml - mr)

        def star(q, F, S, u, P):
            g = q[0] * (S - u) / (S - Ss)
            qs = [g] + [g * (Ss if k == 1 + d else q[k] / q[0]) for k in range(1, len(q) - 1)]
            qs.append(g * (q[-1] / q[0] + (Ss - u) * (Ss + P / (q[0] * (S - u)))))
            return F + S * (torch.stack(qs) - q)
        mid = torch.where(Ss >= 0, star(ql, Fl, Sl, ul, Pl), star(qr, Fr, Sr, ur, Pr))
    return torch.where(Sl >= 0, Fl, torch.where(Sr <= 0, Fr, mid))


def _quad_weights(c):
    nu = c["nu"]
    q = np.ones(nu)
    q[0] = q[-1] = 0.5
    if c["romberg"]:
        L = 0
        while (nu - 1) % (2 << L) == 0:
            L += 1
        T = []
        for k in range(L + 1):
            st = 1 << (L - k)
            w = np.zeros(nu)
            w[::st] = st
            w[0] = w[-1] = 0.5 * st
            T.append(w)
        for i in range(1, L + 1):
            T = [T[0]] * i + [T[k] + (T[k] - T[k - 1]) / (4.0 ** i - 1) for k in range(i, L + 1)]
        q = T[L]
    return _t(q)


def _bounds(c, S):
    """(lo, hi)[nv][E] of stencils S[nv][E][n]."""
    d = len(S) - 2
    chunk = max(1, int(3e8 / (S.shape[2] * c["nu"] ** d)))
    parts = [_bounds_chunk(c, S[:, a:a + chunk]) for a in range(0, S.shape[1], chunk)]
    return torch.cat([x[0] for x in parts], 1), torch.cat([x[1] for x in parts], 1)


def _bounds_chunk(c, S):
    d, nu = len(S) - 2, c["nu"]
    rho, P = S[0], _pressure(S)
    th = P / rho
    j = torch.arange(nu, dtype=torch.float64, device=S.device)
    us, ws, gs = [], [], []
    for a in range(d):
        U = S[1 + a] / rho
        lo = (U - c["k"] * th.sqrt()).min(1).values
        h = ((U + c["k"] * th.sqrt()).max(1).values - lo) / (nu - 1)
        u = lo[:, None] + j * h[:, None]
        us.append(u)
        ws.append(_quad_weights(c) * h[:, None])
        gs.append(torch.exp(-(u[:, None, :] - U[:, :, None]) ** 2 / (2 * th[:, :, None])))
    A = rho / (2 * math.pi * th) ** (d / 2)
    T = A[:, :, None] * gs[0]
    if d == 2:
        T = (T[:, :, None, :] * gs[1][:, :, :, None]).flatten(2)      # [E][n][y][x]
    Il = T * ((2 / (GAMMA - 1) - d) * th / 2)[:, :, None]
    Tl, Th = T.min(1).values, T.max(1).values
    Il, Ih = Il.min(1).values, Il.max(1).values
    if d == 2:
        M = (ws[1][:, :, None] * ws[0][:, None, :]).flatten(1)
        u = [us[0][:, None, :].expand(-1, nu, -1).flatten(1), us[1][:, :, None].expand(-1, -1, nu).flatten(1)]
    else:
        M, u = ws[0], us
    rm, rp = 1 - c["r_fac"], 1 + c["r_fac"]
    lo, hi = [rm * (M * Tl).sum(1)], [rp * (M * Th).sum(1)]
    for a in range(d):
        n, p = u[a].clamp(max=0), u[a].clamp(min=0)
        lo.append(rp * (M * Th * n).sum(1) + rm * (M * Tl * p).sum(1))
        hi.append(rm * (M * Tl * n).sum(1) + rp * (M * Th * p).sum(1))
    ke = 0.5 * sum(x * x for x in u)
    lo.append(rm * (M * (Tl * ke + Il)).sum(1))
    hi.append(rp * (M * (Th * ke + Ih)).sum(1))
    lo[0] = lo[0].clamp(min=1e-12)
    return torch.stack(lo), torch.stack(hi)


def _limit(c, U, F, W, lo, hi, eps_rule=0):
    """Limited U[nv][E][ns] (faces F[nv][E][nf], mean weights W), and alpha[2][E]."""
    nv = len(U)
    mean = (W * U).sum(2) / W.sum(-1)
    V = torch.cat([U, F], 2)
    dmx, dmn = V.max(2).values - mean, V.min(2).values - mean
    flat = (dmx.abs() < 1e-13) | (dmn.abs() < 1e-13)
    one = torch.ones_like(dmx)
    a = torch.minimum(((hi - mean) / torch.where(flat, one, dmx)).abs(), ((lo - mean) / torch.where(flat, one, dmn)).abs())
    a = torch.where(flat, one * eps_rule, a.clamp(max=1.0))
    alpha = a.min(0).values
    av = a if c["uncoupled"] else alpha[None].expand(nv, -1)
    Ut, Vt = (mean[..., None] + av[..., None] * (x - mean[..., None]) for x in (U, V))
    pm, pb = _pressure(Vt).min(1).values, _pressure(mean)
    cut = pm < 1e-12
    ok = cut & (pb > 1e-12)
    aP = torch.where(ok, ((1e-12 - pb) / torch.where(ok, pm - pb, torch.ones_like(pm))).abs(), torch.zeros_like(pm))
    aP = torch.where(cut, aP, torch.ones_like(aP))
    U2 = torch.where(cut[None, :, None], mean[..., None] + aP[None, :, None] * (Ut - mean[..., None]), Ut)
    return U2, torch.stack([alpha, aP])


class _Cart:
    """Line or quad mesh of order p: traces, stencils and residual."""

    def __init__(self, c, mesh, p):
        self.c, self.d, self.n = c, mesh.dim, p + 1
        x, w = np.polynomial.legendre.leggauss(p + 1)
        self.D = _t(_lagrange(x, x)[1])
        self.l = _t(_lagrange(x, np.array([-1.0, 1.0]))[0])           # [side][i]
        self.g = _t(np.stack([-_lagrange(x, np.array([-1.0]))[0][0] / w, _lagrange(x, np.array([1.0]))[0][0] / w]))
        self.W = _t(w if mesh.dim == 1 else np.outer(w, w).ravel())
        self.nbr = _t(mesh.nbr.astype(np.int64))
        self.h, self.bc = _t(mesh.h), _t(np.asarray(mesh.bc, np.float64).reshape(len(mesh.bc), -1))

    def traces(self, w):       # [nv][E][face][k]
        if self.d == 1:
            return torch.einsum("vei,si->ves", w, self.l)[..., None]
        q = w.reshape(*w.shape[:2], self.n, self.n)
        return torch.cat([torch.einsum("veji,si->vesj", q, self.l), torch.einsum("veji,sj->vesi", q, self.l)], 2)

    def exterior(self, wf):
        nv = len(wf)
        opp = torch.arange(2 * self.d, device=wf.device) ^ 1
        ext = wf[:, self.nbr.clamp(min=0), opp[None, :]]              # [nv][E][face][k]
        b = (self.nbr < 0)
        bc = self.bc[:, :nv][(-self.nbr - 1).clamp(min=0)].permute(2, 0, 1)[..., None]
        return torch.where(b[None, :, :, None], bc, ext)

    def stencil(self, w, wf):
        return torch.cat([w, wf.flatten(2), self.exterior(wf).flatten(2)], 2)

    def rhs(self, w, wf):
        we, R, n = self.exterior(wf), 0, self.n
        for d in range(self.d):
            F = _flux(w, d)
            if self.d == 1:
                F = F[:, :, None, :]                                  # lines [nv][E][k][i]
            else:
                F = F.reshape(*F.shape[:2], n, n)
                F = F if d == 0 else F.transpose(2, 3)
            dF = F @ self.D.T
            for s in (0, 1):
                f = 2 * d + s
                qi, qe = wf[:, :, f], we[:, :, f]
                Fc = _common_flux(self.c["flux"], *((qe, qi) if s == 0 else (qi, qe)), d)
                dF = dF + (Fc - F @ self.l[s])[..., None] * self.g[s]
            dF = dF if (d == 0 or self.d == 1) else dF.transpose(2, 3)
            R = R - (2 / self.h[:, d])[None, :, None] * dF.flatten(2)
        return R

    def dt(self, w, cfl):
        a = (GAMMA * _pressure(w) / w[0]).sqrt()
        return cfl * min((self.h[:, k, None] / ((w[1 + k] / w[0]).abs() + a)).min() for k in range(self.d))


def _stage(c, m, s, wn, ws, dt, eps_rule):
    wf = m.traces(ws)
    lo, hi = _bounds(c, m.stencil(ws, wf))
    t = ws + dt * m.rhs(ws, wf)
    t = t if s == 0 else (0.75 * wn + 0.25 * t if s == 1 else wn / 3 + 2 / 3 * t)
    return _limit(c, t, m.traces(t).flatten(2), m.W, lo, hi, eps_rule)[0]


def _step(c, m, w, dt, eps_rule=0):
    ws = w
    for s in range(3):
        ws = _stage(c, m, s, w, ws, dt, eps_rule)
    return ws


def _tri_points(p):
    """Points (r, s) and weights of the interior symmetric rules of degree 2 and 4 (closed form)."""
    if p == 1:
        orbits = [(1 / 6, 1 / 6)]
    else:
        r, q = math.sqrt(10.0), math.sqrt(38 - 44 * math.sqrt(0.4))
        wr = math.sqrt(213125 - 53320 * r)
        orbits = [((8 - r - q) / 18, (620 - wr) / 7440), ((8 - r + q) / 18, (620 + wr) / 7440)]
    rs = [pt for a, _ in orbits for pt in ((a, a), (1 - 2 * a, a), (a, 1 - 2 * a))]
    return np.array(rs), np.repeat([w for _, w in orbits], 3)


class _Tri:
    """Triangles, affine or the quadratic map of six points: traces, stencils and the residual in its
    transformed-flux form (on affine elements the strong-form nodal DG residual); w[4][E][ns]."""

    def __init__(self, c, m):
        p = c["p"]
        self.c = c
        rs, w = _tri_points(p)

        def mono(z, deg, dr=0, ds=0):
            return np.stack([(a - b) ** dr * b ** ds * z[:, 0] ** max(a - b - dr, 0) * z[:, 1] ** max(b - ds, 0)
                             for a in range(deg + 1) for b in range(a + 1)], 1)
        C = np.linalg.inv(mono(rs, p))
        xg, wg = np.polynomial.legendre.leggauss(p + 1)
        V = np.array([[0.0, 0.0], [1.0, 0.0], [0.0, 1.0]])
        ev = V[[1, 2, 0]] - V                                         # reference edges
        fr = np.concatenate([V[f] + 0.5 * (1 + xg[:, None]) * ev[f] for f in range(3)])
        phi = mono(fr, p) @ C                                         # [q][j]
        self.phi, self.Dr, self.Ds = (_t(a) for a in (phi, mono(rs, p, 1, 0) @ C, mono(rs, p, 0, 1) @ C))
        X = m.xy if m.xy6 is None else m.xy6                          # map nodes and their degree
        deg = 1 if m.xy6 is None else 2
        ref = np.concatenate([V, 0.5 * (V + V[[1, 2, 0]])])[:X.shape[1]]
        N = np.linalg.inv(mono(ref, deg))

        def jac(z):                                                   # x_r, x_s, y_r, y_s at z
            dr, ds = mono(z, deg, 1, 0) @ N, mono(z, deg, 0, 1) @ N
            return [X[..., 0] @ dr.T, X[..., 0] @ ds.T, X[..., 1] @ dr.T, X[..., 1] @ ds.T]
        xr, xs, yr, ys = jac(rs)
        self.J = [_t(a) for a in (xr, xs, yr, ys)]
        det = xr * ys - xs * yr
        self.det = _t(det)
        self.W = _t(w * det) if m.xy6 is not None else _t(w)
        xr, xs, yr, ys = jac(fr)
        L = np.repeat(np.hypot(ev[:, 0], ev[:, 1]), p + 1)
        ex, ey = (np.repeat(ev[:, k], p + 1) for k in (0, 1))
        tx, ty = xr * ex + xs * ey, yr * ex + ys * ey
        ds = np.hypot(tx, ty)
        self.nx, self.ny, self.sg = _t(ty / ds), _t(-tx / ds), _t(ds / L)
        self.hx, self.hy = _t(ey / L), _t(-ex / L)                    # reference normals
        self.lift = _t((phi * (np.tile(wg, 3) * L)[:, None] / (2 * w)).T)   # [i][q]
        k = np.arange(p + 1)
        self.nb = _t(np.repeat(m.nbr.astype(np.int64), p + 1, axis=1))
        self.nq = _t((m.nbr_edge.astype(np.int64)[:, :, None] * (p + 1) + (p - k)).reshape(len(m.nbr), -1))

    def traces(self, w):
        return torch.einsum("vej,qj->veq", w, self.phi)

    def stencil(self, w, wf):
        return torch.cat([w, wf, wf[:, self.nb, self.nq]], 2)

    def rhs(self, w, wf):
        we, nx, ny = wf[:, self.nb, self.nq], self.nx, self.ny

        def rot(q):
            return torch.stack([q[0], q[1] * nx + q[2] * ny, -q[1] * ny + q[2] * nx, q[3]])
        Fl = _common_flux(self.c["flux"], rot(wf), rot(we), 0)
        Fc = torch.stack([Fl[0], Fl[1] * nx - Fl[2] * ny, Fl[1] * ny + Fl[2] * nx, Fl[3]])
        Fx, Fy = _flux(w, 0), _flux(w, 1)
        xr, xs, yr, ys = self.J
        Fr, Fs = ys * Fx - xs * Fy, xr * Fy - yr * Fx
        jump = self.sg * Fc - (self.traces(Fr) * self.hx + self.traces(Fs) * self.hy)
        return -(torch.einsum("ij,vej->vei", self.Dr, Fr) + torch.einsum("ij,vej->vei", self.Ds, Fs)
                 + torch.einsum("iq,veq->vei", self.lift, jump)) / self.det


def exact(case, seed):
    c, f = case, case["family"]
    if f == "nodes":
        S, W, U, F = (_t(a) for a in _node_sets(c, seed))
        lo, hi = _bounds(c, S.permute(2, 0, 1))
        Ul, al = _limit(c, U.permute(2, 0, 1), F.permute(2, 0, 1), W, lo, hi)
        return {"bnd": torch.stack([lo, hi]), "U": Ul.permute(1, 2, 0).contiguous(), "alpha": al}
    if f == "batch":
        c = {**c, "nu": 32}
        out = []
        for p, mesh, ic in _batch_problems(c, seed):
            m = _Cart(c, mesh, p)
            w = _t(inputs.nodal_field(mesh, np.polynomial.legendre.leggauss(p + 1)[0], ic))
            out.append(_step(c, m, w, m.dt(w, 0.05)).flatten())
        return torch.cat(out)
    if f == "tri":
        mesh, w0 = _problem(c, seed)
        m, w = _Tri(c, mesh), _t(w0).permute(2, 0, 1).contiguous()
        for _ in range(c["steps"]):
            w = _step(c, m, w, 0.05 * 0.25 / (c["n"] * 6.0))
        return w.permute(1, 2, 0).contiguous()
    mesh, w0 = _problem(c, seed)
    m, w = _Cart(c, mesh, c["p"]), _t(w0)
    if f != "grad":
        for _ in range(c["steps"]):
            w = _step(c, m, w, m.dt(w, _cfl(c)))
        return w
    x, dt = w.requires_grad_(True), _max_dt(mesh, w0, 0.05)
    from torch.utils.checkpoint import checkpoint
    for _ in range(c["steps"]):
        wn = ws = (w if w is not x else x)
        for s in range(3):
            ws = checkpoint(_stage, c, m, s, wn, ws, dt, 1, use_reentrant=False)
        w = ws
    Pw = _pressure(w)
    J = ((0.25 * m.h.prod(1))[:, None] * m.W * w[0] * torch.log(Pw * w[0] ** -GAMMA)).sum()
    J.backward()
    return {"J": J.detach(), "grad": x.grad}
