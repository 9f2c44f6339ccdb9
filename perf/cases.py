"""What a user of the solver has it do, as cases that a timing program can run.

A case is a dict of plain values.  ``prepare`` makes what the user's program holds before the
call (inputs on the GPU and the ``Solver`` / ``Batch`` / ``Cnn`` objects it keeps), ``run`` is one
pass through the public entry points, ``work`` the bytes and operations that pass cannot do
without, ``exact`` the same outputs in 64 bits from plain torch.

Four kinds of pass:

* ``step``:  the linear solve of one Newton step, ``update_linearisation(w)`` and
  ``gmres_solve(b)`` to the default 1e-8; b = J x* is applied matrix-free in 64 bits by
  ``_apply_jacobian`` below (quadrature, independent of the library), so x* is the exact answer.
* ``slab``:  one time slab of a march from an impulsive start, ``newton_slab`` with the absolute
  tolerances of the time march.
* ``batch``: several uneven problems solved together by ``Batch.gmres_solve``.
* ``cnn``:   one training step of the warm-start network (gradients and the Adam update).
"""
import math
import types

import numpy as np
import torch

from paper_2210_02690_gb300 import Batch, Cnn, Solver

NU = 1e-3
FORMS = {"f64": dict(vcycle_prec="f64", factor_prec="f64"), "f32": dict(vcycle_prec="f32", factor_prec="f32"),
         "bf16": dict(vcycle_prec="f32", factor_prec="bf16")}
NU1 = NU2 = 2   # V(2,2), the smoothing steps of the repository's workloads
ITERS = 6       # FGMRES iterations to 1e-8 of these problems, for work()
NEWTON = 3      # Newton steps of a slab, for work()


def _step(name, domain, n, levels, k, form, newton=False, order=2, autotune=False):
    c = dict(kind="step", domain=domain, dim=len(n), nx=n[0], ny=n[1], nz=n[2] if len(n) == 3 else 1, levels=levels,
             k=k, form=form, newton=newton, order=order, autotune=autotune)
    return dict(name=name, **c) if name else c


def _slab(name, n, levels, k, form, obstacle=False):
    c = dict(kind="slab", domain="channel", dim=2, nx=n[0], ny=n[1], nz=1, levels=levels, k=k, form=form, newton=True,
             order=2, obstacle=obstacle)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest call: the 8 x 8 model problem, where launches and host latency are all there is
        _step("square8_k0_f64", "square", (8, 8), 3, 0, "f64"),
        # one slab of the 128 x 32 time march (the warm-start workload): many small solves in a row
        _slab("march128_k1_f32", (128, 32), 4, 1, "f32"),
        # one slab of the channel with an obstacle (drag and lift runs), dG(2)
        _slab("obstacle176_k2_f32", (176, 32), 3, 2, "f32", obstacle=True),
        # the benchmark's step: the 704 x 128 channel, Newton Jacobian, mixed precision, autotuned
        _step("channel704_k1_f32", "channel", (704, 128), 4, 1, "f32", newton=True, autotune=True),
        # the same step by a user who asks for 64 bits throughout
        _step("channel704_k1_f64", "channel", (704, 128), 4, 1, "f64", newton=True, autotune=True),
        # higher order in time on the unit square: dG(2) with BF16 factors, dG(3) with FP32 factors
        _step("square256_k2_bf16", "square", (256, 256), 5, 2, "bf16"),
        _step("square256_k3_f32", "square", (256, 256), 5, 3, "f32"),
        # 3D: the largest problem of the benchmark, and dG(2) with its 255 x 255 patches
        _step("cube48_k1_f32", "cube", (48, 48, 48), 4, 1, "f32"),
        _step("cube24_k2_f32", "cube", (24, 24, 24), 3, 2, "f32"),
        # the Q4 / P3disc pair of the paper's 2D experiment
        _step("channel352_q4_k1_f32", "channel", (352, 64), 4, 1, "f32", newton=True, order=4),
        # uneven problems in one graph (a parameter study)
        dict(name="batch16_f32", kind="batch", count=16, form="f32", smallest=32, largest=128),
        # one training step of the warm-start network on the 128 x 32 channel's node grid
        dict(name="cnn257x65_b16", kind="cnn", height=65, width=257, batch=16, hidden=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["step2", "step3", "slab", "batch", "cnn"], [9, 5, 3, 2, 1])[0]
    if kind == "step2":
        levels = rng.randint(2, 5)
        order = 4 if rng.random() < 0.2 else 2
        k = rng.randint(0, 2 if order == 4 else 4)
        form = rng.choice(["f32", "f32", "bf16", "f64"])
        cy = rng.randint(3, 16)
        cx = max(2, int(round(cy * math.exp(rng.uniform(0.0, math.log(5.5))))))
        cap = 25000 if order == 4 else 90000       # cells of the finest level
        cap = cap // (1 + k) if form == "f64" else cap // (1 + k // 2)
        while levels > 2 and cx * cy * 4 ** (levels - 1) > cap:
            levels -= 1
        f = 2 ** (levels - 1)
        return _step(None, rng.choice(["channel", "square"]), (cx * f, cy * f), levels, k, form,
                     newton=rng.random() < 0.5, order=order, autotune=rng.random() < 0.3)
    if kind == "step3":
        k = rng.randint(0, 2)
        form = rng.choice(["f32", "f32", "bf16", "f64" if k < 2 else "f32"])
        levels = rng.randint(2, 4)
        c = [rng.randint(2, 5) for _ in range(3)]
        cap = 2000 if form == "f64" else (32000, 16000, 8000)[k]
        while levels > 2 and c[0] * c[1] * c[2] * 8 ** (levels - 1) > cap:
            levels -= 1
        f = 2 ** (levels - 1)
        return _step(None, rng.choice(["cube", "duct"]), tuple(x * f for x in c), levels, k, form,
                     newton=rng.random() < 0.5, autotune=rng.random() < 0.3)
    if kind == "slab":
        levels = rng.randint(2, 4)
        cy = rng.randint(4, 8)
        cx = rng.randint(3 * cy, 6 * cy)
        f = 2 ** (levels - 1)
        obstacle = rng.random() < 0.5 and cy >= 6
        return _slab(None, (cx * f, cy * f), levels, rng.randint(0, 3), rng.choice(["f32", "f32", "f64"]), obstacle)
    if kind == "batch":
        return dict(kind="batch", count=_log_int(rng, 3, 24), form=rng.choice(["f32", "bf16"]),
                    smallest=rng.choice([16, 32]), largest=rng.choice([64, 128]))
    return dict(kind="cnn", height=_log_int(rng, 17, 129), width=_log_int(rng, 33, 513), batch=_log_int(rng, 1, 16),
                hidden=rng.randint(5, 24))


# ------------------------------------------------------------------ meshes and fields
def _spec(case):
    """The mesh as Solver takes it."""
    d = case["dim"]
    n = (case["nx"], case["ny"], case["nz"])[:d]
    channel = case["domain"] == "channel"
    if channel:   # [0, 2.2] x [0, 0.41] for the 704 x 128 mesh; cells of the same shape on the others
        hi = (0.41 * n[0] / n[1] * (2.2 * 128) / (0.41 * 704), 0.41)
    else:         # cubes of cells, the longest side 1
        hi = tuple(x / max(n) for x in n)
    faces = (1 << (2 * d)) - 1
    if case["domain"] in ("channel", "duct"):
        faces &= ~2   # do-nothing outflow at x = high
    obstacle = ()
    if case.get("obstacle"):   # two coarse cells around a tenth of the length, off the walls
        f = 2 ** (case["levels"] - 1)
        cx, cy = n[0] // f, n[1] // f
        obstacle = (max(1, cx // 10), max(1, cx // 10) + 2, cy // 2 - 1, cy // 2 + 1)
    return types.SimpleNamespace(dim=d, n=n, lo=(0.0,) * d, hi=hi, n_levels=case["levels"], dirichlet=faces,
                                 obstacle=obstacle, order=case["order"])


def _gen(seed, more=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * more + int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, dtype=torch.float64, device="cuda")


def _curl(spec, g, modes=4):
    """Divergence-free field at the velocity nodes (x fastest): the curl of random sine series."""
    d = spec.dim
    S, C = [], []
    for e in range(d):
        u = torch.linspace(0.0, 1.0, spec.order * spec.n[e] + 1, dtype=torch.float64, device="cuda")
        m = torch.arange(1, modes + 1, dtype=torch.float64, device="cuda")[:, None] * math.pi
        S.append(torch.sin(m * u))
        C.append(m / spec.hi[e] * torch.cos(m * u))

    def grad(a, e):   # derivative along e of sum a prod sin, on the grid with x fastest
        t = [C[i] if i == e else S[i] for i in range(d)]
        if d == 2:
            return torch.einsum("ab,ax,by->yx", a, *t).reshape(-1)
        return torch.einsum("abc,ax,by,cz->zyx", a, *t).reshape(-1)

    if d == 2:
        a = _randn(g, modes, modes)
        w = torch.stack([grad(a, 1), -grad(a, 0)], 1)
    else:
        a, b, c = (_randn(g, modes, modes, modes) for _ in range(3))
        w = torch.stack([grad(c, 1) - grad(b, 2), grad(a, 2) - grad(c, 0), grad(b, 0) - grad(a, 1)], 1)
    return w / w.norm(dim=1).max()


def _poiseuille(spec, u_max=1.5):
    y = torch.linspace(0.0, 1.0, spec.order * spec.n[1] + 1, dtype=torch.float64, device="cuda")
    v = torch.zeros(spec.order * spec.n[1] + 1, spec.order * spec.n[0] + 1, 2, dtype=torch.float64, device="cuda")
    v[:, :, 0] = (4.0 * u_max * y * (1.0 - y))[:, None]
    return v.reshape(-1, 2)


def _w(spec, case, seed):
    """Linearisation velocity (k+1, R): a smooth field that varies a little over the Radau nodes."""
    g = _gen(seed, 1)
    base = _curl(spec, g)
    if case["domain"] == "channel":
        base = _poiseuille(spec) + 0.3 * base
    change = 0.05 * _curl(spec, g)
    c = _time_basis(case["k"])[0]
    return torch.stack([(base + c[a] * change).reshape(-1) for a in range(case["k"] + 1)])


def _pressure_dofs(spec):
    return spec.dim + 1 if spec.order == 2 else 10


def _sizes(spec):
    """Values per Radau node: velocity R, pressure S."""
    nodes = math.prod(spec.order * n + 1 for n in spec.n)
    return spec.dim * nodes, _pressure_dofs(spec) * math.prod(spec.n)


def _enclosed(spec):
    return spec.dirichlet == (1 << (2 * spec.dim)) - 1


def _solution(spec, case, seed):
    """x* ~ N(0, 1), the mean pressure of an enclosed flow removed."""
    R, S = _sizes(spec)
    x = _randn(_gen(seed, 2), case["k"] + 1, R + S)
    if _enclosed(spec):
        p = x[:, R:].view(case["k"] + 1, -1, _pressure_dofs(spec))
        p[:, :, 0] -= p[:, :, 0].mean(dim=1, keepdim=True)
    return x


# ------------------------------------------------------------------ J x in 64 bits
def _time_basis(k):
    """Right Radau nodes on (0, 1], weights, T_ab = int chi_b' chi_a + chi_a(0) chi_b(0)."""
    leg = np.polynomial.legendre
    c = np.zeros(k + 2)
    c[k], c[k + 1] = 1.0, -1.0
    x = np.sort(leg.legroots(c).real)
    for _ in range(3):
        dx = leg.legval(x, c) / leg.legval(x, leg.legder(c))
        x = x - dx
    x[-1] = 1.0
    t = 0.5 * (x + 1.0)
    q, qw = leg.leggauss(k + 1)
    q, qw = 0.5 * (q + 1.0), 0.5 * qw

    def lag(a, s):
        return np.prod([(s - t[b]) / (t[a] - t[b]) for b in range(k + 1) if b != a] + [np.ones_like(s)], axis=0)

    def dlag(a, s):
        out = np.zeros_like(s)
        for m in range(k + 1):
            if m != a:
                out = out + np.prod([(s - t[b]) / (t[a] - t[b]) for b in range(k + 1) if b not in (a, m)]
                                    + [np.ones_like(s) / (t[a] - t[m])], axis=0)
        return out

    zero = np.zeros(1)
    T = [[float(np.sum(qw * dlag(b, q) * lag(a, q)) + lag(a, zero)[0] * lag(b, zero)[0]) for b in range(k + 1)]
         for a in range(k + 1)]
    return t, [float(np.sum(qw * lag(a, q))) for a in range(k + 1)], T


def _lagrange(order, s):
    """Values and derivatives of the 1D Lagrange basis on [-1, 1] at the points s: (points, order + 1)."""
    nd = np.linspace(-1.0, 1.0, order + 1)
    L, D = np.ones((len(s), order + 1)), np.zeros((len(s), order + 1))
    for i in range(order + 1):
        for m in range(order + 1):
            if m != i:
                L[:, i] *= (s - nd[m]) / (nd[i] - nd[m])
                t = np.ones(len(s)) / (nd[i] - nd[m])
                for l in range(order + 1):
                    if l not in (i, m):
                        t *= (s - nd[l]) / (nd[i] - nd[l])
                D[:, i] += t
    return L, D


def _tables(spec, points):
    """Basis values (Q, L), physical gradients (Q, L, d) and pressure functions (Q, P) at tensor points
    (one array of reference coordinates per direction, x fastest)."""
    d, r = spec.dim, spec.order
    h = [spec.hi[e] / spec.n[e] for e in range(d)]
    LD = [_lagrange(r, np.asarray(p)) for p in points]

    def kron(ms):   # x fastest
        out = ms[0]
        for m in ms[1:]:
            out = np.kron(m, out)
        return out

    phi = kron([LD[e][0] for e in range(d)])
    dphi = np.stack([kron([LD[f][1] * 2.0 / h[f] if f == e else LD[f][0] for f in range(d)]) for e in range(d)], -1)
    xs = [kron([np.asarray(points[f])[:, None] if f == e else np.ones((len(points[f]), 1)) for f in range(d)])[:, 0]
          for e in range(d)]
    if r == 2:
        pres = np.stack([np.ones_like(xs[0])] + xs, -1)
    else:
        powers = [(0, 0), (1, 0), (0, 1), (2, 0), (1, 1), (0, 2), (3, 0), (2, 1), (1, 2), (0, 3)]
        pres = np.stack([xs[0] ** a * xs[1] ** b for a, b in powers], -1)
    return [torch.from_numpy(np.ascontiguousarray(m)).cuda() for m in (phi, dphi, pres)]


def _apply_jacobian(spec, case, w, x, tau, gamma=35.0):
    """J x of the dG(k) slab problem at w: time coupling, convection (and Newton's term), viscosity,
    Nitsche's terms on the Dirichlet faces and the velocity-pressure coupling, cell by cell."""
    d, r, k = spec.dim, spec.order, case["k"]
    R, _ = _sizes(spec)
    _, tw, T = _time_basis(k)
    h = [spec.hi[e] / spec.n[e] for e in range(d)]
    g, gw = np.polynomial.legendre.leggauss(r + 1)
    nn = [r * n + 1 for n in spec.n]
    ax = [torch.arange(n, device="cuda") for n in spec.n]
    cells = torch.meshgrid(*reversed(ax), indexing="ij")[::-1]          # x fastest
    cells = [c.reshape(-1) for c in cells]
    stride = [math.prod(nn[:e]) for e in range(d)]
    loc = torch.meshgrid(*([torch.arange(r + 1, device="cuda")] * d), indexing="ij")[::-1]
    off = sum(l.reshape(-1) * s for l, s in zip(loc, stride))
    idx = sum(r * c * s for c, s in zip(cells, stride))[:, None] + off[None, :]

    def rule(face=None):
        pts, wts = [], []
        for e in range(d):
            if face is not None and e == face // 2:
                pts.append(np.array([1.0 if face & 1 else -1.0]))
                wts.append(np.ones(1))
            else:
                pts.append(g)
                wts.append(gw * h[e] / 2.0)
        out = wts[0]
        for v in wts[1:]:
            out = np.kron(v, out)
        return _tables(spec, pts), torch.from_numpy(np.ascontiguousarray(out)).cuda()

    vol = rule()
    faces = [(f, rule(f)) for f in range(2 * d) if spec.dirichlet >> f & 1]
    y = torch.zeros_like(x)
    v = x[:, :R].reshape(k + 1, -1, d)
    for a in range(k + 1):
        s = tau * tw[a]
        p = x[a, R:].reshape(len(cells[0]), -1)
        ve = v[a][idx]
        te = sum(T[a][b] * v[b] for b in range(k + 1))[idx]
        we = w[a].reshape(-1, d)[idx]
        (phi, dphi, pres), wq = vol
        vq, dv = torch.einsum("ql,clm->cqm", phi, ve), torch.einsum("qle,clm->cqme", dphi, ve)
        wv = torch.einsum("ql,clm->cqm", phi, we)
        val = torch.einsum("cqme,cqe->cqm", dv, wv)
        if case["newton"]:
            val = val + torch.einsum("cqme,cqe->cqm", torch.einsum("qle,clm->cqme", dphi, we), vq)
        val = s * val + torch.einsum("ql,clm->cqm", phi, te)
        der = s * NU * dv
        pq = s * torch.einsum("qj,cj->cq", pres, p)
        for e in range(d):
            der[:, :, e, e] -= pq
        out = torch.einsum("q,ql,cqm->clm", wq, phi, val) + torch.einsum("q,qle,cqme->clm", wq, dphi, der)
        yp = s * torch.einsum("q,qj,cq->cj", wq, pres, torch.einsum("cqee->cq", dv))
        for f, ((phi, dphi, pres), wq) in faces:
            e, n = f // 2, 1.0 if f & 1 else -1.0
            on = torch.nonzero(cells[e] == (spec.n[e] - 1 if f & 1 else 0))[:, 0]
            vq = torch.einsum("ql,clm->cqm", phi, ve[on])
            dn = n * torch.einsum("ql,clm->cqm", dphi[:, :, e].contiguous(), ve[on])
            t = -NU * dn + gamma * NU / h[e] * vq
            t[:, :, e] += gamma / h[e] * vq[:, :, e] + n * torch.einsum("qj,cj->cq", pres, p[on])
            add = torch.einsum("q,ql,cqm->clm", wq, phi, t)
            add -= NU * n * torch.einsum("q,ql,cqm->clm", wq, dphi[:, :, e].contiguous(), vq)
            out.index_add_(0, on, s * add)
            yp.index_add_(0, on, -s * n * torch.einsum("q,qj,cq->cj", wq, pres, vq[:, :, e]))
        ya = torch.zeros(R // d, d, dtype=torch.float64, device="cuda")
        ya.index_put_((idx.reshape(-1),), out.reshape(-1, d), accumulate=True)
        y[a, :R] = ya.reshape(-1)
        y[a, R:] = yp.reshape(-1)
    return y


# ------------------------------------------------------------------ the cases
def _tau(case):
    return 0.005 if case["domain"] == "channel" else 0.01


def _split(spec, k, x):
    """Velocity (k+1, R) and pressure (k+1, S) of a whole solution vector.  The pressure of an enclosed
    flow is free up to a constant per Radau node, so its user takes the mean out."""
    R, _ = _sizes(spec)
    x = x.view(k + 1, -1)
    if _enclosed(spec):
        p = x[:, R:].unflatten(1, (-1, _pressure_dofs(spec)))[:, :, 0]
        p -= p.mean(dim=1, keepdim=True)
    return {"velocity": x[:, :R], "pressure": x[:, R:]}


def _batch_cases(case, seed):
    """The problems of a batch: n_x, n_y powers of two between the smallest and the largest, k 1 or 2."""
    g = np.random.default_rng(12345 + case["count"])    # the mesh sizes belong to the case, not to the seed
    sizes = [s for s in (16, 32, 64, 128) if case["smallest"] <= s <= case["largest"]]
    out = []
    for _ in range(case["count"]):
        nx, ny = (int(v) for v in g.choice(sizes, 2))
        levels = int(math.log2(min(nx, ny) // 4)) + 1
        out.append(_step(None, "square", (nx, ny), levels, int(g.choice([1, 2])), case["form"]))
    return out


def _cnn_inputs(case, seed):
    g = _gen(seed, 3)
    ch = [4, case["hidden"], case["hidden"], 4]
    shape = (case["batch"], 4, case["height"], case["width"])
    x, t = _randn(g, *shape).float(), (0.1 * _randn(g, *shape)).float()
    params = []
    for cin, cout in zip(ch[:-1], ch[1:]):
        params += [_randn(g, cout * cin * 9) / math.sqrt(9.0 * cin), 0.05 * _randn(g, cout)]
    return ch, x, t, torch.cat(params).float()


def _solver(spec, case, w, **more):
    return Solver(spec, case["k"], NU, _tau(case), w, linearisation="newton" if case["newton"] else "oseen", nu1=NU1,
                  nu2=NU2, **FORMS[case["form"]], **more)


def prepare(case, seed):
    if case["kind"] == "cnn":
        ch, x, t, params = _cnn_inputs(case, seed)
        net = Cnn(ch, case["height"], case["width"], case["batch"])
        net.set_params(params.cpu().numpy())
        return dict(case=case, net=net, x=x, t=t)
    if case["kind"] == "batch":
        specs, solvers, rhs = [], [], []
        for i, c in enumerate(_batch_cases(case, seed)):
            spec = _spec(c)
            w = _w(spec, c, 64 * seed + i)
            specs.append((spec, c["k"]))
            rhs.append(_apply_jacobian(spec, c, w, _solution(spec, c, 64 * seed + i), _tau(c)).reshape(-1))
            solvers.append(_solver(spec, c, w.reshape(-1)))
        return dict(case=case, specs=specs, solvers=solvers, batch=Batch(solvers), rhs=rhs)
    spec = _spec(case)
    if case["kind"] == "slab":
        # the first slab of a march: Poiseuille flow plus a perturbation at t = 0, inflow data g
        R, S = _sizes(spec)
        k = case["k"]
        v0 = _poiseuille(spec) + 0.5 * _curl(spec, _gen(seed, 4))
        data = _poiseuille(spec)
        if spec.obstacle:   # no slip on the removed box
            nx, ny = (2 * n + 1 for n in spec.n)
            f = 2 ** (case["levels"] - 1)
            x0, x1, y0, y1 = (2 * f * o for o in spec.obstacle)
            for v in (v0, data):
                v.view(ny, nx, 2)[y0:y1 + 1, x0:x1 + 1] = 0.0
        X0 = torch.zeros(k + 1, R + S, dtype=torch.float64, device="cuda")
        X0[:, :R] = v0.reshape(-1)
        solver = _solver(spec, case, v0.reshape(-1).repeat(k + 1), gmres_rtol=0.0, gmres_atol=1e-9)
        return dict(case=case, spec=spec, solver=solver, X0=X0.reshape(-1), v0=v0.reshape(-1),
                    g=data.reshape(-1).repeat(k + 1))
    w = _w(spec, case, seed)
    b = _apply_jacobian(spec, case, w, _solution(spec, case, seed), _tau(case)).reshape(-1)
    solver = _solver(spec, case, w.reshape(-1))
    if case["autotune"]:
        solver.autotune()
    return dict(case=case, spec=spec, solver=solver, w=w.reshape(-1), b=b)


def run(state):
    kind = state["case"]["kind"]
    if kind == "cnn":
        loss, grad = state["net"].gradients(state["x"], state["t"])
        state["net"].adam_step(grad, 2e-3)
        return {"loss": loss, "grad": grad}
    if kind == "batch":
        xs, its, _, _ = state["batch"].gmres_solve(state["rhs"])
        return [dict(_split(spec, k, x), iterations=n) for (spec, k), x, n in zip(state["specs"], xs, its)]
    if kind == "slab":
        X, steps, its, _, _ = state["solver"].newton_slab(state["X0"], v_prev=state["v0"], g=state["g"], rtol=0.0,
                                                          atol=1e-8)
        return dict(_split(state["spec"], state["case"]["k"], X), steps=steps, iterations=its)
    state["solver"].update_linearisation(state["w"])
    x, its, _, _ = state["solver"].gmres_solve(state["b"])
    return dict(_split(state["spec"], state["case"]["k"], x), iterations=its)


def exact(case, seed):
    if case["kind"] == "cnn":
        ch, x, t, params = _cnn_inputs(case, seed)
        p = params.double().requires_grad_()
        y, at = x.double(), 0
        for i, (cin, cout) in enumerate(zip(ch[:-1], ch[1:])):
            weight = p[at:at + cout * cin * 9].view(cout, cin, 3, 3)
            bias = p[at + cout * cin * 9:at + cout * cin * 9 + cout]
            at += cout * cin * 9 + cout
            cols = torch.nn.functional.unfold(y, 3, padding=1)
            y = torch.einsum("ok,bkp->bop", weight.view(cout, -1), cols) + bias[None, :, None]
            y = y.view(x.shape[0], cout, x.shape[2], x.shape[3])
            if i < len(ch) - 2:
                y = torch.tanh(y)
        loss = (y - t.double()).square().mean()
        loss.backward()
        return {"loss": float(loss), "grad": p.grad}

    def solution(c, s):
        spec = _spec(c)
        return dict(_split(spec, c["k"], _solution(spec, c, s).reshape(-1)), iterations=None)

    if case["kind"] == "batch":
        return [solution(c, 64 * seed + i) for i, c in enumerate(_batch_cases(case, seed))]
    if case["kind"] == "step":
        return solution(case, seed)
    return None   # a nonlinear slab: no closed form


def _solve_work(case, solves, iters):
    """Set-up and solve: every level's local inverses formed and written once per set-up, read once a
    sweep (they are larger than any cache at the sizes that count); the vectors of the call once."""
    d, r, k = case["dim"], case["order"], case["k"]
    n = (k + 1) * ((r + 1) ** d * d + (d + 1 if r == 2 else 10))
    size = {"f64": 8, "f32": 4, "bf16": 2}[case["form"]]
    cells = [math.prod((case["nx"], case["ny"], case["nz"])[:d]) // 2 ** (d * l) for l in range(case["levels"] - 1)]
    spec = _spec(case)
    R, S = _sizes(spec)
    sweeps = iters * (NU1 + NU2)
    return {"bytes": solves * (sum(cells) * n * n * size * (1 + sweeps) + 8 * (k + 1) * (2 * (R + S) + R)),
            "flops": solves * sum(cells) * (2 * n ** 3 + sweeps * 2 * n * n)}


def work(case):
    if case["kind"] == "cnn":
        h = case["hidden"]
        pixels = case["batch"] * case["height"] * case["width"]
        weights = 9 * (4 * h + h * h + 4 * h)
        # forward, weight gradient and data gradient (not of the first layer): 2 flops a weight and pixel
        return {"bytes": 4 * (8 * pixels + 5 * weights), "flops": 2 * pixels * (3 * weights - 9 * 4 * h)}
    if case["kind"] == "batch":
        parts = [_solve_work(c, 1, ITERS) for c in _batch_cases(case, 0)]
        # the solve alone: the local inverses are read, not formed
        for c, p in zip(_batch_cases(case, 0), parts):
            n = (c["k"] + 1) * 21
            p["flops"] -= 2 * n ** 3 * sum(c["nx"] * c["ny"] // 4 ** l for l in range(c["levels"] - 1))
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    if case["kind"] == "slab":
        return _solve_work(case, NEWTON, ITERS)
    return _solve_work(case, 1, ITERS)
