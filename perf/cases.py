"""Performance cases of the library: whole calls through its Python binding.

One pass of a case is what a user's program does between two looks at its
fields: load the canonical moments from device memory (or start from host
memory), advance a number of time steps, and read the canonical moments back;
or one loss gradient through ``autograd.evolve``.  Sizes and parameters are
those of this repository's benchmark, tests and experiments.

``listed`` gives the fixed cases, ``draw`` one more of the same ranges,
``prepare`` the inputs and handles a program keeps, ``run`` one pass, ``work``
the bytes and operations of one pass, ``exact`` the same result in 64 bits from
plain torch.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2301_01622_gb300 import autograd, llb

STORAGE = {"f32": llb.LLB_F32, "f64": llb.LLB_F64, "f16": llb.LLB_F16S, "bf16": llb.LLB_BF16S}
ELEM = {"f32": 4, "f64": 8, "f16": 2, "bf16": 2}
# floating operations of one node and step: collision, Q populations and their sums
# (two components: also the gradient, the forcing and the colour populations)
FLOPS = {("one", 19): 230, ("one", 27): 320, ("two", 19): 480, ("two", 27): 660}


def listed():
    return [
        # the benchmark's flow: long runs of a large turbulent box, rarely read back
        dict(name="flow 256^3 q19", kind="flow", nx=256, ny=256, nz=256, q=19, dtype="f32", tau=0.6, steps=50, graph=False),
        # the smallest box of the tests, a long run of short steps replayed from a graph: launches and latency
        dict(name="flow 32^3 q19 graph", kind="flow", nx=32, ny=32, nz=32, q=19, dtype="f32", tau=0.8, steps=200, graph=True),
        # an odd box of middling size on the larger lattice
        dict(name="flow 131x97x75 q27", kind="flow", nx=131, ny=97, nz=75, q=27, dtype="f32", tau=0.6, steps=50, graph=False),
        # half the memory: 16-bit states, for the boxes that would not fit otherwise
        dict(name="flow 192^3 q19 f16", kind="flow", nx=192, ny=192, nz=192, q=19, dtype="f16", tau=0.6, steps=50, graph=False),
        # validation and viscosity runs in double precision
        dict(name="flow 96x80x65 q19 f64", kind="flow", nx=96, ny=80, nz=65, q=19, dtype="f64", tau=0.8, steps=20, graph=False),
        # the largest two-component run: an off-axis droplet pair with the near-contact force
        dict(name="drops 384x192x192 q27", kind="drops", nx=384, ny=192, nz=192, q=27, dtype="f32", tau=1.0, steps=30,
             A_h=0.01, looks=0),
        # the paper's box, its diagnostics followed during the run
        dict(name="drops 128^3 q19 diag", kind="drops", nx=128, ny=128, nz=128, q=19, dtype="f32", tau=1.0, steps=50,
             A_h=0.05, looks=2),
        # an ensemble of droplet collisions of different sizes advanced together
        dict(name="ensemble 16 boxes q27", kind="ensemble", boxes=16, small=48, large=96, q=27, dtype="f32", tau=1.0, steps=20,
             A_h=0.01),
        # gradient of a loss through the one-component evolution (initial field and relaxation time)
        dict(name="grad 128x96x64 q19", kind="grad", nx=128, ny=96, nz=64, q=19, dtype="f32", tau=0.6, steps=40),
        # the same through the two-component evolution: the benchmark's gradient box
        dict(name="grad drops 96^3 q27", kind="grad2", nx=96, ny=96, nz=96, q=27, dtype="f32", tau=1.0, steps=40),
        # the scheme with stored colour populations the moment-only one is compared with (local-error experiment)
        dict(name="populations 128^3 q19", kind="pop2", nx=128, ny=128, nz=128, q=19, dtype="f32", tau=1.0, steps=30,
             A_h=0.05),
        # end to end from pinned host memory to pinned host memory
        dict(name="host 192x160x144 q19", kind="host", nx=192, ny=160, nz=144, q=19, dtype="f32", tau=0.6, steps=2),
    ]


def _size(rng, lo, hi, most):
    """Three log-uniform extents, odd ones among them, of at most `most` nodes together."""
    while True:
        n = [int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) for _ in range(3)]
        if n[0] * n[1] * n[2] <= most:
            return dict(nx=n[0], ny=n[1], nz=n[2])


def draw(rng):
    kind = rng.choice(["flow", "flow", "flow", "flow", "drops", "drops", "drops", "ensemble", "grad", "grad2", "pop2", "host"])
    q = rng.choice([19, 27])
    if kind == "flow":
        dtype = rng.choice(["f32", "f32", "f32", "f16", "bf16", "f64"])
        s = _size(rng, 24, 300, 2 ** 20 if dtype == "f64" else 2 ** 24)
        n = s["nx"] * s["ny"] * s["nz"]
        return dict(kind=kind, **s, q=q, dtype=dtype, tau=rng.choice([0.6, 0.7, 0.8]), graph=n < 2 ** 18,
                    steps=200 if n < 2 ** 18 and dtype != "f64" else rng.choice([10, 25, 40]))
    if kind == "drops":
        return dict(kind=kind, **_size(rng, 48, 384, 2 ** 23), q=q, dtype="f32", tau=rng.choice([0.8, 1.0, 1.2]),
                    steps=rng.choice([10, 20, 30]), A_h=rng.choice([0.0, 0.01, 0.05]), looks=rng.choice([0, 0, 1, 2]))
    if kind == "ensemble":
        return dict(kind=kind, boxes=rng.randrange(4, 25), small=rng.choice([40, 48, 56]), large=rng.choice([72, 88, 96]), q=q,
                    dtype="f32", tau=1.0, steps=rng.choice([10, 20]), A_h=rng.choice([0.0, 0.01]))
    if kind in ("grad", "grad2"):
        return dict(kind=kind, **_size(rng, 40, 128, 2 ** 20), q=q, dtype="f32", tau=0.7 if kind == "grad" else 1.0,
                    steps=rng.choice([20, 30, 40]))
    if kind == "pop2":
        return dict(kind=kind, **_size(rng, 48, 160, 2 ** 21), q=q, dtype="f32", tau=1.0, steps=rng.choice([10, 20, 30]),
                    A_h=rng.choice([0.0, 0.05]))
    return dict(kind=kind, **_size(rng, 96, 256, 2 ** 22), q=q, dtype="f32", tau=0.6, steps=rng.choice([1, 2, 4]))


# ----------------------------------------------------------------------------- inputs


def _grid(nx, ny, nz):
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") for n in (nz, ny, nx)]
    z, y, x = torch.meshgrid(*ax, indexing="ij")
    return x, y, z


def _flow(nx, ny, nz, seed):
    """Canonical moments of a 3D Taylor-Green vortex at equilibrium, u0 about 0.05, a phase and
    U(-1e-3, 1e-3) velocity noise from the seed."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    ph = torch.rand(4, generator=g, device="cuda", dtype=torch.float64)
    x, y, z = _grid(nx, ny, nz)
    ax, ay, az = (2 * math.pi * (c / n + p) for c, n, p in ((x, nx, ph[0]), (y, ny, ph[1]), (z, nz, ph[2])))
    u0 = 0.045 + 0.01 * ph[3]
    u = torch.stack([u0 * torch.sin(ax) * torch.cos(ay) * torch.cos(az), -u0 * torch.cos(ax) * torch.sin(ay) * torch.cos(az),
                     torch.zeros_like(x)])
    u += 1e-3 * (2 * torch.rand(u.shape, generator=g, device="cuda", dtype=torch.float64) - 1)
    return _equilibrium(torch.ones_like(x)[None], u)


def _drops(nx, ny, nz, seed):
    """Two droplets of fluid 1 moving towards each other along x off axis in a matrix of fluid 2, tanh
    interfaces of width 2; places, radii and speeds vary with the seed."""
    r = np.random.default_rng(seed)
    R = min(0.156 * min(ny, nz), 0.11 * nx)
    off = min(2 * R, nx / 4)
    x, y, z = _grid(nx, ny, nz)
    phi = torch.full_like(x, -1.0)
    u = torch.zeros((3,) + x.shape, dtype=torch.float64, device="cuda")
    for sgn in (-1.0, 1.0):
        c = [nx / 2 + sgn * off, ny / 2 + sgn * R / 4, nz / 2] + r.uniform(-1, 1, 3)
        rad, speed = R * r.uniform(0.9, 1.1), -sgn * 0.05 * r.uniform(0.8, 1.2)
        d = [(a - b + n / 2) % n - n / 2 for a, b, n in ((x, c[0], nx), (y, c[1], ny), (z, c[2], nz))]
        p = torch.tanh(rad - torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2))
        phi = torch.maximum(phi, p)
        u[0] += speed * (1 + p) / 2
    return _equilibrium(torch.stack([(1 + phi) / 2, (1 - phi) / 2]), u)


def _equilibrium(rhos, u):
    rho = rhos.sum(0)
    P = [rho * u[a] * u[b] + (rho / 3 if a == b else 0) for a, b in PAIRS]
    return torch.cat([rhos, rho * u, torch.stack(P)])


def _boxes(case, seed):
    r = np.random.default_rng(1000 + case["boxes"])  # the sizes are the case's, the fields the seed's
    dims = [tuple(int(v) for v in r.integers(case["small"], case["large"] + 1, 3)) for _ in range(case["boxes"])]
    return dims, [_drops(*d, 97 * seed + i) for i, d in enumerate(dims)]


def _field(case, seed):
    f = _flow if case["kind"] in ("flow", "grad", "host") else _drops
    return f(case["nx"], case["ny"], case["nz"], seed)


def _float(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


# ----------------------------------------------------------------------------- the calls


class _Handle:
    """A context or batch handle, released with the program's last reference to it."""

    def __init__(self, h, destroy):
        self.h, self.destroy = h, destroy

    def __del__(self):
        self.destroy(self.h)


def _params(case):
    p = dict(storage=STORAGE[case["dtype"]], stream=torch.cuda.current_stream().cuda_stream)
    if case["kind"] in ("drops", "ensemble", "pop2"):
        p.update(ncomp=2, A_h=case["A_h"])
    if case["kind"] == "pop2":
        p.update(scheme=llb.LLB_SCHEME_POPULATION_BGK)
    return llb.llb_params_default(**p)


def prepare(case, seed):
    s = dict(case=case)
    if case["kind"] == "ensemble":
        dims, fields = _boxes(case, seed)
        s["m0"] = [f.to(_float(case)) for f in fields]
        s["out"] = [torch.empty_like(m) for m in s["m0"]]
        s["h"] = _Handle(llb.llb_batch_create(dims, case["q"], case["tau"], _params(case)), llb.llb_batch_destroy)
        s["ctx"] = [llb.llb_batch_domain(s["h"].h, i) for i in range(len(dims))]
        return s
    m0 = _field(case, seed).to(_float(case)).contiguous()
    if case["kind"] in ("grad", "grad2"):
        s["m0"] = m0.requires_grad_()
        s["tau"] = torch.tensor(case["tau"], dtype=torch.float32, device="cuda", requires_grad=True)
        return s
    if case["kind"] == "host":
        s["m0"] = m0.cpu().pin_memory()
        s["out"] = torch.empty_like(s["m0"], pin_memory=True)
    else:
        s["m0"], s["out"] = m0, torch.empty_like(m0)
    s["h"] = _Handle(llb.llb_create(case["nx"], case["ny"], case["nz"], case["q"], case["tau"], _params(case)),
                     llb.llb_destroy)
    return s


TWO = dict(beta=0.7, A_s=0.01, grad_eps=0.02)
DIAG = ("rho1_sum", "n_in", "rho1_avg", "min_rho")


def _look(ctx):
    d = llb.llb_diagnostics(ctx)
    return d["mass"] + d["momentum"] + [d[k] for k in DIAG]


def run(state):
    case = state["case"]
    kind, steps = case["kind"], case["steps"]
    if kind in ("grad", "grad2"):
        m0, tau = state["m0"], state["tau"]
        m0.grad = tau.grad = None
        out = autograd.evolve(m0, tau, steps, lattice=case["q"], two_component=TWO if kind == "grad2" else None)
        j = 2 if kind == "grad2" else 1
        (0.5 * out[j:j + 3].square().sum()).backward()  # kinetic energy at the end
        return out.detach(), m0.grad, tau.grad
    if kind == "ensemble":
        for c, m in zip(state["ctx"], state["m0"]):
            llb.llb_init_moments_device(c, m)
        llb.llb_batch_step_graph(state["h"].h, steps)
        for c, o in zip(state["ctx"], state["out"]):
            llb.llb_get_moments_device(c, o)
        return state["out"]
    ctx = state["h"].h
    if kind == "host":
        llb.llb_step_host(ctx, state["m0"], state["out"], steps)
        return state["out"]
    llb.llb_init_moments_device(ctx, state["m0"])
    looks = []
    if case.get("looks"):
        for _ in range(case["looks"]):
            llb.llb_step(ctx, steps // case["looks"])
            looks.append(_look(ctx))
    elif case.get("graph"):
        llb.llb_step_graph(ctx, steps)
    else:
        llb.llb_step(ctx, steps)
    llb.llb_get_moments_device(ctx, state["out"])
    return (state["out"], torch.tensor(looks)) if looks else state["out"]


def work(case):
    two = case["kind"] not in ("flow", "grad", "host")
    nf, es = (11 if two else 10), ELEM[case["dtype"]]
    if case["kind"] == "ensemble":
        r = np.random.default_rng(1000 + case["boxes"])
        n = sum(int(np.prod(r.integers(case["small"], case["large"] + 1, 3))) for _ in range(case["boxes"]))
    else:
        n = case["nx"] * case["ny"] * case["nz"]
    steps = case["steps"] // case["looks"] * case["looks"] if case.get("looks") else case["steps"]
    flops = FLOPS["two" if two else "one", case["q"]] * n * steps
    ends = 2 * n * nf * (es + (8 if case["dtype"] == "f64" else 4))  # canonical moments in and out, to and from the state
    step = 2 * n * nf * es  # a step reads and writes the state once
    if case["kind"] in ("grad", "grad2"):
        # a forward step, and an adjoint step that reads the state and a cotangent and writes one
        return {"bytes": ends + ends // 2 + steps * (step + 3 * n * nf * es), "flops": 3 * flops}
    if case["kind"] == "pop2":
        return {"bytes": ends + steps * 2 * n * 2 * case["q"] * es, "flops": flops}
    return {"bytes": ends + steps * step + case.get("looks", 0) * n * nf * es, "flops": flops}


# ----------------------------------------------------------------------------- 64-bit results from plain torch

PAIRS = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))


def _lattice(q):
    w = {19: (1 / 3, 1 / 18, 1 / 36), 27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[q]
    every = [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]
    return [(c, w[sum(v * v for v in c)]) for c in every if sum(v * v for v in c) < len(w)]


def _pull(f, c):
    """f(x - c), periodic."""
    s = [(v, d) for v, d in ((c[2], 0), (c[1], 1), (c[0], 2)) if v]
    return torch.roll(f, [v for v, _ in s], [d for _, d in s]) if s else f


def _dot(c, v):
    t = None
    for a in range(3):
        if c[a]:
            t = c[a] * v[a] if t is None else t + c[a] * v[a]
    return 0.0 if t is None else t


def _population(c, w, rho, j, A, tr):
    """w [rho + 3 c.j + 4.5 c c : A - 1.5 tr A]"""
    t = rho - 1.5 * tr
    for k, (a, b) in enumerate(PAIRS):
        if c[a] * c[b]:
            t = t + (4.5 if a == b else 9.0) * c[a] * c[b] * A[k]
    return w * (t + 3 * _dot(c, j))


def _sum_up(new, h, c):
    new[0] = new[0] + h
    for a in range(3):
        if c[a]:
            new[1 + a] = new[1 + a] + c[a] * h
    for k, (a, b) in enumerate(PAIRS):
        if c[a] * c[b]:
            new[4 + k] = new[4 + k] + c[a] * c[b] * h


def _step_one(m, q, tau):
    rho, j = m[0], m[1:4]
    om = 1 / tau
    A = [(1 - om) * (m[4 + k] - (rho / 3 if a == b else 0)) + om * j[a] * j[b] / rho for k, (a, b) in enumerate(PAIRS)]
    tr = A[0] + A[1] + A[2]
    new = [torch.zeros_like(rho)] * 10
    for c, w in _lattice(q):
        _sum_up(new, _pull(_population(c, w, rho, j, A, tr), c), c)
    return torch.stack(new)


def _collide_two(r1, rho, j, P, q, tau, prm):
    """Post-collision j, A and the colour quantities of the two-component step."""
    lat = _lattice(q)
    phi = 2 * r1 / rho - 1
    G = [torch.zeros_like(rho) for _ in range(3)]
    for c, w in lat:
        if any(c):
            v = 3 * w * _pull(phi, (-c[0], -c[1], -c[2]))
            for a in range(3):
                if c[a]:
                    G[a] = G[a] + c[a] * v
    eps = prm.get("grad_eps", 0.0)
    g2 = G[0] * G[0] + G[1] * G[1] + G[2] * G[2]
    if eps:
        gn = torch.sqrt(g2 + eps * eps)
        n, on = [g / gn for g in G], 1.0
    else:
        gn = torch.sqrt(g2)
        on = (gn >= 1e-6).to(rho.dtype)
        n = [on * g / torch.where(gn > 0, gn, 1.0) for g in G]
    F = [0.0, 0.0, 0.0]
    if prm.get("A_h"):
        nz, ny, nx = rho.shape
        z, y, x = torch.nonzero(gn >= 0.05, as_tuple=True)
        hit = torch.zeros(z.shape, dtype=torch.bool, device=z.device)
        for k in (1, 2, 3):
            o = [torch.round(-k * n[a][z, y, x]).long() for a in range(3)]
            hit |= phi[(z + o[2]) % nz, (y + o[1]) % ny, (x + o[0]) % nx] > phi[z, y, x] + 0.01
        near = torch.zeros_like(rho)
        near[z, y, x] = hit.to(rho.dtype)
        F = [prm["A_h"] * near * g for g in G]
    om = 1 / tau
    u = [(j[a] + 0.5 * F[a]) / rho for a in range(3)]
    A = [(1 - om) * (P[k] - (rho / 3 if a == b else 0)) + om * rho * u[a] * u[b]
         + (1 - 0.5 * om) * (u[a] * F[b] + F[a] * u[b]) + 0.01 / 9 * on * gn * n[a] * n[b] for k, (a, b) in enumerate(PAIRS)]
    return [j[a] + F[a] for a in range(3)], A, n, r1 / rho, 0.7 * r1 * (rho - r1) / rho


def _colour(c, w, h, n, r, e):
    if not any(c):
        return r * h
    return r * h + e * w / math.sqrt(sum(v * v for v in c)) * _dot(c, n)


def _step_two(m, q, tau, prm):
    rho = m[0] + m[1]
    j, A, n, r, e = _collide_two(m[0], rho, m[2:5], m[5:11], q, tau, prm)
    tr = A[0] + A[1] + A[2]
    new, r1 = [torch.zeros_like(rho)] * 10, torch.zeros_like(rho)
    for c, w in _lattice(q):
        h = _population(c, w, rho, j, A, tr)
        r1 = r1 + _pull(_colour(c, w, h, n, r, e), c)
        _sum_up(new, _pull(h, c), c)
    return torch.stack([r1, new[0] - r1] + new[1:])


def _populations_two(m, q, tau, prm, steps):
    """Colour-gradient lattice Boltzmann with both population sets stored, from moments to moments."""
    lat = _lattice(q)
    om = 1 / tau

    def shifted(rho, P):
        A = [P[k] - (rho / 3 if a == b else 0) for k, (a, b) in enumerate(PAIRS)]
        return A, A[0] + A[1] + A[2]

    rho = m[0] + m[1]
    A, tr = shifted(rho, m[5:11])
    f = [_population(c, w, rho, m[2:5], A, tr) for c, w in lat]
    f1 = [m[0] / rho * v for v in f]

    def project():
        new = [torch.zeros_like(rho)] * 10
        for (c, _), v in zip(lat, f):
            _sum_up(new, v, c)
        return sum(f1[1:], f1[0]), new

    for _ in range(steps):
        r1, t = project()
        j, A, n, r, e = _collide_two(r1, t[0], t[1:4], t[4:10], q, tau, prm)
        tr = A[0] + A[1] + A[2]
        A0, tr0 = shifted(t[0], t[4:10])
        for i, (c, w) in enumerate(lat):
            h = _population(c, w, t[0], j, A, tr) + (1 - om) * (f[i] - _population(c, w, t[0], t[1:4], A0, tr0))
            f[i], f1[i] = _pull(h, c), _pull(_colour(c, w, h, n, r, e), c)
    r1, t = project()
    return torch.stack([r1, t[0] - r1] + t[1:])


def exact(case, seed):
    kind, q, tau, steps = case["kind"], case["q"], case["tau"], case["steps"]
    if kind == "ensemble":
        got = []
        for m in _boxes(case, seed)[1]:
            m = m.to(_float(case)).double()
            for _ in range(steps):
                m = _step_two(m, q, tau, case)
            got.append(m)
        return got
    m = _field(case, seed).to(_float(case)).double()
    if kind == "pop2":
        return _populations_two(m, q, tau, case, steps)
    if kind in ("grad", "grad2"):
        t = torch.tensor(case["tau"], dtype=torch.float32, device="cuda").double().requires_grad_()
        m.requires_grad_()
        step = (lambda s, w: _step_one(s, q, w)) if kind == "grad" else (lambda s, w: _step_two(s, q, w, TWO))
        out = m
        for _ in range(steps):
            out = checkpoint(step, out, t, use_reentrant=False)
        j = 1 if kind == "grad" else 2
        (0.5 * out[j:j + 3].square().sum()).backward()
        return out.detach(), m.grad, t.grad
    looks = []
    every = steps // case["looks"] if case.get("looks") else steps
    for _ in range(case.get("looks") or 1):
        for _ in range(every):
            m = _step_one(m, q, tau) if kind in ("flow", "host") else _step_two(m, q, tau, case)
        if case.get("looks"):
            rho, drop = m[0] + m[1], m[0][m[0] > 0.5]
            looks.append([float(v) for v in (m[0].sum(), m[1].sum(), *m[2:5].sum((1, 2, 3)), drop.sum(), drop.numel(),
                                             drop.mean() if drop.numel() else 0.0, rho.min())])
    m = m.cpu() if kind == "host" else m
    return (m, torch.tensor(looks, dtype=torch.float64)) if looks else m
