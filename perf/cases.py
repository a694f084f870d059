"""The work this library is timed on: solver runs, their start, and the surrogate's training.

A case is a plain dict; ``listed()`` gives the fixed ones, ``draw(rng)`` one more of the same
ranges, ``prepare(case, seed)`` what a program holds before the call (mesh or batch handle,
states on the GPU), ``run(state)`` one pass through the public entry points, ``work(case)`` the
bytes and operations a pass cannot do without, and ``exact(case, seed)`` the same results in
64 bits, computed here with torch alone.

Start states are built here in 64 bits (fields with fronts of one to a few cells over
smooth variation, as a run holds them once shocks have formed) and rounded to FP32.  A pass of a
solver run starts from the stored state each time, as a run resumed from a snapshot does.
"""
import math
import random

import numpy as np
import torch

from paper_2601_16911_gb300 import cvweno as cv
from paper_2601_16911_gb300 import inputs as I

DEV = "cuda"
SYSTEMS = {"burgers": I.BURGERS, "linadv": I.LINADV, "kpp": I.KPP, "euler": I.EULER}


def listed():
    return [
        # the 1D workload: a short run of the step/sine datum, one tile, latency throughout
        dict(name="burgers1d-128-p2", do="advance", system="burgers", dim=1, nx=128, ny=1, p=2, steps=10),
        # a small 2D mesh, the least work a 2D step has: launches and latency
        dict(name="dg-burgers-64-q1", do="advance", system="burgers", nx=64, ny=64, p=1, steps=2),
        # the KPP workload, DG Q3: one step of the benchmark's mesh
        dict(name="dg-kpp-256-q3", do="advance", system="kpp", nx=256, ny=256, p=3, steps=1),
        # the KPP workload, CG Q3
        dict(name="cg-kpp-256-q3", do="advance", kind="cg", system="kpp", nx=256, ny=256, p=3, steps=1),
        # the start of a run: projection of the initial datum (a large mesh of the batch workload)
        dict(name="project-fourier-512-q3", do="project", system="burgers", ic="fourier", nx=512, ny=512, p=3),
        # method of lines with the caller's own integrator: the residual alone, the highest
        # degree, a ragged mesh with open sides
        dict(name="residual-linadv-330x170-q4", do="residual", system="linadv", nx=330, ny=170, p=4, open=True),
        # the Euler workload: one step on the benchmark's mesh, open sides
        dict(name="euler-512-q3", do="advance", system="euler", nx=512, ny=512, p=3, steps=1, open=True),
        # a production Euler run: positivity limiter, CFL-controlled step, conservation totals
        dict(name="euler-cfl-190x125-q2", do="cfl", system="euler", nx=190, ny=125, p=2, open=True),
        # the HWENO-limited scheme (limiter after every stage), a ragged mesh
        dict(name="limiter-burgers-301x150-q2", do="advance", system="burgers", nx=301, ny=150, p=2, steps=1, limiter=True),
        # the batched workload: 64 independent problems of uneven size and degree
        dict(name="batch-burgers-64", do="batch", count=64, nmin=64, nmax=512),
        # the surrogate workload: the network in place of the sensor on KPP 1024^2 Q2
        dict(name="surrogate-kpp-1024-q2", do="surrogate", system="kpp", nx=1024, ny=1024, p=2, steps=1),
        # training the surrogate: a few of an epoch's minibatches, of the benchmark's size
        dict(name="train-16384-b4096", do="train", samples=16384, batch=4096),
    ]


def draw(rng: random.Random):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    do = rng.choice(["burgers1d", "dg", "dg", "dg", "cg", "cg", "euler", "euler", "cfl", "residual", "limiter", "batch",
                     "surrogate", "train", "project"])
    scalar = rng.choice(["burgers", "kpp", "linadv"])
    # degrees as the workloads run them: KPP and the continuous space up to 3, the others up to 4
    p = rng.randint(1, 3 if do == "cg" or do == "limiter" or (scalar == "kpp" and do not in ("euler", "cfl")) else 4)
    top = {1: 900, 2: 700, 3: 512, 4: 400}[p]
    most = 4 if p < 3 else 2 if p == 3 else 1  # steps of a 2D pass
    nx = log_int(24, top)
    ny = max(8, int(nx * rng.uniform(0.4, 1.2)))
    if do == "burgers1d":
        kind = rng.choice(["dg", "dg", "cg"])
        return dict(do="advance", system=rng.choice(["burgers", "linadv"]), dim=1, nx=log_int(20, 4000), ny=1,
                    p=min(p, 3) if kind == "cg" else p, steps=rng.randint(1, 20 if kind == "dg" else 4), kind=kind)
    if do == "dg":
        return dict(do="advance", system=scalar, nx=nx, ny=ny, p=p, steps=rng.randint(1, most), open=rng.random() < 0.3)
    if do == "cg":
        return dict(do="advance", kind="cg", system=scalar, nx=nx, ny=ny, p=p, steps=rng.randint(1, 2))
    if do == "euler":
        return dict(do="advance", system="euler", nx=nx, ny=ny, p=p, steps=rng.randint(1, min(2, most)), open=rng.random() < 0.7)
    if do == "cfl":
        return dict(do="cfl", system="euler", nx=nx, ny=ny, p=p, open=rng.random() < 0.7)
    if do == "residual":
        return dict(do="residual", system=rng.choice([scalar, "euler"]), nx=nx, ny=ny, p=p, open=rng.random() < 0.5)
    if do == "limiter":
        return dict(do="advance", system=scalar, nx=nx, ny=ny, p=p, steps=rng.randint(1, min(2, most)), limiter=True)
    if do == "batch":
        return dict(do="batch", count=rng.randint(4, 48), nmin=rng.randint(24, 96), nmax=rng.randint(128, 400))
    if do == "surrogate":
        return dict(do="surrogate", system="kpp", nx=log_int(100, 1024), ny=log_int(100, 900), p=2, steps=rng.randint(1, 2))
    if do == "train":
        batch = rng.choice([1024, 4096, 4096, 16384])
        return dict(do="train", samples=batch * rng.randint(2, 3) + rng.randint(1, batch), batch=batch)
    system, ic = rng.choice([("burgers", "fourier"), ("kpp", "circle"), ("euler", "quadrants")])
    return dict(do="project", system=system, ic=ic, nx=nx, ny=ny, p=p)


# ---- descriptions, start states, the calls -----------------------------------------------


def desc(case):
    system = case["system"]
    dim = case.get("dim", 2)
    nx, ny = case["nx"], case["ny"]
    # square cells, the workloads' boxes: [-2,2]^2 for KPP, the unit length otherwise
    if system == "kpp":
        box = (-2.0, 2.0, -2.0, -2.0 + 4.0 * ny / nx)
    else:
        box = (0.0, 1.0, 0.0, ny / nx if dim == 2 else 1.0)
    extra = dict(lambda_const=1.0) if system == "kpp" else {}
    if system == "linadv":
        extra.update(adv_vx=1.0, adv_vy=0.5 if dim == 2 else 0.0)
    return I.mesh(dim, nx, ny, degree=case["p"], system=SYSTEMS[system], domain=box,
                  bc=I.TRANSMISSIVE if case.get("open") else I.PERIODIC, kind=I.CG if case.get("kind") == "cg" else I.DG,
                  hweno_limiter=1 if case.get("limiter") else 0, positivity=1 if case["do"] == "cfl" else 0, **extra)


def cfl(d):
    """CFL number 0.3 / (2p + 1), a quarter of it at p = 4, where the explicit viscous term sets the limit."""
    return (0.3 if d["degree"] < 4 else 0.075) / (2 * d["degree"] + 1)


def time_step(d):
    """dt = cfl dx / (dim max|f'|) for speeds up to about 3 (1 for KPP)."""
    dx = (d["x1"] - d["x0"]) / d["nx"]
    lam = 1.0 if d["system"] == I.KPP else 3.5 if d["system"] == I.EULER else 3.0
    return cfl(d) * dx / (d["dim"] * lam)


def datum(case, seed):
    """(ic_type, params) of a projected start, drawn as the workloads draw it."""
    if case["ic"] == "fourier":
        return I.IC_FOURIER, I.fourier_modes(I.SplitMix64(seed))
    if case["ic"] == "circle":
        return I.IC_CIRCLE, [0.0, 0.0, I.SplitMix64(seed).uniform(0.5, 1.0), 3.5 * math.pi, 0.25 * math.pi]
    return I.euler_quadrants(seed, n=8, degree=1)[1]


def field(d, seed, x, y):
    """The start state as functions of position (64 bits): [variables, *x.shape]."""
    g = I.SplitMix64(seed)
    dx = (d["x1"] - d["x0"]) / d["nx"]
    lx, ly = d["x1"] - d["x0"], (d["y1"] - d["y0"]) if d["dim"] == 2 else 1.0
    if d["system"] == I.KPP:
        R, wob, ph = g.uniform(0.5, 1.0), g.uniform(0.05, 0.15), g.uniform(0.0, 6.0)
        cy = 0.5 * (d["y0"] + d["y1"])
        r, th = torch.sqrt(x * x + (y - cy) ** 2), torch.atan2(y - cy, x)
        R = min(R, 0.4 * ly)
        front = 0.5 * (1.0 + torch.tanh((R * (1.0 + wob * torch.sin(3.0 * th + ph)) - r) / (3.0 * dx)))
        return (math.pi * (0.25 + 3.25 * front))[None]
    if d["system"] == I.EULER:
        prim = [(g.uniform(0.1, 1.5), g.uniform(-1.0, 1.0), g.uniform(-1.0, 1.0), g.uniform(0.1, 1.5)) for _ in range(4)]
        sx = 0.5 * (1.0 + torch.tanh((x - d["x0"] - g.uniform(0.4, 0.6) * lx) / (0.8 * dx)))
        sy = 0.5 * (1.0 + torch.tanh((y - d["y0"] - g.uniform(0.4, 0.6) * ly) / (0.8 * dx)))
        wave = 1.0 + 0.05 * torch.sin(2 * math.pi * ((x - d["x0"]) / lx + 2 * (y - d["y0"]) / ly) + g.uniform(0.0, 6.0))
        rho, vx, vy, pr = ((1 - sx) * (1 - sy) * a + sx * (1 - sy) * b + (1 - sx) * sy * c + sx * sy * e
                           for a, b, c, e in zip(*prim))
        rho, pr = rho * wave, pr * wave
        return torch.stack([rho, rho * vx, rho * vy, pr / 0.4 + 0.5 * rho * (vx * vx + vy * vy)])
    u = torch.zeros_like(x)
    for _ in range(4):
        a, kx, ky = g.uniform(0.0, 0.5), g.randint(0, 3), g.randint(1, 3)
        u = u + a * torch.sin(2 * math.pi * (kx * (x - d["x0"]) / lx + (ky * (y - d["y0"]) / ly if d["dim"] == 2 else 0.0)) +
                              g.uniform(0.0, 6.0))
    s = torch.sin(2 * math.pi * ((x - d["x0"]) / lx + (y - d["y0"]) / ly if d["dim"] == 2 else (x - d["x0"]) / lx) +
                  g.uniform(0.0, 6.0))
    width = 3.0 if d["kind"] == I.CG else 1.0
    return (u + 0.5 * torch.tanh(s / (2 * math.pi) * lx / (width * dx)))[None]


def start_state(d, seed):
    """FP32 start state in the library's layout."""
    dim, n, nx, ny = d["dim"], d["degree"] + 1, d["nx"], d["ny"]
    f64 = dict(dtype=torch.float64, device=DEV)
    dx, dy = (d["x1"] - d["x0"]) / nx, (d["y1"] - d["y0"]) / ny
    if d["kind"] == I.CG:
        xg = torch.tensor(gll(d["degree"])[:-1], **f64)
        x = (d["x0"] + dx * (torch.arange(nx, **f64)[:, None] + 0.5 + 0.5 * xg)).reshape(-1)
        y = (d["y0"] + dy * (torch.arange(ny, **f64)[:, None] + 0.5 + 0.5 * xg)).reshape(-1) if dim == 2 else x.new_zeros(1)
        Y, X = torch.meshgrid(y, x, indexing="ij")
        return field(d, seed, X, Y).reshape(1, -1).float()
    q, w = (torch.tensor(v, **f64) for v in np.polynomial.legendre.leggauss(6))
    L = torch.tensor(np.polynomial.legendre.legvander(q.cpu().numpy(), n - 1), **f64) * w[:, None]
    L = L * (torch.arange(n, **f64) + 0.5)
    x = d["x0"] + dx * (torch.arange(nx, **f64)[:, None] + 0.5 + 0.5 * q)
    if dim == 1:
        u = field(d, seed, x, torch.zeros_like(x))
        return torch.einsum("viq,qm->vim", u, L).float().contiguous()
    out = []
    for j0 in range(0, ny, 64):  # row bands, so that the sampled field stays small
        y = d["y0"] + dy * (torch.arange(j0, min(ny, j0 + 64), **f64)[:, None] + 0.5 + 0.5 * q)
        Y, X = torch.broadcast_tensors(y[:, None, :, None], x[None, :, None, :])
        out.append(torch.einsum("vjiab,am,bk->vjimk", field(d, seed, X, Y), L, L))
    u = torch.cat(out, 1)
    return u.reshape(u.shape[0], nx * ny, n * n).float().contiguous()


def network(seed):
    """Parameters of a network as the library holds it: weights of the usual initial size, output biases
    as training leaves them (smooth cells dominate: gamma near 1, confident in most)."""
    w = I.mlp_init(seed)
    w[-2], w[-1] = 3.0, 2.0
    return w


def batch_descs(case, seed):
    """The instances: the sizes and degrees are the case's (the same for every seed), the data the seed's."""
    g = I.SplitMix64(1000 * case["count"] + case["nmax"])
    sizes = [(g.randint(case["nmin"], case["nmax"]), g.randint(1, 4)) for _ in range(case["count"])]
    return [I.mesh(2, n, n, degree=p, system=I.BURGERS) for n, p in sizes]


def samples(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    X = torch.randn(case["samples"], 12, generator=g, device=DEV).mul_(1.5).clamp_(-8.0, 8.0)
    # the target falls with the spread of the inputs, as the sensor does
    y = torch.exp(-0.15 * X.square().sum(1).sqrt() * (0.6 + 0.4 * torch.tanh(X[:, 0])))
    return X, y


def prepare(case, seed):
    do = case["do"]
    if do == "train":
        X, y = samples(case, seed)
        return dict(case=case, X=X, y=y, net=cv.Mlp(network(seed)))
    if do == "batch":
        ds = batch_descs(case, seed)
        b = cv.Batch(ds)
        u0 = torch.cat([start_state(d, seed + 31 * k).reshape(-1) for k, d in enumerate(ds)])
        # the launch shape the benchmark's tuning keeps on this workload; a program keeps its tuned plan
        b.set_plan(schedule=cv.BATCH_GROUPED, tile=0, dynamic=1, ctas_per_sm=0)
        return dict(case=case, batch=b, u0=u0, u=u0.clone(), dt=[time_step(d) for d in ds])
    d = desc(case)
    mesh = cv.Mesh(d)
    st = dict(case=case, mesh=mesh, dt=time_step(d), cfl=cfl(d))
    if do == "project":
        return dict(st, ic=datum(case, seed))
    st["u0"] = start_state(d, seed).reshape(mesh.state_shape)
    st["u"] = st["u0"].clone()
    if do == "surrogate":
        st["net"] = cv.Mlp(network(seed))
        mesh.set_surrogate(st["net"], 0.5)
    return st


def run(st):
    case = st["case"]
    do = case["do"]
    if do == "train":
        loss = st["net"].train(st["X"], st["y"], batch=case["batch"], epochs=1, lr=1e-3)
        return dict(loss=loss, params=torch.tensor(st["net"].params()))
    if do == "batch":
        st["u"].copy_(st["u0"])
        st["batch"].advance(st["u"], st["dt"], 1)
        return st["u"]
    mesh = st["mesh"]
    if do == "project":
        return mesh.project(*st["ic"])
    if do == "residual":
        return mesh.residual(st["u0"])
    if do == "cfl":
        u, _ = mesh.positivity(st["u0"], out=st["u"])
        dt = mesh.step(u, cfl=st["cfl"])
        return dict(u=u, dt=dt, totals=torch.tensor(mesh.mass_total(u)))
    st["u"].copy_(st["u0"])
    mesh.advance(st["u"], st["dt"], case["steps"])
    return st["u"]


def work(case):
    """Bytes: the state read and written once per step (inputs and outputs of the other calls); operations: the
    method's sum-factorised count per cell and stage, as the benchmark states it, without troubled cells."""
    do = case["do"]
    if do == "train":
        s = case["samples"]
        return dict(bytes=52.0 * s, flops=6.0 * 4992 * s)

    def stage_flops(d):
        n = d["degree"] + 1
        cells = d["nx"] * d["ny"]
        if d["dim"] == 1:
            return 2.0 * cells * (14 * n * n + 20 * n)
        per = (8 * n ** 3 + 4 * n ** 2) + 4 * n * n + (8 * n ** 3 + 6 * n ** 4)
        vol = 14 * n ** 3 + 20 * n * n
        return 2.0 * cells * (per + vol * (4 if d["system"] == I.EULER else 1))

    def floats(d):
        n = d["degree"] + 1
        cells = d["nx"] * d["ny"]
        if d["kind"] == I.CG:
            return cells * d["degree"] ** d["dim"]
        return cells * n ** d["dim"] * (4 if d["system"] == I.EULER else 1)

    if do == "batch":
        ds = batch_descs(case, 0)
        return dict(bytes=8.0 * sum(map(floats, ds)), flops=3.0 * sum(map(stage_flops, ds)))
    d = desc(case)
    if do == "project":
        n = case["p"] + 1
        modes = 4 if case["ic"] == "fourier" else 1
        return dict(bytes=4.0 * floats(d), flops=d["nx"] * d["ny"] * 144.0 * (10 * modes) + 2.0 * floats(d) * (144 / n + 12))
    if do == "residual":
        return dict(bytes=8.0 * floats(d), flops=stage_flops(d))
    return dict(bytes=8.0 * floats(d) * case.get("steps", 1), flops=3.0 * stage_flops(d) * case.get("steps", 1))


# ---- the same results in 64 bits ------------------------------------------------------------


def gll(p):
    """Gauss-Lobatto-Legendre nodes."""
    c = np.zeros(p + 1)
    c[p] = 1.0
    inner = np.polynomial.legendre.legroots(np.polynomial.legendre.legder(c)) if p > 1 else []
    return np.concatenate([[-1.0], np.sort(np.real(inner)), [1.0]])


def leg(x, m, k=0):
    """D^j P_i(x) for i < m at every x: [k + 1][len(x)][m]."""
    out = np.zeros((k + 1, len(x), m))
    for i in range(m):
        c = np.zeros(m)
        c[i] = 1.0
        for j in range(k + 1):
            out[j, :, i] = np.polynomial.legendre.legval(np.asarray(x), np.polynomial.legendre.legder(c, j) if j else c)
    return out


class Space:
    """Tables of one mesh: per direction Gauss values, corner derivatives, semi-norm Gram matrix, Taylor maps.  A 1D
    mesh is a 2D one with a single constant mode, one node of weight 2 and no faces in y."""

    def __init__(self, d):
        self.d, p = d, d["degree"]
        self.dim, self.nx, self.ny = d["dim"], d["nx"], d["ny"] if d["dim"] == 2 else 1
        self.p, n = p, p + 1
        t = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device=DEV)  # noqa: E731
        self.dx = (d["x1"] - d["x0"]) / self.nx
        self.dy = (d["y1"] - d["y0"]) / self.ny if self.dim == 2 else 1.0
        self.h = math.hypot(self.dx, self.dy) if self.dim == 2 else self.dx
        self.per = [d["bc"][0] == I.PERIODIC, self.dim == 1 or d["bc"][2] == I.PERIODIC]
        x, w = np.polynomial.legendre.leggauss(n)
        x8, w8 = np.polynomial.legendre.leggauss(8)

        def tables(m):
            if m == 1:
                one = t([[1.0]])
                return dict(D=one[None], w=t([2.0]), E=(one, one), g=t([[[2.0]]]), T=(one, one), n=1)
            D8 = leg(x8, m, p)
            T = [[[(i + 0.5) * np.sum(w8 * D8[0][:, i] * (x8 - s) ** k) / math.factorial(k) for k in range(m)]
                  for i in range(m)] for s in (-1.0, 1.0)]
            return dict(D=t(leg(x, m, p)), w=t(w), E=tuple(t(leg([s], m, p)[:, 0]) for s in (-1.0, 1.0)),
                        g=t(np.einsum("q,kqa,kqb->kab", w8, D8, D8)), T=(t(T[0]), t(T[1])), n=m)

        self.x, self.y = tables(n), tables(n if self.dim == 2 else 1)
        # weights (h 2/dx)^(2kx) (h 2/dy)^(2ky) of the pointwise semi-norm, and the element one with |J| / h^dim
        kx, ky = torch.arange(self.x["n"], device=DEV), torch.arange(self.y["n"], device=DEV)
        sg = ((2 * self.h / self.dx) ** (2 * kx.double()))[None, :] * ((2 * self.h / self.dy) ** (2 * ky.double()))[:, None]
        sg[0, 0] = 0.0
        self.sigma = sg
        jac = self.dx * self.dy / 4 / self.h ** 2 if self.dim == 2 else 0.25 * self.dx / self.h  # (y rule has weight 2)
        nd = self.x["n"] * self.y["n"]
        self.G = jac * torch.einsum("lk,lab,kcd->acbd", sg, self.y["g"], self.x["g"]).reshape(nd, nd)
        i = torch.arange(self.x["n"], device=DEV).double()
        j = torch.arange(self.y["n"], device=DEV).double()
        self.minv = 0.25 * (2 * j[:, None] + 1) * (2 * i + 1)
        self.W = self.y["w"][:, None] * self.x["w"]

    def at(self, c, ky=0, kx=0):
        """D^(ky,kx) at the Gauss nodes, reference derivatives: [..., qy, qx]."""
        return torch.einsum("qb,ra,...ba->...qr", self.y["D"][ky], self.x["D"][kx], c)

    def grad(self, c):
        gx = self.at(c, 0, 1) * (2 / self.dx)
        return gx, (self.at(c, 1, 0) * (2 / self.dy) if self.dim == 2 else torch.zeros_like(gx))

    def vertices(self, c):
        """Vertex candidates t*[ny + 1, nx + 1, ky, kx] (the last row/column repeats the first on periodic sides)."""
        P = self.d
        A = c.new_zeros((self.ny + 1, self.nx + 1) + tuple(c.shape[2:]))
        S = c.new_zeros((self.ny + 1, self.nx + 1))
        for cy in ((0, 1) if self.dim == 2 else (0,)):
            for cx in (0, 1):
                t = torch.einsum("lb,ka,jiba->jilk", self.y["E"][cy], self.x["E"][cx], c)
                w = (P["eps"] + (self.sigma * t * t).sum((-1, -2)).sqrt()) ** -P["r"]
                A[cy:cy + self.ny, cx:cx + self.nx] += w[..., None, None] * t
                S[cy:cy + self.ny, cx:cx + self.nx] += w
        for v in (A, S):
            if self.per[0]:
                v[:, 0] += v[:, -1]
                v[:, -1] = v[:, 0]
            if self.dim == 2 and self.per[1]:
                v[0] += v[-1]
                v[-1] = v[0]
        if self.dim == 1:
            A, S = A[:1], S[:1]
        return A / S[..., None, None]

    def norm(self, v):
        return torch.einsum("...a,ab,...b->...", v, self.G, v).clamp_min(0).sqrt()

    def sensor(self, c, net=None):
        """(gamma, ||u||_e, reconstruction's modes) of the cells c[ny, nx, my, mx]."""
        P, T = self.d, self.vertices(c)
        flat = lambda v: torch.cat([torch.zeros_like(v.flatten(-2)[..., :1]), v.flatten(-2)[..., 1:]], -1)  # noqa: E731
        v0 = flat(c)
        n0 = self.norm(v0)
        nc = 2 ** self.dim
        om = (1 - nc * P["gamma_vertex"]) / (P["eps"] + n0) ** P["r"]
        num, den, feats = om[..., None] * v0, om, []
        for cy in ((0, 1) if self.dim == 2 else (0,)):
            for cx in (0, 1):
                t = T[cy:cy + self.ny, cx:cx + self.nx]
                whole = torch.einsum("bl,ak,jilk->jiba", self.y["T"][cy], self.x["T"][cx], t)
                if net is not None:
                    feats += [whole[..., 0, 0] - c[..., 0, 0], self.h * 2 / self.dx * t[..., 0, 1], self.h * 2 / self.dy * t[..., 1, 0]]
                t = t.clone()
                t[..., 0, 0] = 0.0
                v = flat(torch.einsum("bl,ak,jilk->jiba", self.y["T"][cy], self.x["T"][cx], t))
                om = P["gamma_vertex"] / (P["eps"] + self.norm(v)) ** P["r"]
                num, den = num + om[..., None] * v, den + om
        star = num / den[..., None]
        gam = 1 - (self.norm(v0 - star) / n0.clamp_min(1e-300)).clamp_max(1.0)
        gam = torch.where(n0 <= 1e-30, torch.ones_like(gam), gam)
        if net is not None:
            X = (torch.stack(feats, -1) / (n0 + P["eps"])[..., None]).clamp(-8, 8)
            o = mlp(net, X, rounded=True)
            g = torch.where(torch.sigmoid(o[..., 1]) >= 0.5, torch.sigmoid(o[..., 0]), gam)
            gam = torch.where(n0 > 1e-5 * (c[..., 0, 0].abs() + 1), g, torch.ones_like(g))
        return gam, n0, star.reshape(c.shape)

    def alpha(self, c, gam, n0, f):
        """Shock-capturing weights for the dissipation f[V, ny, nx, qy, qx], indicator from c[ny, nx, my, mx]."""
        s = sum(self.sigma[l, k] * self.at(c, l, k) ** 2 for l in range(self.y["n"]) for k in range(self.x["n"]) if l + k).sqrt()
        s1, s2 = (self.W * f).sum((-1, -2)), (self.W * s * f).sum((-1, -2))
        on = (gam < self.d["c_gamma"]) & (n0 > 1e-30) & (s1 > 0) & (s2 > 0)
        return torch.where(on[..., None, None], s * (s1 / torch.where(on, s2, torch.ones_like(s2)))[..., None, None], torch.ones_like(f))


def flux(d, u):
    """(f_x, f_y, speed for nu, |f_x'|, |f_y'|) of states u[V, ...]; for Euler also the sound speed and velocity."""
    s = d["system"]
    if s == I.BURGERS:
        f = 0.5 * u * u
        return f, f, (math.sqrt(2.0) if d["dim"] == 2 else 1.0) * u[0].abs(), u[0].abs(), u[0].abs()
    if s == I.KPP:
        return torch.sin(u), torch.cos(u), torch.ones_like(u[0]), torch.cos(u[0]).abs(), torch.sin(u[0]).abs()
    if s == I.LINADV:
        o = torch.ones_like(u[0])
        vx, vy = d["adv_vx"], d["adv_vy"]
        return vx * u, vy * u, (math.hypot(vx, vy) if d["dim"] == 2 else abs(vx)) * o, abs(vx) * o, abs(vy) * o
    g = d["gas_gamma"]
    vx, vy = u[1] / u[0], u[2] / u[0]
    p = (g - 1) * (u[3] - 0.5 * (u[1] * vx + u[2] * vy))
    c = (g * p.clamp_min(0) / u[0].abs()).sqrt()
    fx = torch.stack([u[1], u[1] * vx + p, u[2] * vx, (u[3] + p) * vx])
    fy = torch.stack([u[2], u[1] * vy, u[2] * vy + p, (u[3] + p) * vy])
    return fx, fy, (vx * vx + vy * vy).sqrt() + c, (vx, c), (vy, c)


def face_flux(d, ul, ur, axis):
    fl, fr = flux(d, ul), flux(d, ur)
    a, b = fl[axis], fr[axis]
    if d["system"] == I.EULER:
        (vl, cl), (vr, cr) = fl[3 + axis], fr[3 + axis]
        sl, sr = torch.minimum(vl - cl, vr - cr), torch.maximum(vl + cl, vr + cr)
        mid = (sr * a - sl * b + sl * sr * (ur - ul)) / (sr - sl)
        return torch.where(sl >= 0, a, torch.where(sr <= 0, b, mid))
    lam = d["lambda_const"] if d["lambda_const"] > 0 else torch.maximum(fl[3 + axis], fr[3 + axis])
    return 0.5 * (a + b) - 0.5 * lam * (ur - ul)


def traces(S, c):
    """Values at the face nodes: left, right [V, ny, nx, qy], bottom, top [V, ny, nx, qx]."""
    ex, ey = S.x["E"], S.y["E"]
    out = [torch.einsum("qb,a,...ba->...q", S.y["D"][0], ex[s][0], c) for s in (0, 1)]
    return out + [torch.einsum("b,qa,...ba->...q", ey[s][0], S.x["D"][0], c) for s in (0, 1)] if S.dim == 2 else out


def dg_residual(S, c, net=None):
    """du/dt of c[V, ny, nx, my, mx]."""
    d = S.d
    gam, n0, _ = S.sensor(c[0], net)
    u = S.at(c)
    tr = traces(S, c)
    fx, fy, speed = flux(d, u)[:3]
    if d["lambda_const"] > 0:
        lam = torch.full_like(gam, d["lambda_const"])
    else:
        lam = speed.amax((-1, -2))
        for v in tr:
            lam = torch.maximum(lam, flux(d, v)[2].amax(-1))
    mu = ((1 - gam) * lam * S.h / (2 * S.p))[..., None, None]
    gx, gy = S.grad(c)
    al = S.alpha(c[0], gam, n0, gx * gx + gy * gy)
    r = (2 / S.dx) * torch.einsum("qb,ra,...qr->...ba", S.y["D"][0], S.x["D"][1] if S.x["n"] > 1 else S.x["D"][0] * 0, S.W * (fx - mu * al * gx))
    if S.dim == 2:
        r = r + (2 / S.dy) * torch.einsum("qb,ra,...qr->...ba", S.y["D"][1], S.x["D"][0], S.W * (fy - mu * al * gy))
    for axis in range(S.dim):
        lo, hi = tr[2 * axis], tr[2 * axis + 1]
        at = 2 if axis == 0 else 1
        right = torch.roll(lo, -1, at)
        if not S.per[axis]:
            last = (slice(None),) * at + (-1,)
            right[last] = hi[last]
        F = face_flux(d, hi, right, axis)           # flux at each cell's upper face
        Fl = torch.roll(F, 1, at)
        if not S.per[axis]:
            first = (slice(None),) * at + (0,)
            Fl[first] = face_flux(d, lo[first], lo[first], axis)
        if axis == 0:
            T = lambda f, s: torch.einsum("q,qb,a,...q->...ba", S.y["w"], S.y["D"][0], S.x["E"][s][0], f)  # noqa: E731
            r = r - (2 / S.dx) * (T(F, 1) - T(Fl, 0))
        else:
            T = lambda f, s: torch.einsum("q,b,qa,...q->...ba", S.x["w"], S.y["E"][s][0], S.x["D"][0], f)  # noqa: E731
            r = r - (2 / S.dy) * (T(F, 1) - T(Fl, 0))
    return r * S.minv


def limited(S, c):
    """Average-preserving reconstruction in the cells whose sensor is below c_gamma."""
    gam, n0, star = S.sensor(c[0])
    star = star.clone()
    star[..., 0, 0] = c[0, ..., 0, 0]
    return torch.where(((gam < S.d["c_gamma"]) & (n0 > 1e-30))[..., None, None], star, c[0])[None]


def positive(S, c):
    """Scaling limiter at the volume and face Gauss nodes."""
    nodes = torch.cat([S.at(c).flatten(-2)] + traces(S, c), -1)     # [4, ny, nx, points]
    mean = c[..., 0, 0]
    pr = lambda u: 0.4 * (u[3] - 0.5 * (u[1] ** 2 + u[2] ** 2) / u[0])  # noqa: E731
    pb = pr(mean)
    ok = (mean[0] > 0) & (pb > 0)
    eps = 1e-3 * torch.minimum(mean[0], pb)
    rmin = torch.minimum(nodes[0].amin(-1), mean[0])
    th1 = torch.where(rmin < eps, ((mean[0] - eps) / (mean[0] - rmin).clamp_min(1e-300)).clamp_max(1.0), torch.ones_like(eps))
    dev = nodes - mean[..., None]
    dev[0] = dev[0] * th1[..., None]
    bad = pr(mean[..., None] + dev) < eps[..., None]
    lo, hi = torch.zeros_like(dev[0]), torch.ones_like(dev[0])
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        above = pr(mean[..., None] + mid * dev) >= eps[..., None]
        lo, hi = torch.where(above, mid, lo), torch.where(above, hi, mid)
    th2 = torch.where(bad, lo, torch.ones_like(lo)).amin(-1)
    th1, th2 = (torch.where(ok, t, torch.ones_like(t)) for t in (th1, th2))
    out = c * th2[..., None, None]
    out[0] = out[0] * th1[..., None, None]
    out[..., 0, 0] = mean
    return out


def rk3(u, dt, f, after=lambda v: v):
    u1 = after(u + dt * f(u))
    u2 = after(0.75 * u + 0.25 * (u1 + dt * f(u1)))
    return after(u / 3 + 2 / 3 * (u2 + dt * f(u2)))


class CgSpace(Space):
    """The continuous space: nodal values [nny, nnx] on the periodic Gauss-Lobatto lattice."""

    def __init__(self, d):
        super().__init__(d)
        p, n = self.p, self.p + 1
        t = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device=DEV)  # noqa: E731
        xg = gll(p)
        x8, w8 = np.polynomial.legendre.leggauss(8)
        x, _ = np.polynomial.legendre.leggauss(n)
        inv = np.linalg.inv(leg(xg, n)[0])                     # modes of the nodal basis: P(xg) c = u
        nodal = lambda at, k=0: leg(at, n, k)[k] @ inv          # noqa: E731  [q][a] values of D^k l_a
        M = np.einsum("q,qa,qb->ab", w8, nodal(x8), nodal(x8))
        one = t([[1.0]])
        mk = lambda: dict(V=t(inv), L=t(nodal(x)), D=t(nodal(x, 1)), M=t(M), w=t(M.sum(1)))  # noqa: E731
        self.cx = mk()
        self.cy = mk() if self.dim == 2 else dict(V=one, L=one, D=one * 0, M=2 * one, w=t([2.0]))
        ix = (p * torch.arange(self.nx, device=DEV)[:, None] + torch.arange(n, device=DEV)) % (p * self.nx)
        iy = ((p * torch.arange(self.ny, device=DEV)[:, None] + torch.arange(n, device=DEV)) % (p * self.ny) if self.dim == 2
              else torch.zeros(1, 1, dtype=torch.long, device=DEV))
        self.nnx, self.nny = p * self.nx, p * self.ny if self.dim == 2 else 1
        self.index = (iy[:, None, :, None] * self.nnx + ix[None, :, None, :])
        self.jac = self.dx * self.dy / 4 if self.dim == 2 else self.dx / 4
        self.ml = self.add(self.jac * (self.cy["w"][:, None] * self.cx["w"]).expand(self.ny, self.nx, -1, -1))

    def add(self, loc):
        return loc.new_zeros(self.nnx * self.nny).index_add_(0, self.index.reshape(-1), loc.reshape(-1))

    def residual(self, u):
        d, X, Y = self.d, self.cx, self.cy
        ul = u[self.index]
        c = torch.einsum("mb,ka,jiba->jimk", Y["V"], X["V"], ul)
        gam, n0, _ = self.sensor(c)
        uq = self.at(c)
        if d["lambda_const"] > 0:
            lam = torch.full_like(gam, d["lambda_const"])
        else:
            lam = flux(d, uq[None])[2].amax((-1, -2))
            for v in traces(self, c[None]):
                lam = torch.maximum(lam, flux(d, v)[2].amax(-1))
        gx, gy = self.grad(c)
        W = self.jac * self.W
        ph = []
        for gr in (gx, gy):
            b = self.add(torch.einsum("qb,ra,jiqr->jiba", Y["L"], X["L"], W * gr)) / self.ml
            ph.append(torch.einsum("qb,ra,jiba->jiqr", Y["L"], X["L"], b[self.index]))
        g = gam[..., None, None]
        al = self.alpha(c, gam, n0, gx * gx + gy * gy - g * (gx * ph[0] + gy * ph[1]))
        fx, fy = flux(d, uq[None])[:2]
        nu = (lam * self.h / (2 * self.p))[..., None, None] * al
        r = (2 / self.dx) * torch.einsum("qb,ra,jiqr->jiba", Y["L"], X["D"], W * (fx[0] - nu * (gx - g * ph[0])))
        if self.dim == 2:
            r = r + (2 / self.dy) * torch.einsum("qb,ra,jiqr->jiba", Y["D"], X["L"], W * (fy[0] - nu * (gy - g * ph[1])))
        r = self.add(r)
        du = r / self.ml
        for _ in range(2):
            mdu = self.add(self.jac * torch.einsum("mb,ka,jiba->jimk", Y["M"], X["M"], du[self.index]))
            du = du + (r - mdu) / self.ml
        return du


def bf16(x):
    return x.float().bfloat16().double()


def mlp(w, X, rounded=False):
    """The network on inputs X[..., 12]; weights w (flat) and inputs in bfloat16, activations too where rounded."""
    W1, b1, W2, b2, W3, b3 = (w[a:b] for a, b in ((0, 768), (768, 832), (832, 4928), (4928, 4992), (4992, 5120), (5120, 5122)))

    def gelu(z):
        a = 0.5 * z * (1 + torch.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3)))
        return bf16(a) if rounded else a

    a = gelu(bf16(X) @ bf16(W1).reshape(64, 12).T + b1)
    a = gelu(a @ bf16(W2).reshape(64, 64).T + b2)
    return a @ bf16(W3).reshape(2, 64).T + b3


class RoundWeights(torch.autograd.Function):
    """bfloat16 rounding whose gradient is passed through (the gradient is taken at the rounded weights)."""

    @staticmethod
    def forward(ctx, x):
        return bf16(x)

    @staticmethod
    def backward(ctx, g):
        return g


def train_exact(case, seed):
    X, y = samples(case, seed)
    X, y = bf16(X), y.double()
    w = torch.tensor(network(seed), dtype=torch.float32, device=DEV).double()
    weights = torch.ones(5122, dtype=torch.bool, device=DEV)
    weights[768:832] = weights[4928:4992] = weights[5120:] = False
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    t = 0
    for b0 in range(0, case["samples"], case["batch"]):
        xb, yb = X[b0:b0 + case["batch"]], y[b0:b0 + case["batch"]]
        w.requires_grad_(True)
        r = torch.where(weights, RoundWeights.apply(w), w)
        gelu = lambda z: 0.5 * z * (1 + torch.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3)))  # noqa: E731
        a = gelu(xb @ r[:768].reshape(64, 12).T + r[768:832])
        a = gelu(a @ r[832:4928].reshape(64, 64).T + r[4928:4992])
        o = a @ r[4992:5120].reshape(2, 64).T + r[5120:]
        gh = torch.sigmoid(o[:, 0])
        hit = ((gh - yb).abs() < 0.05).double().detach()
        loss = ((gh - yb) ** 2 + 0.1 * (torch.nn.functional.softplus(o[:, 1]) - hit * o[:, 1])).mean()
        (g,) = torch.autograd.grad(loss, w)
        w, t = w.detach(), t + 1
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        w = w - 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return dict(loss=loss.detach(), params=w)


def project_exact(case, seed):
    d = desc(case)
    kind, prm = datum(case, seed)
    nx, ny, n = d["nx"], d["ny"], d["degree"] + 1
    f64 = dict(dtype=torch.float64, device=DEV)
    qn, qw = np.polynomial.legendre.leggauss(12)
    q = torch.tensor(qn, **f64)
    L = torch.tensor(leg(qn, n)[0] * qw[:, None] * (np.arange(n) + 0.5), **f64)
    dx, dy = (d["x1"] - d["x0"]) / nx, (d["y1"] - d["y0"]) / ny
    x = d["x0"] + dx * (torch.arange(nx, **f64)[:, None] + 0.5 + 0.5 * q)
    out = []
    for j0 in range(0, ny, 32):
        y = d["y0"] + dy * (torch.arange(j0, min(ny, j0 + 32), **f64)[:, None] + 0.5 + 0.5 * q)
        Y, X = torch.broadcast_tensors(y[:, None, :, None], x[None, :, None, :])
        if kind == I.IC_FOURIER:
            u = torch.zeros_like(X)[None]
            for k in range(int(prm[0])):
                a, kx, ky, ph = prm[1 + 4 * k:5 + 4 * k]
                u = u + a * torch.sin(2 * math.pi * (kx * (X - d["x0"]) / (d["x1"] - d["x0"]) + ky * (Y - d["y0"]) / (d["y1"] - d["y0"])) + ph)
        elif kind == I.IC_CIRCLE:
            u = torch.where(X * X + Y * Y <= prm[2] ** 2, prm[3] + 0 * X, prm[4] + 0 * X)[None]
        else:
            s = torch.tensor(prm[2:18], **f64).reshape(4, 4)[(X >= prm[0]).long() + 2 * (Y >= prm[1]).long()]
            rho, vx, vy, pr = s.unbind(-1)
            u = torch.stack([rho, rho * vx, rho * vy, pr / 0.4 + 0.5 * rho * (vx * vx + vy * vy)])
        out.append(torch.einsum("vjiab,am,bk->vjimk", u, L, L))
    u = torch.cat(out, 1)
    return u.reshape(u.shape[0], nx * ny, n * n)


def advance_exact(d, u32, dt, steps, net=None, residual_only=False):
    if d["kind"] == I.CG:
        S = CgSpace(d)
        u = u32.double().reshape(-1)
        for _ in range(steps):
            u = rk3(u, dt, S.residual)
        return u.reshape(u32.shape)
    S = Space(d)
    c = u32.double().reshape(u32.shape[0], S.ny, S.nx, S.y["n"], S.x["n"])
    f = lambda v: dg_residual(S, v, net)  # noqa: E731
    if residual_only:
        return f(c).reshape(u32.shape)
    after = (lambda v: limited(S, v)) if d["hweno_limiter"] else (lambda v: positive(S, v)) if d["positivity"] else (lambda v: v)
    for _ in range(steps):
        c = rk3(c, dt, f, after)
    return c.reshape(u32.shape)


def exact(case, seed):
    do = case["do"]
    if do == "train":
        return train_exact(case, seed)
    if do == "project":
        return project_exact(case, seed)
    if do == "batch":
        return torch.cat([advance_exact(d, start_state(d, seed + 31 * k), time_step(d), 1).reshape(-1)
                          for k, d in enumerate(batch_descs(case, seed))])
    d = desc(case)
    u = start_state(d, seed)
    if do == "residual":
        return advance_exact(d, u, 0.0, 0, residual_only=True)
    if do == "cfl":
        S = Space(d)
        c = positive(S, u.double().reshape(4, S.ny, S.nx, S.y["n"], S.x["n"]))
        lam = max(float(flux(d, v)[2].max()) for v in [S.at(c)] + traces(S, c))
        dt = cfl(d) * min(S.dx, S.dy) / (2 * lam)
        c = rk3(c, dt, lambda v: dg_residual(S, v), lambda v: positive(S, v))
        return dict(u=c.reshape(u.shape), dt=dt, totals=c[..., 0, 0].sum((1, 2)) * S.dx * S.dy)
    net = None
    if do == "surrogate":
        net = torch.tensor(network(seed), dtype=torch.float32, device=DEV).double()
    return advance_exact(d, u, time_step(d), case["steps"], net)
