"""What a user of this library has it do, over the range of sizes in which it is used.

A case is one call (or the few calls that belong together) on one node set: a nonlocal sum, RK4
steps of the neural field, a model of §5, a gradient through RK4 steps, or the setup of a node
set (stencils and quadrature weights).  The listed cases follow the workloads of
``nodesets/workloads.py`` and of the benchmark; ``draw`` spreads the same calls over sizes,
kernels, operator paths and trajectory counts.

``exact`` evaluates the same formulas with torch in FP64 (dense matrices, batched solves).
"""
from __future__ import annotations

import math

import torch

import paper_2504_13379_gb300 as nf

DEV = "cuda"
HAT = "1.0,0.1,0.5,0.2"          # the lateral-inhibition kernel of the workloads (s2 = 2 s1)
WIDE = "1.2,0.08,0.6,0.25"       # the gradient workload's target kernel (no integer width ratio)
ONE = "1.0,0.1,0.0,0.2"          # one Gaussian
SIGMA = 1.0 / 40.0               # width of the convergence study's Gaussian kernel
PATHS = {"mf": nf.MATRIX_FREE, "fp32": nf.DENSE_FP32, "bf16x2": nf.DENSE_BF16X2, "sym": nf.DENSE_SYM_FP32,
         "sym_bf16x2": nf.DENSE_SYM_BF16X2}


def listed():
    return [
        # one right-hand side on a small surface mesh, as an outside integrator asks for it
        dict(name="apply_sphere_2003", do="apply", path="mf", shape="sphere", n=2003, B=1, kernel=HAT),
        # the flat unit square's whole run: 100 small RK4 steps in one call
        dict(name="flat_1500_rk4x100", do="rk4", path="mf", shape="square", n=1500, B=1, kernel=HAT, steps=100, dt=0.05),
        # the manufactured solution on the sphere: forced steps at a medium size
        dict(name="sphere_20000_forced", do="rk4", path="mf", shape="sphere", n=20000, B=1, kernel=HAT, steps=10,
             dt=0.01, forcing="sphere"),
        # a step of the torus workload, the largest Euclidean one
        dict(name="torus_100000_step", do="rk4", path="mf", shape="torus", n=100000, B=1, kernel=HAT, steps=1, dt=0.05),
        # a step of the convergence study on the periodic square (narrow Gaussian, moving forcing)
        dict(name="periodic_131072_step", do="rk4", path="mf", shape="periodic", n=131072, B=1, kernel="gauss", steps=1,
             dt=0.01, forcing="flat"),
        # a parameter sweep: twelve trajectories of one ellipsoid, without a stored matrix
        dict(name="sweep_15000x12", do="rk4", path="mf", shape="ellipsoid", n=15000, B=12, kernel=HAT, steps=1, dt=0.05),
        # three trajectories over a stored operator in its bf16 hi + lo form
        dict(name="dense_bf16x2_30000x3", do="rk4", path="bf16x2", shape="ellipsoid", n=30000, B=3, kernel=HAT, steps=1,
             dt=0.05),
        # one trajectory over the symmetric stored operator, a size whose steps are short
        dict(name="dense_sym_8000", do="rk4", path="sym", shape="sphere", n=8000, B=1, kernel=HAT, steps=10, dt=0.05),
        # the batched workload: 448 trajectories of four node sets on the tensor cores
        dict(name="batched_448_step", do="grouped", sets="40000x256,8000x64,15000x64,30000x64", kernel=HAT, steps=1,
             dt=0.05),
        # a training step of the differentiation workload: forward, loss and gradients
        dict(name="gradient_40000", do="grad", shape="torus", n=40000, B=1, kernel=HAT, steps=20, every=10, dt=0.02),
        # from a triangulated surface to its quadrature weights
        dict(name="setup_torus_100000", do="setup", shape="torus", n=100000, k=48, deg=4),
        # the synaptic-depression model of §5 with its Adams-Bashforth integrator
        dict(name="depression_30000", do="model", path="mf", shape="torus", n=30000, B=1, kernel=HAT, steps=12, dt=0.05,
             integrator="ab5"),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    do = rng.choice(["flow", "flow", "periodic", "sweep", "dense", "dense", "grouped", "grad", "setup", "setup", "model"])
    kernel = rng.choice([HAT, HAT, WIDE, ONE])
    if do == "flow":
        n, B = size(500, 100000), rng.choice([1, 1, 2, 3])
        if rng.random() < 0.3:
            return dict(do="apply", path="mf", shape=rng.choice(["square", "sphere", "torus"]), n=n, B=B, kernel=kernel)
        return dict(do="rk4", path="mf", shape=rng.choice(["square", "sphere", "ellipsoid", "torus"]), n=n, B=B,
                    kernel=kernel, steps=rng.randint(1, max(1, min(40, int(4e10 / (n * n * B))))), dt=0.05)
    if do == "periodic":
        return dict(do="rk4", path="mf", shape="periodic", n=size(4000, 131072), B=1, kernel="gauss", steps=1, dt=0.01,
                    forcing="flat")
    if do == "sweep":
        return dict(do="rk4", path="mf", shape=rng.choice(["sphere", "ellipsoid", "torus"]), n=size(1500, 20000),
                    B=rng.randint(4, 32), kernel=kernel, steps=1, dt=0.05)
    if do == "dense":
        path = rng.choice(["fp32", "bf16x2", "sym", "sym_bf16x2"])
        B = rng.choice([1, 1, 2, 3, 4, 6]) if path != "fp32" else rng.choice([1, 2, 5, 16, 64])
        n = size(700, 32000)
        return dict(do="rk4", path=path, shape=rng.choice(["square", "sphere", "torus"]), n=n, B=B, kernel=kernel,
                    steps=rng.randint(1, max(1, min(20, int(4e9 / (n * n * B))))), dt=0.05)
    if do == "grouped":
        sets = ",".join("%dx%d" % (size(2000, 20000), rng.randint(8, 160)) for _ in range(rng.randint(1, 4)))
        return dict(do="grouped", sets=sets, kernel=kernel, steps=rng.randint(1, 3), dt=0.05)
    if do == "grad":
        steps = rng.randint(2, 20)
        return dict(do="grad", shape=rng.choice(["torus", "sphere"]), n=size(2000, 40000), B=rng.choice([1, 1, 2]),
                    kernel=rng.choice([HAT, HAT, WIDE]), steps=steps, every=rng.randint(1, steps), dt=0.02)
    if do == "setup":
        k, deg = rng.choice([(21, 2), (24, 2), (32, 3), (48, 4)])
        return dict(do="setup", shape=rng.choice(["torus", "square"]), n=size(1500, 100000), k=k, deg=deg)
    n = size(2000, 60000)
    return dict(do="model", path=rng.choice(["mf", "mf", "sym"] if n <= 30000 else ["mf"]), shape="torus", n=n,
                B=rng.choice([1, 2]), kernel=kernel, steps=rng.randint(5, 12), dt=0.05,
                integrator=rng.choice(["ab5", "rk4"]))


# ---------------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _lattice(n, aspect, closed):
    """Rows and columns of a staggered lattice of about n nodes (rows even where it closes on
    itself), and its triangles."""
    rows = max(4, int(round(math.sqrt(n / aspect))))
    if closed:  # a row count that divides n where there is one nearby
        rows += rows % 2
        near = [r for r in range(4, 2 * rows, 2) if n % r == 0 and 8 * abs(r - rows) <= rows]
        rows = min(near, key=lambda r: abs(r - rows)) if near else rows
    cols = max(4, n // rows)
    t = torch.arange(rows, device=DEV).view(-1, 1)
    p = torch.arange(cols, device=DEV).view(1, -1)
    if not closed:
        t, p = t[:-1], p[:, :-1]
    t1, p1 = (t + 1) % rows, (p + 1) % cols
    a, b, c, d = t * cols + p, t * cols + p1, t1 * cols + p, t1 * cols + p1
    even = ((t % 2) == 0).expand_as(a)
    one = torch.where(even.unsqueeze(-1), torch.stack([a, b, c], -1), torch.stack([a, d, c], -1))
    two = torch.where(even.unsqueeze(-1), torch.stack([b, d, c], -1), torch.stack([a, b, d], -1))
    return rows, cols, torch.cat([one.reshape(-1, 3), two.reshape(-1, 3)]).to(torch.int32).contiguous()


def _nodes(shape, n, g):
    """Nodes (FP64), local areas, outward normals, triangles (None where a case needs none)."""
    if shape in ("sphere", "ellipsoid"):
        i = torch.arange(n, device=DEV, dtype=torch.float64)
        z = 1.0 - (2.0 * i + 1.0) / n
        rho, phi = (1.0 - z * z).clamp_min(0).sqrt(), i * (math.pi * (3.0 - math.sqrt(5.0)))
        x = torch.stack([rho * phi.cos(), rho * phi.sin(), z], 1)
        x = x + 0.2 * math.sqrt(4.0 * math.pi / n) * (_uniform(g, n, 3) - 0.5)
        x = x / x.norm(dim=1, keepdim=True)
        area = torch.full((n,), 4.0 * math.pi / n, device=DEV, dtype=torch.float64)
        if shape == "ellipsoid":
            ax = torch.tensor([1.0, 0.8, 0.6], device=DEV, dtype=torch.float64)
            area = area * ax.prod() * (x / ax).norm(dim=1)
            x = x * ax
        return x, area, None, None
    if shape == "torus":
        rows, cols, tris = _lattice(n, math.sqrt(3.0) / 2.0 * 2.5, True)
        t = torch.arange(rows, device=DEV, dtype=torch.float64).view(-1, 1).expand(rows, cols).reshape(-1)
        p = torch.arange(cols, device=DEV, dtype=torch.float64).view(1, -1).expand(rows, cols).reshape(-1)
        j = 0.3 * (_uniform(g, rows * cols, 2) - 0.5)
        phi, th = (p + 0.5 * (t % 2) + j[:, 0]) * (2 * math.pi / cols), (t + j[:, 1]) * (2 * math.pi / rows)
        w = 1.0 + 0.4 * th.cos()
        x = torch.stack([w * phi.cos(), w * phi.sin(), 0.4 * th.sin()], 1)
        nrm = torch.stack([th.cos() * phi.cos(), th.cos() * phi.sin(), th.sin()], 1)
        return x, 0.4 * w * (4 * math.pi ** 2 / (rows * cols)), nrm, tris
    if shape == "square":  # scattered nodes of the unit square, on a staggered lattice
        rows, cols, tris = _lattice(n, math.sqrt(3.0) / 2.0, False)
        t = torch.arange(rows, device=DEV, dtype=torch.float64).view(-1, 1).expand(rows, cols).reshape(-1)
        p = torch.arange(cols, device=DEV, dtype=torch.float64).view(1, -1).expand(rows, cols).reshape(-1)
        j = 0.3 * (_uniform(g, rows * cols, 2) - 0.5)
        x = torch.stack([(p + 0.5 * (t % 2) + j[:, 0]) / cols, (t + j[:, 1]) / rows], 1)
        return x, torch.full((x.shape[0],), 1.0 / x.shape[0], device=DEV, dtype=torch.float64), None, tris
    x = 2 * math.pi * _halton(n, g)  # the periodic square [0, 2 pi)^2
    return x, torch.full((n,), 4 * math.pi ** 2 / n, device=DEV, dtype=torch.float64), None, None


def _halton(n, g):
    """n Halton (2, 3) points of the unit square, shifted by a random offset (modulo 1)."""
    out = []
    for base in (2, 3):
        i, f, v = torch.arange(1, n + 1, device=DEV), 1.0, torch.zeros(n, device=DEV, dtype=torch.float64)
        while int(i.max()) > 0:
            f /= base
            v += f * (i % base)
            i = i // base
        out.append(v)
    return (torch.stack(out, 1) + _uniform(g, 1, 2)) % 1.0


def _kernel(case):
    if case["kernel"] == "gauss":  # the convergence study: a normalised Gaussian, period 2 pi
        return (1.0 / (2 * math.pi * SIGMA ** 2), math.sqrt(2.0) * SIGMA, 0.0, 1.0, 2 * math.pi)
    return tuple(float(v) for v in case["kernel"].split(",")) + (0.0,)


def _bumps(x, B, g):
    """B states of six localised bumps at random nodes."""
    at = x[torch.randint(0, x.shape[0], (B, 6), generator=g, device=DEV)]
    amp = 0.5 + 0.5 * _uniform(g, B, 6, 1)
    d2 = ((x.view(1, 1, -1, x.shape[1]) - at.unsqueeze(2)) ** 2).sum(-1)
    return (amp * torch.exp(-d2 / 0.15 ** 2)).sum(1)


def _node_set(shape, n, g):
    """x (n x 3) and q in FP32, as the operators take them: areas with the scatter of RBF weights."""
    x, area, _, _ = _nodes(shape, n, g)
    if x.shape[1] == 2:
        x = torch.cat([x, torch.zeros_like(x[:, :1])], 1)
    q = area * (1.0 + 0.2 * (_uniform(g, x.shape[0]) - 0.5))
    return x.float().contiguous(), q.float().contiguous()


def _parameters(B, g):
    """(beta, theta): the workloads' values for one trajectory, per-trajectory ones for several."""
    if B == 1:
        return 20.0, 0.2
    return (10.0 + 30.0 * _uniform(g, B)).float(), (0.1 + 0.2 * _uniform(g, B)).float()


def _forcing_state(x, beta, theta):
    z = 0.5 + 0.3 * (0.5 * x[:, 2] + x[:, 0] * x[:, 1])
    return (theta + torch.log(z / (1.0 - z)) / beta).view(1, -1)


def _inputs(case, seed):
    """Everything but the library's own objects."""
    g = _gen(seed)
    if case["do"] == "setup":
        x, _, nrm, tris = _nodes(case["shape"], case["n"], g)
        return dict(x=x.contiguous(), nrm=None if nrm is None else nrm.contiguous(), tris=tris)
    if case["do"] == "grouped":
        s = dict(sets=[], u=[], beta=[], theta=[])
        for j, part in enumerate(case["sets"].split(",")):
            n, B = (int(v) for v in part.split("x"))
            x, q = _node_set("sphere" if j == 0 else "ellipsoid", n, g)
            s["sets"].append((x, q, B))
            s["u"].append(_bumps(x.double(), B, g).float().reshape(-1))
            s["beta"].append((10.0 + 30.0 * _uniform(g, B)).float())
            s["theta"].append((0.1 + 0.2 * _uniform(g, B)).float())
        for key in ("u", "beta", "theta"):
            s[key] = torch.cat(s[key])
        return s
    x, q = _node_set(case["shape"], case["n"], g)
    beta, theta = _parameters(case["B"], g)
    s = dict(x=x, q=q, beta=beta, theta=theta, forcing=None)
    if case.get("forcing") == "sphere":
        s["forcing"] = nf.Forcing.sphere()
        s["u"] = (_forcing_state(x.double(), beta, theta) + 1e-3 * (_uniform(g, 1, x.shape[0]) - 0.5)).float()
    elif case.get("forcing") == "flat":
        s["beta"], s["theta"], s["forcing"] = 5.0, 0.5, nf.Forcing.flat()
        xd = x.double()
        s["u"] = (_flat_solution(xd, 0.0)[0].view(1, -1) + 1e-3 * (_uniform(g, 1, x.shape[0]) - 0.5)).float()
    else:
        s["u"] = _bumps(x.double(), case["B"], g).float().contiguous()
    if case["do"] == "model":
        s["s"] = (1.0 - 0.3 * _uniform(g, case["B"], x.shape[0])).float()
    if case["do"] == "grad":
        s["target"] = _bumps(x.double(), case["B"], g).float().contiguous()
        s["kp"] = torch.tensor(_kernel(case)[:4], device=DEV, dtype=torch.float32)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    if case["do"] == "grouped":
        s["ops"] = [nf.Operator(x, q, _kernel(case), nf.DENSE_BF16X2) for x, q, _ in s["sets"]]
        s["op"] = nf.GroupedOperator(s["ops"], [B for _, _, B in s["sets"]])
    elif case["do"] not in ("setup", "grad"):
        s["op"] = nf.Operator(s["x"], s["q"], _kernel(case), PATHS[case["path"]])
    if case["do"] == "grad":
        s["u"].requires_grad_(True)
        s["kp"].requires_grad_(True)
    return s


# ---------------------------------------------------------------------------- the calls

def run(s):
    case = s["case"]
    do = case["do"]
    if do == "apply":
        return nf.nf_nonlocal_apply(s["op"], s["u"], s["beta"], s["theta"])
    if do in ("rk4", "grouped"):  # in place, as a time loop calls it
        return nf.nf_rk4_advance(s["op"], s["u"], 0.0, case["dt"], case["steps"], s["beta"], s["theta"],
                                 forcing=s.get("forcing"))
    if do == "model":
        nf.nf_field_advance(s["op"], s["u"], case["dt"], case["steps"], s["beta"], s["theta"], s=s["s"],
                            rate=nf.RATE_SMOOTHSTEP, tau=20.0, beta_d=0.5, integrator=case["integrator"])
        return {"u": s["u"], "s": s["s"]}
    if do == "grad":
        u = nf.NeuralFieldRK4.apply(s["u"], s["kp"], s["x"], s["q"], s["beta"], s["theta"], 0.0, case["dt"],
                                    case["steps"], case["every"])
        loss = (s["q"] * (u - s["target"]) ** 2).sum()
        gu, gk = torch.autograd.grad(loss, (s["u"], s["kp"]))
        return {"u": u.detach(), "grad_u0": gu, "grad_kernel": gk}
    stencils = nf.nf_build_stencils(s["x"], s["tris"], case["k"])
    return {"stencils": stencils, "q": nf.nf_quad_weights(s["x"], s["tris"], stencils, case["deg"], s["nrm"])}


def work(case):
    """Per sum: each unordered pair's distance and exponentials once (10 operations), two per
    ordered pair and trajectory; the stored matrix read once per sum on the dense paths."""
    do = case["do"]
    if do == "setup":
        n, m, k = case["n"], 2 * case["n"], case["k"]
        N = k + (case["deg"] + 1) * (case["deg"] + 2) // 2
        return {"bytes": n * (24 + 24 + 8) + m * 12 + m * k * 4, "flops": m * (2 * N ** 3 / 3 + 30 * k * k + 300 * k)}
    if do == "grouped":
        sets = [tuple(int(v) for v in part.split("x")) for part in case["sets"].split(",")]
        sums = 4 * case["steps"]
        return {"bytes": sum(sums * 4 * n * n + 8 * n * B for n, B in sets), "flops": sum(sums * 6 * n * n * B for n, B in sets)}
    n, B = case["n"], case["B"]
    if do == "grad":  # forward, its recomputation from the checkpoints, and the adjoint's sums
        sums = 4 * case["steps"]
        return {"bytes": 4 * n * (3 * B + 4) + 4 * n * B * (1 + case["steps"] // case["every"]),
                "flops": sums * n * n * (2 * (5 + 2 * B) + 5 + 10 * B)}
    sums = 1 if do == "apply" else 4 * case["steps"]
    if do == "model" and case["integrator"] == "ab5":
        sums = 16 + max(0, case["steps"] - 4)
    if case["path"] == "mf":
        return {"bytes": n * (16 + 8 * B), "flops": sums * n * n * (5 + 2 * B)}
    half = 0.5 if case["path"].startswith("sym") else 1.0
    return {"bytes": sums * 4 * half * n * n + 8 * n * B, "flops": sums * 2 * n * n * B}


# ---------------------------------------------------------------------------- in 64 bits

def _f32(v):
    return float(torch.tensor(v, dtype=torch.float32))


def _pair_terms(x, kernel, rows):
    """e1, e2 and r^2 of the given rows against all nodes, FP64."""
    _, s1, _, s2, per = kernel
    r2 = torch.zeros(len(rows), x.shape[0], device=DEV, dtype=torch.float64)
    for d in range(x.shape[1]):
        t = x[rows, d].view(-1, 1) - x[:, d].view(1, -1)
        if per > 0 and d < 2:
            t = t - per * torch.round(t / per)
        r2.add_(t * t)
    return torch.exp(r2 * (-1.0 / s1 ** 2)), torch.exp(r2 * (-1.0 / s2 ** 2)), r2


def _matrix(x, kernel):
    n = x.shape[0]
    W = torch.empty(n, n, device=DEV, dtype=torch.float64)
    step = max(1, int(2e8 // n))
    for a in range(0, n, step):
        rows = torch.arange(a, min(n, a + step), device=DEV)
        e1, e2, _ = _pair_terms(x, kernel, rows)
        W[a:a + step] = kernel[0] * e1 - kernel[2] * e2
    return W


def _times(W, g):
    """(W g_b) for every row b of g, W symmetric."""
    return torch.matmul(g, W) if g.shape[0] > 1 else torch.mv(W, g[0]).view(1, -1)


def _flat_solution(x, t, c=0.1, radius=0.2, sigma=1.1, L=2 * math.pi):
    """u* of the periodic square's manufactured solution, with z, its Gaussian and offsets."""
    x0 = (radius * math.cos(t), radius * math.sin(t))
    a = [x[:, d] - x0[d] - L * torch.round((x[:, d] - x0[d]) / L) for d in (0, 1)]
    G = torch.exp(-(a[0] ** 2 + a[1] ** 2) / (2 * sigma ** 2)) / (2 * math.pi * sigma ** 2)
    z = G + c
    return 0.5 + torch.log(z / (1 - z)) / 5.0, z, G, a


def _flat_forcing(x, t, kernel, c=0.1, radius=0.2, sigma=1.1, L=2 * math.pi):
    us, z, G, a = _flat_solution(x, t)
    dz = G * (a[0] * (-radius * math.sin(t)) + a[1] * (radius * math.cos(t))) / sigma ** 2
    dus = dz / (5.0 * z * (1 - z))
    A1, s1 = kernel[0], kernel[1]
    p, r = 1.0 / s1 ** 2, 1.0 / (2 * sigma ** 2)

    def piece(b, lo, hi):  # int_lo^hi exp(-p d^2 - r (d - b)^2) dd
        s = p + r
        m, k = r * b / s, math.sqrt(s)
        return torch.exp(-p * r * b * b / s) * 0.5 * math.sqrt(math.pi / s) * (torch.erf(k * (hi - m)) - torch.erf(k * (lo - m)))

    def factor(b):  # the nearest image of x0 changes where b - d leaves the cell
        h = torch.full_like(b, 0.5 * L)
        pos = piece(b - L, -h, b - h) + piece(b, b - h, h)
        neg = piece(b, -h, b + h) + piece(b + L, b + h, h)
        return torch.where(b >= 0, pos, neg)

    e = math.sqrt(math.pi) * s1 * math.erf(0.5 * L / s1)
    C = A1 * (c * e * e + factor(a[0]) * factor(a[1]) / (2 * math.pi * sigma ** 2))
    return (dus + us - C).view(1, -1)


def _sphere_forcing(x, t, kernel, beta, theta, c=0.5, a0=0.3):
    lam = [0.0, 0.0, 0.0]
    for amp, s in ((kernel[0], kernel[1]), (-kernel[2], kernel[3])):  # Funk-Hecke, in closed form
        a = 2.0 / s ** 2
        E = math.exp(-2 * a)
        I0 = -math.expm1(-2 * a) / a
        I1 = (1 + E) / a - I0 / a
        I2 = I0 - 2 * I1 / a
        lam = [lam[0] + amp * 2 * math.pi * I0, lam[1] + amp * 2 * math.pi * I1,
               lam[2] + amp * math.pi * (3 * I2 - I0)]
    Y1, Y2 = 0.5 * x[:, 2], x[:, 0] * x[:, 1]
    a, da = a0 * math.cos(t), -a0 * math.sin(t)
    z = c + a * (Y1 + Y2)
    us = theta + torch.log(z / (1 - z)) / beta
    dus = da * (Y1 + Y2) / (beta * z * (1 - z))
    return (dus + us - (lam[0] * c + a * (lam[1] * Y1 + lam[2] * Y2))).view(1, -1)


def _smooth_step(u, a=0.06, b=0.54):
    a, b = _f32(a), _f32(b)
    t = ((u - a) / (b - a)).clamp(0.0, 1.0)
    return t ** 5 * (126.0 - 420.0 * t + 540.0 * t ** 2 - 315.0 * t ** 3 + 70.0 * t ** 4)


def _rk4(u, f, t, dt, steps, keep=None):
    for j in range(steps):
        t0, v, acc = t + j * dt, u, 0.0
        for c, b in ((0.0, 1.0), (0.5, 2.0), (0.5, 2.0), (1.0, 1.0)):
            U = u if c == 0.0 else [p + c * dt * k for p, k in zip(u, v)]
            if keep is not None:
                keep.append(U[0])
            v = f(t0 + c * dt, U)
            acc = [b * k for k in v] if b == 1.0 and c == 0.0 else [p + b * k for p, k in zip(acc, v)]
        u = [p + dt / 6.0 * k for p, k in zip(u, acc)]
    return u


def exact(case, seed):
    s = _inputs(case, seed)
    do = case["do"]
    if do == "setup":
        return {"stencils": None, "q": _exact_weights(s, case["k"], case["deg"])}
    kernel = tuple(_f32(v) for v in _kernel(case))
    col = lambda v: (v.double().view(-1, 1) if isinstance(v, torch.Tensor) else float(v))  # noqa: E731
    if do == "grouped":
        out, at, tr = [], 0, 0
        for x, q, B in s["sets"]:
            n = x.shape[0]
            W = _matrix(x.double(), kernel)
            beta, theta = col(s["beta"][tr:tr + B]), col(s["theta"][tr:tr + B])
            rhs = lambda t, U, W=W, q=q.double(), be=beta, th=theta: [  # noqa: E731
                -U[0] + _times(W, q * torch.sigmoid(be * (U[0] - th)))]
            u = s["u"][at:at + n * B].double().view(B, n)
            out.append(_rk4([u], rhs, 0.0, case["dt"], case["steps"])[0].reshape(-1))
            at, tr = at + n * B, tr + B
            del W, rhs
        return torch.cat(out)
    x, q, u = s["x"].double(), s["q"].double(), s["u"].double()
    beta, theta = col(s["beta"]), col(_f32(s["theta"]) if isinstance(s["theta"], float) else s["theta"])
    if do == "grad":
        return _exact_gradient(case, s, x, q, u, beta, theta, kernel)
    W = _matrix(x, kernel)
    if do == "apply":
        return _times(W, q * torch.sigmoid(beta * (u - theta)))
    if do == "model":
        ss = s["s"].double()
        tau, bd, dt = 20.0, 0.5, case["dt"]

        def field(t, U):
            f = _smooth_step(U[0])
            return [-U[0] + _times(W, q * U[1] * f), (1.0 - U[1] - bd * U[1] * f) / tau]

        if case["integrator"] == "rk4":
            y = _rk4([u, ss], field, 0.0, dt, case["steps"])
            return {"u": y[0], "s": y[1]}
        y, hist = [u, ss], []
        for j in range(case["steps"]):
            hist.append(field(0.0, y))
            if j < 4:
                y = _rk4(y, field, 0.0, dt, 1)
                continue
            w = [1901 / 720, -2774 / 720, 2616 / 720, -1274 / 720, 251 / 720]
            y = [y[i] + dt * sum(w[k] * hist[j - k][i] for k in range(5)) for i in (0, 1)]
        return {"u": y[0], "s": y[1]}

    def rhs(t, U):
        v = -U[0] + _times(W, q * torch.sigmoid(beta * (U[0] - theta)))
        if case.get("forcing") == "sphere":
            v = v + _sphere_forcing(x, t, kernel, beta, theta)
        elif case.get("forcing") == "flat":
            v = v + _flat_forcing(x, t, kernel)
        return [v]

    return _rk4([u], rhs, 0.0, case["dt"], case["steps"])[0]


def _exact_gradient(case, s, x, q, u, beta, theta, kernel):
    """The discrete adjoint of the RK4 steps: nu_s are the stages' cotangents."""
    A1, s1, A2, s2, _ = kernel
    n, dt = x.shape[0], case["dt"]
    W = _matrix(x, kernel)
    f = lambda U: torch.sigmoid(beta * (U - theta))  # noqa: E731
    stages = []
    uT = _rk4([u], lambda t, U: [-U[0] + _times(W, q * f(U[0]))], 0.0, dt, case["steps"], keep=stages)[0]
    lam = 2.0 * q * (uT - s["target"].double())
    nus, gs = [], []  # cotangents and firing rates of every stage, for the kernel's gradient
    b, c = (1 / 6, 1 / 3, 1 / 3, 1 / 6), (0.5, 0.5, 1.0)
    for j in reversed(range(case["steps"])):
        mu, add = None, 0.0
        for st in (3, 2, 1, 0):
            nu = dt * b[st] * lam + (0.0 if mu is None else c[st] * dt * mu)
            F = f(stages[4 * j + st])
            mu = -nu + q * beta * F * (1 - F) * _times(W, nu)
            add = add + mu
            nus.append(nu)
            gs.append(q * F)
        lam = lam + add
    del W
    N, Gm = torch.cat(nus), torch.cat(gs)  # (stages * B) x n
    gk = torch.zeros(4, device=DEV, dtype=torch.float64)
    step = max(1, int(1e8 // n))
    for a in range(0, n, step):  # sum over pairs of nu_i g_j against each derivative of w
        rows = torch.arange(a, min(n, a + step), device=DEV)
        e1, e2, r2 = _pair_terms(x, kernel, rows)
        P = torch.matmul(N[:, rows].t(), Gm)
        e1.mul_(P)
        e2.mul_(P)
        gk += torch.stack([e1.sum(), 2 * A1 / s1 ** 3 * (e1 * r2).sum(), -e2.sum(), -2 * A2 / s2 ** 3 * (e2 * r2).sum()])
    return {"u": uT, "grad_u0": lam, "grad_kernel": gk}


def _exact_weights(s, k, deg):
    """RBF quadrature weights (§3.1-3.3), element by element in batches."""
    x, tris = s["x"], s["tris"].long()
    n, dim, m = x.shape[0], x.shape[1], tris.shape[0]
    normal = nbr = None
    if dim == 3:
        A, B, C = (x[tris[:, i]] for i in range(3))
        normal = torch.linalg.cross(B - A, C - A)
        normal = normal / normal.norm(dim=1, keepdim=True)
        ref = sum(s["nrm"][tris[:, i]] for i in range(3))
        normal = torch.where((normal * ref).sum(1, keepdim=True) < 0, -normal, normal)
        ends = torch.stack([tris, tris.roll(-1, 1)], -1).reshape(-1, 2)  # edge 3 e + i: vertices i, i + 1
        key = ends.min(1).values * n + ends.max(1).values
        order = torch.argsort(key)  # closed surface: the two elements of an edge follow each other
        other = torch.empty_like(order)
        other[order[0::2]], other[order[1::2]] = order[1::2], order[0::2]
        nbr = (other // 3).view(m, 3)
    q = torch.zeros(n, device=DEV, dtype=torch.float64)
    step = max(1, int(4e8 // n))
    for a in range(0, m, step):
        T = tris[a:a + step]
        c = (x[T[:, 0]] + x[T[:, 1]] + x[T[:, 2]]) / 3.0
        d2 = sum((c[:, d].view(-1, 1) - x[:, d].view(1, -1)) ** 2 for d in range(dim))
        S = torch.topk(d2, k, dim=1, largest=False).indices
        del d2
        X, V = x[S], x[T]
        jac = torch.ones(S.shape, device=DEV, dtype=torch.float64)
        if dim == 2:
            xi, tv = X - c.unsqueeze(1), V - c.unsqueeze(1)
        else:
            nE = normal[a:a + step]
            dn = nE.unsqueeze(1) - normal[nbr[a:a + step]]  # the three cutting planes
            rhs = (dn * V).sum(-1)
            inv = torch.linalg.inv_ex(dn).inverse
            cond = dn.abs().sum(2).max(1).values * inv.abs().sum(2).max(1).values
            central = (torch.isfinite(cond) & (cond < 1e10)).view(-1, 1)
            p = torch.nan_to_num(torch.matmul(inv, rhs.unsqueeze(-1)).squeeze(-1))
            xp = X - p.unsqueeze(1)
            t = ((c - p) * nE).sum(1).view(-1, 1) / (xp * nE.unsqueeze(1)).sum(-1)
            un = xp / xp.norm(dim=2, keepdim=True)
            ns = s["nrm"][S]
            jc = (nE.unsqueeze(1) * un).sum(-1).abs() / (ns * un).sum(-1).abs() / t ** 2
            jp = 1.0 / (ns * nE.unsqueeze(1)).sum(-1).abs()
            flat = X - ((X - c.unsqueeze(1)) * nE.unsqueeze(1)).sum(-1, keepdim=True) * nE.unsqueeze(1)
            Y = torch.where(central.unsqueeze(-1), p.unsqueeze(1) + xp * t.unsqueeze(-1), flat)
            jac = torch.where(central, jc, jp)
            e1 = V[:, 1] - V[:, 0]
            e1 = e1 / e1.norm(dim=1, keepdim=True)
            frame = torch.stack([e1, torch.linalg.cross(nE, e1)], 2)  # columns e1, e2
            xi, tv = torch.matmul(Y - c.unsqueeze(1), frame), torch.matmul(V - c.unsqueeze(1), frame)
        rho = xi.norm(dim=2).max(1).values.view(-1, 1, 1)
        xi, tv = xi / rho, tv / rho
        pw = [(i, t - i) for t in range(deg + 1) for i in range(t, -1, -1)]
        P = torch.stack([xi[..., 0] ** i * xi[..., 1] ** j for i, j in pw], 2)
        Phi = (xi.unsqueeze(2) - xi.unsqueeze(1)).norm(dim=3) ** 3
        M = torch.cat([torch.cat([Phi, P], 2),
                       torch.cat([P.transpose(1, 2), torch.zeros(len(T), len(pw), len(pw), device=DEV, dtype=torch.float64)], 2)], 1)
        z = torch.cat([_cubic_integrals(xi, tv), torch.stack([_monomial_integral(i, j, tv) for i, j in pw], 1)], 1)
        w = torch.linalg.solve(M, z.unsqueeze(-1)).squeeze(-1)[:, :k] * rho.view(-1, 1) ** 2 * jac
        q.index_add_(0, S.reshape(-1), w.reshape(-1))
    return q


def _cubic_integrals(xi, tv):
    """int_T |x - p|^3 for every stencil point p: signed fan of three wedges."""
    det = (tv[:, 1, 0] - tv[:, 0, 0]) * (tv[:, 2, 1] - tv[:, 0, 1]) - (tv[:, 1, 1] - tv[:, 0, 1]) * (tv[:, 2, 0] - tv[:, 0, 0])
    total = 0.0
    for e in range(3):
        A, B = tv[:, e].unsqueeze(1), tv[:, (e + 1) % 3].unsqueeze(1)
        L = (B - A).norm(dim=2, keepdim=True)
        t = (B - A) / L
        v = A - xi
        cr = v[..., 0] * t[..., 1] - v[..., 1] * t[..., 0]
        d = cr.abs().clamp_min(1e-300)
        a = (v * t).sum(-1)

        def wedge(a, d):
            rr = (a * a + d * d).sqrt()
            return 0.25 * d * a * rr ** 3 + 0.375 * d ** 3 * a * rr + 0.375 * d ** 5 * torch.asinh(a / d)

        total = total + torch.sign(cr) * (wedge(a + L[..., 0], d) - wedge(a, d)) / 5.0
    return torch.where(det.view(-1, 1) > 0, total, -total)


def _monomial_integral(a, b, tv):
    """int_T x^a y^b by the barycentric expansion."""
    det = (tv[:, 1, 0] - tv[:, 0, 0]) * (tv[:, 2, 1] - tv[:, 0, 1]) - (tv[:, 1, 1] - tv[:, 0, 1]) * (tv[:, 2, 0] - tv[:, 0, 0])
    F = math.factorial
    total = torch.zeros_like(det)
    for i0 in range(a + 1):
        for i1 in range(a + 1 - i0):
            i2 = a - i0 - i1
            cx = F(a) / (F(i0) * F(i1) * F(i2)) * tv[:, 0, 0] ** i0 * tv[:, 1, 0] ** i1 * tv[:, 2, 0] ** i2
            for j0 in range(b + 1):
                for j1 in range(b + 1 - j0):
                    j2 = b - j0 - j1
                    cy = F(b) / (F(j0) * F(j1) * F(j2)) * tv[:, 0, 1] ** j0 * tv[:, 1, 1] ** j1 * tv[:, 2, 1] ** j2
                    total = total + cx * cy * (F(i0 + j0) * F(i1 + j1) * F(i2 + j2) / F(a + b + 2))
    return total * det.abs()
