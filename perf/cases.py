"""The work that users of this library have it do, as measurable cases.

Every case goes through the package's public entry points on the inputs a
user's program has in hand: a plan with its contrast, device vectors, network
weights.  Kinds:

  operator     one application y = w - M (N w) on one grid (vie_matvec)
  batch        one application on several uneven guides (vie_matvec_batch)
  jm_operator  one application of the JM-VIE operator (vie_jm_matvec)
  setup        one wavelength of a sweep: plan, contrast, right-hand side
  solve        one problem to a tight residual in mixed precision, plain or
               with the block-circulant preconditioner built for it
  net_apply    the learned preconditioner applied to one vector
  net_train    gradients of the network over a mini-batch of training pairs

`exact` restates each result in 64-bit torch from the method's formulas: the
Galerkin entries by Gauss and Duffy quadrature, the operator by padded FFTs,
the solution by unrestarted GMRES, the network by torch's convolutions.
"""
import math

import numpy as np
import torch

from paper_1803_06237_gb300 import vie

EPS_CORE = 12.11          # silicon strip
EPS_BG = 2.085            # silica around it
R_RT = 1e-10              # round-trip reflection the absorbers are designed for
TOL = 1e-11               # solves: tight enough that two correct solves agree

# (name, input channels, output channels) of the network's 3x3x3 convolutions,
# in the order of its parameter array (weights [out][in][27], then biases)
LAYERS = [("enc0", 8, 32), ("enc1", 32, 32), ("enc2", 32, 32), ("enc3", 32, 32),
          ("dec2", 32, 32), ("dec1", 32, 32), ("dec0", 32, 32), ("out", 32, 6)]


def listed():
    return [
        # the smallest call: the 12^3 dielectric cube, where launches and latency count
        dict(name="op_cube_c64", kind="operator", shape="cube", nx=12, ny=12, nz=12, dtype="c64"),
        # the benchmark's 12 um strip guide: the inner operator of every mixed-precision step
        dict(name="op_guide_c64", kind="operator", shape="strip", nx=600, ny=23, nz=11, dtype="c64"),
        # the 100-period Bragg grating of the transmission study: a long guide of another cross-section
        dict(name="op_grating_c64", kind="operator", shape="grating", nx=2030, ny=27, nz=11, dtype="c64"),
        # the ring resonator beside a bus: the largest operator, vectors far beyond L2
        dict(name="op_ring_c64", kind="operator", shape="ring", nx=800, ny=600, nz=11, dtype="c64"),
        # the true residual of mixed refinement and the operator of plain FP64 GMRES
        dict(name="op_guide_c128", kind="operator", shape="strip", nx=600, ny=23, nz=11, dtype="c128"),
        # the absorber batch: guides of six lengths with two absorbers each in one call
        dict(name="op_batch12_c64", kind="batch", nx=300, step=100, ny=23, nz=11, lengths=6, each=2, dtype="c64"),
        # the matched-loss absorber study: electric and magnetic currents on a 500 x 200 nm strip
        dict(name="jm_strip_c64", kind="jm_operator", shape="strip", nx=396, ny=30, nz=12, dtype="c64"),
        # one wavelength's setup in a spectrum sweep (every wavelength needs its own plan)
        dict(name="setup_guide", kind="setup", shape="strip", nx=600, ny=23, nz=11),
        # the benchmark's solve: plain GMRES(30) inside refinement
        dict(name="solve_guide", kind="solve", shape="strip", nx=600, ny=23, nz=11, precondition=False),
        # one point of the absorber study: preconditioner built, then a preconditioned solve
        dict(name="solve_strip_circulant", kind="solve", shape="strip", nx=396, ny=30, nz=12, precondition=True),
        # one preconditioner application inside flexible GMRES
        dict(name="net_apply_guide", kind="net_apply", shape="strip", nx=600, ny=23, nz=11, dtype="c64"),
        # the gradients of one mini-batch of the preconditioner's training on short random guides
        dict(name="net_train_160", kind="net_train", shape="grating", nx=160, ny=40, nz=11, samples=4),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["operator", "operator", "operator", "batch", "jm_operator", "setup", "solve", "net_apply",
                       "net_train"])
    if kind == "operator" and rng.random() < 0.25:       # planes: rings, couplers
        return dict(kind=kind, shape="ring", nx=log(120, 800), ny=log(90, 600), nz=rng.randint(6, 12), dtype="c64")
    if kind == "operator":
        dtype = rng.choice(["c64", "c64", "c128"])
        return dict(kind=kind, shape=rng.choice(["strip", "grating"]), nx=log(20, 2000 if dtype == "c64" else 700),
                    ny=rng.randint(9, 34), nz=rng.randint(6, 14), dtype=dtype)
    if kind == "batch":
        return dict(kind=kind, nx=rng.randint(150, 400), step=rng.randint(20, 80), ny=rng.choice([23, 27, 30]),
                    nz=rng.choice([11, 12]), lengths=rng.randint(2, 6), each=rng.randint(1, 4), dtype="c64")
    if kind == "jm_operator":
        return dict(kind=kind, shape="strip", nx=log(60, 500), ny=rng.randint(10, 32), nz=rng.randint(6, 12),
                    dtype="c64")
    if kind == "setup":
        return dict(kind=kind, shape=rng.choice(["strip", "grating"]), nx=log(80, 1200), ny=rng.randint(10, 34),
                    nz=rng.randint(6, 14))
    if kind == "solve":
        ny, nz = rng.choice([(23, 11), (27, 11), (30, 12), (21, 10)])
        pre = rng.random() < 0.5
        return dict(kind=kind, shape="strip", nx=rng.randint(150, 400 if pre else 500), ny=ny, nz=nz, precondition=pre)
    if kind == "net_apply":
        return dict(kind=kind, shape="strip", nx=log(80, 700), ny=rng.randint(16, 40), nz=rng.randint(5, 12),
                    dtype=rng.choice(["c64", "c64", "c128"]))
    return dict(kind=kind, shape="grating", nx=rng.randint(80, 240), ny=rng.randint(20, 48), nz=rng.randint(6, 12),
                samples=rng.randint(1, 6))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _rng(case, seed):
    return np.random.default_rng([int(seed) % (1 << 31), case["nx"], case["ny"], case["nz"]])


def _physics(case, rng):
    """(voxel size um, free-space wavenumber 1/um, background permittivity): the
    seed picks a wavelength of the telecom window, as a sweep does."""
    k0 = 2 * math.pi / rng.uniform(1.52, 1.57)
    if case.get("shape") == "cube":
        return 0.4 / case["nx"], k0, 1.0
    return 0.02, k0, EPS_BG


def _structure(case):
    """Relative permittivity per voxel, (nz, ny, nx)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape = case.get("shape", "strip")
    if shape == "cube":
        return np.full((nz, ny, nx), 12.25 + 0j)
    core = np.ones((ny, nx), bool)
    if shape == "grating":                   # one voxel narrower on each side every other half period
        narrow = (np.arange(nx) % 16) >= 8
        core[:1, narrow] = False
        core[-1:, narrow] = False
    elif shape == "ring":                    # a bus along x and a ring beside it
        X, Y = np.meshgrid(np.arange(nx) + 0.5, np.arange(ny) + 0.5)
        w, gap, yb = 22.5, 10.0, 20.0
        R = max(10.0, min(0.5 * (ny - yb - gap - 1.5 * w), 0.45 * nx))
        core = (np.abs(Y - yb) <= w / 2) | (np.abs(np.hypot(X - nx / 2, Y - (yb + w + gap + R)) - R) <= w / 2)
    eps = np.full((nz, ny, nx), EPS_BG + 0j)
    eps[:, core] = EPS_CORE
    return eps


def _absorbers(case, h, k0, degree=2):
    """Graded loss over the last third of a guide, over both ends of a ring's bus."""
    nx = case["nx"]
    if case.get("shape") == "cube":
        return []
    L = float(max(1, nx // (4 if case.get("shape") == "ring" else 3)))
    e2 = -(degree + 1) * math.log(R_RT) * math.sqrt(EPS_CORE) / (2.0 * L * h * k0)
    out = [dict(x0=nx - L, length=L, degree=degree, eps2_max=e2, direction=1)]
    if case.get("shape") == "ring":
        out.append(dict(x0=L, length=L, degree=degree, eps2_max=e2, direction=-1))
    return out


def _normal(rng, shape, dtype="c128"):
    v = torch.from_numpy(rng.standard_normal(shape + (2,))).cuda()
    return torch.view_as_complex(v).to(torch.complex64 if dtype == "c64" else torch.complex128)


def _incident(case, rng, h, k0):
    """A y-polarised Gaussian wave packet that enters the guide 1 um from its left end, (3, nz, ny, nx)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    kappa = k0 * math.sqrt(EPS_CORE) * h
    x, y, z = np.arange(nx) + 0.5, np.arange(ny) + 0.5 - ny / 2, np.arange(nz) + 0.5 - nz / 2
    y0, z0 = rng.uniform(-2, 2), rng.uniform(-1, 1)
    prof = np.exp(-((y[None, :, None] - y0) ** 2 + (z[:, None, None] - z0) ** 2) / 10.0 ** 2)
    e = np.zeros((3, nz, ny, nx), complex)
    e[1] = prof * (np.exp(-((x - 50.0) / 8.0) ** 2 - 1j * kappa * x))[None, None, :]
    return e


def _problem(case, seed):
    """What plan and contrast are made from: rng, h, k0, eps_bg, permittivity, absorbers."""
    rng = _rng(case, seed)
    h, k0, eps_bg = _physics(case, rng)
    return rng, h, k0, eps_bg, _structure(case), _absorbers(case, h, k0)


def _chi(case, eps, absorbers, eps_bg):
    nx = case["nx"]
    e2 = np.zeros(nx)
    for a in absorbers:
        u = a["direction"] * (np.arange(nx) + 0.5 - a["x0"]) / a["length"]
        inside = (u >= 0) & (u <= 1)
        e2[inside] += a["eps2_max"] * u[inside] ** a["degree"]
    return (eps - 1j * (np.abs(eps - eps_bg) > 0) * e2) / eps_bg - 1.0


def _net_params(rng):
    """A network as training leaves it: He-sized weights, small biases, an output
    layer whose correction is a fraction of its input."""
    out = []
    for name, ci, co in LAYERS:
        std = math.sqrt(2.0 / (27 * ci)) * (0.3 if name == "out" else 1.0)
        out += [rng.standard_normal(co * ci * 27) * std, rng.standard_normal(co) * 0.01]
    return np.concatenate(out).astype(np.float32)


def _pair(case, rng, shape):
    """One training pair: an error and a residual correlated with it (planar complex64)."""
    e = _normal(rng, shape)
    return (0.7 * e + 0.5 * _normal(rng, shape)).to(torch.complex64), e.to(torch.complex64)


def _guides(case):
    """The grids of a batch: `lengths` lengths, `each` guides of every length."""
    return [dict(case, shape="strip", nx=case["nx"] + case["step"] * i) for i in range(case["lengths"])
            for _ in range(case["each"])]


def _batch_problem(case, seed):
    """Per guide: x length, absorber degree, its vector; one wavelength for the batch."""
    rng = _rng(case, seed)
    h, k0, eps_bg = _physics(case, rng)
    out = []
    for i, g in enumerate(_guides(case)):
        out.append((g, _structure(g), _absorbers(g, h, k0, degree=i % case["each"] + 1),
                    _normal(rng, (3, g["nz"], g["ny"], g["nx"]), case["dtype"])))
    return h, k0, eps_bg, out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        h, k0, eps_bg, guides = _batch_problem(case, seed)
        plans, base = [], None
        for g, eps, absorbers, _ in guides:
            if base is not None and base.n[0] == g["nx"]:
                plan = vie.vie_plan_clone(base)
            else:
                plan = base = vie.vie_plan_create((g["nx"], g["ny"], g["nz"]), h, k0, eps_bg)
            vie.vie_set_permittivity(plan, eps, absorbers)
            plans.append(plan)
        xs = [x.reshape(-1) for *_, x in guides]
        return dict(kind=kind, plans=plans, xs=xs, ys=[torch.empty_like(x) for x in xs])

    rng, h, k0, eps_bg, eps, absorbers = _problem(case, seed)
    grid = (case["nx"], case["ny"], case["nz"])
    shape = (case["nz"], case["ny"], case["nx"])
    if kind == "setup":
        return dict(kind=kind, grid=grid, h=h, k0=k0, eps_bg=eps_bg, eps=eps, absorbers=absorbers,
                    src=_normal(rng, (3,) + shape).reshape(-1))
    plan = vie.vie_plan_create(grid, h, k0, eps_bg)
    vie.vie_set_permittivity(plan, eps, absorbers)
    if kind == "operator":
        x = _normal(rng, (3,) + shape, case["dtype"]).reshape(-1)
        return dict(kind=kind, plan=plan, x=x, y=torch.empty_like(x))
    if kind == "jm_operator":
        vie.vie_set_permeability(plan)
        x = _normal(rng, (6,) + shape, case["dtype"]).reshape(-1)
        return dict(kind=kind, plan=plan, x=x, y=torch.empty_like(x))
    if kind == "solve":
        chi = _chi(case, eps, absorbers, eps_bg)
        b = (chi / (1 + chi))[None] * _incident(case, rng, h, k0)
        b = torch.from_numpy(b.reshape(-1)).cuda()
        return dict(kind=kind, plan=plan, b=b, x=torch.zeros_like(b), precondition=case["precondition"])
    net = vie.vie_net_create(_net_params(rng))
    if kind == "net_apply":
        x = _normal(rng, (3,) + shape, case["dtype"]).reshape(-1)
        return dict(kind=kind, plan=plan, net=net, x=x, y=torch.empty_like(x))
    pairs = [tuple(t.reshape(-1) for t in _pair(case, rng, (3,) + shape)) for _ in range(case["samples"])]
    return dict(kind=kind, plan=plan, net=net, pairs=pairs)


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "operator":
        return vie.vie_matvec(s["plan"], s["x"], s["y"])
    if kind == "batch":
        vie.vie_matvec_batch(s["plans"], s["xs"], s["ys"])
        return s["ys"]
    if kind == "jm_operator":
        vie.vie_jm_matvec(s["plan"], s["x"], s["y"])
        return s["y"]
    if kind == "setup":
        plan = vie.vie_plan_create(s["grid"], s["h"], s["k0"], s["eps_bg"])
        vie.vie_set_permittivity(plan, s["eps"], s["absorbers"])
        b = torch.empty_like(s["src"])
        vie.vie_rhs_from_source(plan, s["src"], b)
        plan.close()
        return b
    if kind == "solve":
        if not s["precondition"]:
            vie.vie_solve(s["plan"], s["b"], s["x"], TOL, mode=vie.VIE_SOLVE_MIXED, restart=30)
            return s["x"]
        c = vie.vie_circulant_create(s["plan"], vie.VIE_CIRC_FP16_FACTORS)
        vie.vie_set_circulant_preconditioner(s["plan"], c)
        vie.vie_solve(s["plan"], s["b"], s["x"], TOL, mode=vie.VIE_SOLVE_MIXED, restart=30, use_preconditioner=True)
        vie.vie_set_circulant_preconditioner(s["plan"], None)
        c.close()
        return s["x"]
    if kind == "net_apply":
        return vie.vie_net_apply(s["net"], s["plan"], s["x"], s["y"])
    vie.vie_net_zero_grad(s["net"])
    losses = [vie.vie_net_accumulate(s["net"], s["plan"], r, e) for r, e in s["pairs"]]
    return dict(losses=losses, grads=vie.vie_net_get_grads(s["net"]))


# --------------------------------------------------------------------------
# the work a pass cannot do without
# --------------------------------------------------------------------------
def _operator_work(nx, ny, nz, es, currents=1):
    """Vectors in and out, contrast and the octant of the spectrum once; 5 L log2 L
    flops per FFT line that carries data on the doubled grid, the 3x3 products."""
    N = nx * ny * nz
    X, Y, Z = 2 * nx, 2 * ny, 2 * nz
    lines = 3 * ny * nz * 5 * X * math.log2(X) + X * (3 * ny * 5 * Z * math.log2(Z) + 3 * Z * 5 * Y * math.log2(Y))
    flops = currents * (2 * lines + 72 * X * Y * Z) + (96 * X * Y * Z if currents == 2 else 0)
    return {"bytes": es * N * (6 * currents + currents + 6 + (3 if currents == 2 else 0)), "flops": flops}


def _net_flops(nx, ny, nz):
    vox = [nx * ny * nz]
    for _ in range(3):
        nx, ny = (nx + 1) // 2, (ny + 1) // 2
        vox.append(nx * ny * nz)
    level = dict(enc0=0, enc1=1, enc2=2, enc3=3, dec2=2, dec1=1, dec0=0, out=0)
    return sum(2 * 27 * ci * co * vox[level[n]] for n, ci, co in LAYERS)


def work(case):
    kind, nx, ny, nz = case["kind"], case["nx"], case["ny"], case["nz"]
    N = nx * ny * nz
    es = 8 if case.get("dtype", "c128") == "c64" else 16
    if kind == "operator":
        return _operator_work(nx, ny, nz, es)
    if kind == "jm_operator":
        return _operator_work(nx, ny, nz, es, currents=2)
    if kind == "batch":
        each = [_operator_work(g["nx"], ny, nz, es) for g in _guides(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if kind == "setup":
        # permittivity and source in, right-hand side out; six FFTs of the embedded entries
        return {"bytes": 16 * 7 * N, "flops": 6 * 5 * 8 * N * math.log2(8 * N) + _operator_work(nx, ny, nz, 16)["flops"]}
    if kind == "solve":
        # about two GMRES(30) steps per voxel of length, or 60 preconditioned ones: an operator, half the
        # basis read for the products and again for the update
        steps = 60 if case["precondition"] else 2 * nx
        op = _operator_work(nx, ny, nz, 8)
        w = {"bytes": steps * (op["bytes"] + 2 * 15 * 3 * N * 8), "flops": steps * (op["flops"] + 16 * 15 * 3 * N)}
        if case["precondition"]:
            n = 3 * ny * nz
            w["bytes"] += steps * nx * n * n * 4
            w["flops"] += nx * (8 / 3) * n ** 3 + steps * nx * n * n * 8
        return w
    if kind == "net_apply":
        return {"bytes": 6 * N * es + 16 * N, "flops": _net_flops(nx, ny, nz)}
    return {"bytes": case["samples"] * (6 * N * 8 + 16 * N), "flops": 3 * case["samples"] * _net_flops(nx, ny, nz)}


# --------------------------------------------------------------------------
# the results in 64 bits
# --------------------------------------------------------------------------
def _gauss(q):
    x, w = np.polynomial.legendre.leggauss(q)
    return 0.5 * (x + 1), 0.5 * w


def _green(r, kappa):
    return torch.exp(-1j * kappa * r) / (4 * math.pi * r)


def _near(D, kappa, q=20):
    """Entries of T (six) and C (three) for an offset D in {0, 1}^3: derivatives moved
    onto the tents, the unit cells at the origin by Duffy's map."""
    x, w = _gauss(q)
    T1, U1, V1 = (a.ravel() for a in np.meshgrid(x, x, x, indexing="ij"))
    W3 = np.multiply.outer(np.multiply.outer(w, w), w).ravel()
    tent = lambda t: np.maximum(0.0, 1 - np.abs(t))  # noqa: E731
    V = S = 0.0
    C = np.zeros(3, complex)
    S = np.zeros(3, complex)                                         # xy, xz, yz
    green = lambda r: np.exp(-1j * kappa * r) / (4 * np.pi * r)      # noqa: E731
    for cell in np.ndindex(2, 2, 2):
        c0 = np.array(D) - 1 + np.array(cell)
        if np.all((c0 == 0) | (c0 == -1)):
            parts = []
            for a in range(3):
                u = np.empty((3, T1.size))
                u[a], u[(a + 1) % 3], u[(a + 2) % 3] = T1, T1 * U1, T1 * V1
                parts.append((np.where(c0[:, None] == -1, -u, u), W3 * T1 ** 2))
        else:
            parts = [(c0[:, None] + np.stack([T1, U1, V1]), W3)]
        for v, wt in parts:
            g = green(np.sqrt((v ** 2).sum(0))) * wt
            rel = v - np.array(D)[:, None]
            L, s = tent(rel), np.sign(rel)
            V = V + np.sum(g * L[0] * L[1] * L[2])
            S += [np.sum(g * s[0] * s[1] * L[2]), np.sum(g * s[0] * s[2] * L[1]), np.sum(g * s[1] * s[2] * L[0])]
            C += [np.sum(g * s[0] * L[1] * L[2]), np.sum(g * L[0] * s[1] * L[2]), np.sum(g * L[0] * L[1] * s[2])]
    T2, U2 = (a.ravel() for a in np.meshgrid(x, x, indexing="ij"))
    W2 = np.multiply.outer(w, w).ravel()
    diag = []
    for p in range(3):
        a, b = (p + 1) % 3, (p + 2) % 3
        F = []
        for t in (D[p] - 1, D[p], D[p] + 1):
            total = 0.0
            for sq in np.ndindex(2, 2):
                ca, cb = D[a] - 1 + sq[0], D[b] - 1 + sq[1]
                if t == 0 and ca in (0, -1) and cb in (0, -1):
                    parts = [(T2, T2 * U2, W2 * T2), (T2 * U2, T2, W2 * T2)]
                    parts = [(-u if ca == -1 else u, -v if cb == -1 else v, wt) for u, v, wt in parts]
                else:
                    parts = [(ca + T2, cb + U2, W2)]
                for va, vb, wt in parts:
                    total = total + np.sum(green(np.sqrt(t * t + va ** 2 + vb ** 2)) * wt * tent(va - D[a]) * tent(vb - D[b]))
            F.append(total)
        diag.append((1.0 if not any(D) else 0.0) + kappa ** 2 * V + F[2] - 2 * F[1] + F[0])
    C[[i for i in range(3) if D[i] == 0]] = 0
    return np.array(diag + list(S)), C


def _entries(n, kappa, curl=False):
    """Octant tables of T (6, nz, ny, nx) and, with curl, of C (3, nz, ny, nx), on the GPU:
    tent-weighted Gauss quadrature of the closed-form kernels, near offsets apart."""
    nx, ny, nz = n
    N = nx * ny * nz
    out = torch.zeros((9 if curl else 6, N), dtype=torch.complex128, device="cuda")
    idx = torch.arange(N, device="cuda")
    D = torch.stack([idx % nx, (idx // nx) % ny, idx // (nx * ny)]).double()
    cheb = D.amax(0)
    for lo, hi, q in ((2, 4, 16), (4, 10, 9), (10, 1e9, 5)):
        x, w = _gauss(q)
        t1, w1 = np.concatenate([x - 1, x]), np.concatenate([w * x, w * (1 - x)])
        P = torch.from_numpy(np.stack([a.ravel() for a in np.meshgrid(t1, t1, t1, indexing="ij")])).cuda()
        W = torch.from_numpy(np.multiply.outer(np.multiply.outer(w1, w1), w1).ravel()).cuda()
        sel = torch.nonzero((cheb >= lo) & (cheb < hi)).reshape(-1)
        for at in torch.split(sel, max(1, 16_000_000 // W.numel())):
            v = [D[a, at][:, None] + P[a][None] for a in range(3)]
            r2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2]
            r = torch.sqrt(r2)
            g = _green(r, kappa) * W
            kr = kappa * r
            A = g * torch.complex(kr * kr - 1, -kr) / r2
            B = g * torch.complex(3 - kr * kr, 3 * kr) / (r2 * r2)
            for c, (p, s) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
                val = B * (v[p] * v[s])
                out[c, at] = (val + A if p == s else val).sum(1)
            if curl:
                G = -g * torch.complex(torch.ones_like(kr), kr) / r2
                for a in range(3):
                    out[6 + a, at] = (G * v[a]).sum(1)
    for Dz in range(min(2, nz)):
        for Dy in range(min(2, ny)):
            for Dx in range(min(2, nx)):
                T, C = _near((Dx, Dy, Dz), kappa)
                at = (Dz * ny + Dy) * nx + Dx
                out[:6, at] = torch.from_numpy(T).cuda()
                if curl:
                    out[6:, at] = torch.from_numpy(C).cuda()
    out = out.reshape(-1, nz, ny, nx)
    return out[:6], out[6:]


# components odd along (x, y, z): xx yy zz xy xz yz, then the curl's x y z
_ODD = [(0, 0, 0), (0, 0, 0), (0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, 0, 0), (0, 1, 0), (0, 0, 1)]
_PAIR = [[0, 3, 4], [3, 1, 5], [4, 5, 2]]


def _spectra(tables, first):
    """Spectra of the doubled circulant embedding of octant tables; `first` is the
    place in _ODD of the first one."""
    out = []
    for c, t in enumerate(tables):
        for axis, odd in zip((2, 1, 0), _ODD[first + c]):
            mirror = torch.flip(t.narrow(axis, 1, t.shape[axis] - 1), (axis,)) if t.shape[axis] > 1 else t.narrow(axis, 0, 0)
            gap = torch.zeros_like(t.narrow(axis, 0, 1))
            t = torch.cat([t, gap, -mirror if odd else mirror], axis)
        out.append(torch.fft.fftn(t))
    return out


def _convolve(spectra_sum, f):
    """Crop of the inverse transforms of spectra_sum(padded spectra of f)."""
    nz, ny, nx = f.shape[1:]
    F = torch.fft.fftn(f, s=(2 * nz, 2 * ny, 2 * nx), dim=(1, 2, 3))
    return torch.stack([torch.fft.ifftn(u)[:nz, :ny, :nx] for u in spectra_sum(F)])


def _apply_T(G, w):
    return _convolve(lambda F: (G[r[0]] * F[0] + G[r[1]] * F[1] + G[r[2]] * F[2] for r in _PAIR), w)


def _apply_curl(C, f):
    cross = ((1, 2), (2, 0), (0, 1))
    return _convolve(lambda F: (C[a] * F[b] - C[b] * F[a] for a, b in cross), f)


def _gmres(apply, b, tol, m=400):
    """x with |b - apply(x)| <= tol |b|: restarted GMRES(m), two Gram-Schmidt passes."""
    x, bn = torch.zeros_like(b), torch.linalg.vector_norm(b).item()
    V = torch.empty((m + 1, b.numel()), dtype=b.dtype, device=b.device)
    for _ in range(8):
        r = b - apply(x)
        beta = torch.linalg.vector_norm(r).item()
        if beta <= tol * bn:
            break
        V[0] = r / beta
        H = torch.zeros((m + 1, m), dtype=b.dtype, device=b.device)
        for j in range(m):
            w = apply(V[j])
            for _ in range(2):
                h = V[:j + 1].conj() @ w
                w = w - h @ V[:j + 1]
                H[:j + 1, j] += h
            H[j + 1, j] = torch.linalg.vector_norm(w)
            V[j + 1] = w / H[j + 1, j]
            if j % 50 == 49 or j == m - 1:
                Hn = H[:j + 2, :j + 1].cpu().numpy()
                e = np.zeros(j + 2, complex)
                e[0] = beta
                y = np.linalg.lstsq(Hn, e, rcond=None)[0]
                if np.linalg.norm(e - Hn @ y) <= 0.3 * tol * bn:
                    break
        x = x + torch.from_numpy(y).cuda() @ V[:len(y)]
    return x


def _net_forward(params, X):
    """The network in 64 bits on X (1, 8, nz, ny, nx); params: per layer (weight, bias)."""
    F = torch.nn.functional

    def conv(x, name):
        return F.conv3d(x, params[name][0], params[name][1], padding=1)

    def pool(x):       # 2 x 2 in (y, x); a ragged edge averages the voxels that exist
        return F.avg_pool3d(x, (1, 2, 2), ceil_mode=True, count_include_pad=False)

    h = [torch.relu(conv(X, "enc0"))]
    for level in (1, 2, 3):
        h.append(torch.relu(conv(pool(h[-1]), "enc%d" % level)))
    u = h[3]
    for level in (2, 1, 0):
        up = u.repeat_interleave(2, 3).repeat_interleave(2, 4)[..., :h[level].shape[3], :h[level].shape[4]]
        u = torch.relu(conv(up + h[level], "dec%d" % level))
    return conv(u, "out")


def _net_exact_inputs(flat):
    """Per layer the weights as the kernels hold them (16-bit) and the biases, in 64 bits."""
    params, at = {}, 0
    for name, ci, co in LAYERS:
        w = torch.from_numpy(flat[at:at + co * ci * 27]).to(torch.bfloat16).double().cuda().reshape(co, ci, 3, 3, 3)
        at += co * ci * 27
        params[name] = (w.requires_grad_(), torch.from_numpy(flat[at:at + co]).double().cuda().requires_grad_())
        at += co
    return params


def _planar(v):
    return torch.cat([v.real, v.imag])


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        h, k0, eps_bg, guides = _batch_problem(case, seed)
        out, spectra = [], {}
        for g, eps, absorbers, x in guides:
            if g["nx"] not in spectra:
                spectra[g["nx"]] = _spectra(_entries((g["nx"], g["ny"], g["nz"]), k0 * math.sqrt(eps_bg) * h)[0], 0)
            chi = torch.from_numpy(_chi(g, eps, absorbers, eps_bg)).cuda()
            w = x.to(torch.complex128)
            out.append((w - chi / (1 + chi) * _apply_T(spectra[g["nx"]], w)).reshape(-1))
        return out

    rng, h, k0, eps_bg, eps, absorbers = _problem(case, seed)
    n, shape = (case["nx"], case["ny"], case["nz"]), (case["nz"], case["ny"], case["nx"])
    chi = torch.from_numpy(_chi(case, eps, absorbers, eps_bg)).cuda()
    kappa = k0 * math.sqrt(eps_bg) * h
    if kind in ("net_apply", "net_train"):
        params = _net_exact_inputs(_net_params(rng))
        chi_channels = torch.stack([chi.real, chi.imag])

        def scaled(v):
            s = math.sqrt(v.numel() / v.abs().square().sum().item())
            return s, torch.cat([_planar(v * s), chi_channels])[None]

        if kind == "net_apply":
            v = _normal(rng, (3,) + shape, case["dtype"]).to(torch.complex128)
            s, X = scaled(v)
            with torch.no_grad():
                y = _net_forward(params, X)[0]
            return (v + torch.complex(y[:3], y[3:]) / s).reshape(-1)
        losses = []
        for _ in range(case["samples"]):
            r, e = (t.to(torch.complex128) for t in _pair(case, rng, (3,) + shape))
            s, X = scaled(r)
            loss = (_net_forward(params, X)[0] - _planar((e - r) * s)).square().sum() / (e * s).abs().square().sum()
            loss.backward()
            losses.append(loss.item())
        return dict(losses=losses, grads=torch.cat([p.grad.reshape(-1) for name, _, _ in LAYERS for p in params[name]]))

    T, C = _entries(n, kappa, curl=kind == "jm_operator")
    G = _spectra(T, 0)
    M = chi / (1 + chi)
    if kind == "setup":
        src = _normal(rng, (3,) + shape)
        return (M * (_apply_T(G, src) - src)).reshape(-1)
    if kind == "operator":
        w = _normal(rng, (3,) + shape, case["dtype"]).to(torch.complex128)
        return (w - M * _apply_T(G, w)).reshape(-1)
    if kind == "jm_operator":
        K = _spectra(C, 6)
        mu = 1 + 1j * chi.imag / (1 + chi.real)
        Mm = (mu - 1) / mu
        u = _normal(rng, (6,) + shape, case["dtype"]).to(torch.complex128)
        e, m = u[:3], u[3:]
        ye = e - M * (_apply_T(G, e) - 1j * kappa * _apply_curl(K, m))
        ym = m - Mm * (_apply_T(G, m) + 1j * kappa * _apply_curl(K, e))
        return torch.cat([ye, ym]).reshape(-1)
    b = M * torch.from_numpy(_incident(case, rng, h, k0)).cuda()
    return _gmres(lambda v: (v.reshape((3,) + shape) - M * _apply_T(G, v.reshape((3,) + shape))).reshape(-1),
                  b.reshape(-1), 1e-13)
