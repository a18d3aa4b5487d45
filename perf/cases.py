"""What users of this library have it do, as cases that can be timed and compared.

  apply     Q_M v, the interpolated preconditioner, on device vectors: the
            call of a program that brings its own Krylov method
  operator  P_N x, the periodic finite-difference Helmholtz operator
  solve     P_N u = f by restarted (F)GMRES, the library's main use
  serve     requests on host arrays through the solve server

Axis lengths are those of the workloads and the parity tests: 48 ... 2400,
powers of two, with a factor 3 and with a factor 5.  Plans keep the default
launch shapes, so that a result does not depend on a timing made while
tuning.
"""
import math

import numpy as np
import torch

C_O = 1.0          # background speed, the speed inside the absorbing layer
ZETA_MAX = 0.15    # strength of the absorbing layer
TAPER = 8          # cells over which a medium blends into the layer


def listed():
    return [
        # the smallest serving grid: a few small kernels, set by latency and launches
        {"name": "apply_c64_256", "kind": "apply", "shape": "256x256", "M": 6, "Mt": 2, "rhs": 1, "prec": 1},
        # the 2D single-source workload
        {"name": "apply_c64_1024", "kind": "apply", "shape": "1024x1024", "M": 12, "Mt": 4, "rhs": 1, "prec": 1},
        # many sources on one medium
        {"name": "apply_c64_512_rhs16", "kind": "apply", "shape": "512x512", "M": 9, "Mt": 3, "rhs": 16, "prec": 1},
        # the 3D workload, the largest apply
        {"name": "apply_c64_256cube", "kind": "apply", "shape": "256x256x256", "M": 12, "Mt": 4, "rhs": 1, "prec": 1},
        # the FP64 preconditioner on a grid with factors 3 and 5 (the complexity study's lengths)
        {"name": "apply_c128_480x720", "kind": "apply", "shape": "480x720", "M": 8, "Mt": 0, "rhs": 1, "prec": 0},
        # the operator at Example 1's grid, with damping
        {"name": "operator_2400", "kind": "operator", "shape": "2400x2400", "rhs": 1, "prec": 0, "damped": True},
        # the operator on a complex64 vector, as flexible GMRES applies it, on a 3D serving grid
        {"name": "operator_c64_192cube", "kind": "operator", "shape": "192x192x192", "rhs": 1, "prec": 1, "damped": False},
        # a small solve with everything in FP64
        {"name": "solve_fp64_128", "kind": "solve", "shape": "128x128", "medium": "bumps", "M": 6, "Mt": 2, "rhs": 1,
         "prec": 0, "restart": 30, "width": 16, "ppw": 10.0, "alpha": 0.15, "graphs": True, "steps": 30},
        # the 2D single-source workload, solved
        {"name": "solve_1024", "kind": "solve", "shape": "1024x1024", "medium": "gradient", "M": 12, "Mt": 4, "rhs": 1,
         "prec": 1, "restart": 40, "width": 32, "ppw": 8.0, "alpha": 0.1, "graphs": True, "steps": 100},
        # several sources on one medium
        {"name": "solve_512_rhs8", "kind": "solve", "shape": "512x512", "medium": "bumps", "M": 9, "Mt": 3, "rhs": 8,
         "prec": 1, "restart": 40, "width": 16, "ppw": 10.0, "alpha": 0.1, "graphs": True, "steps": 70},
        # the largest single-GPU workload, solved
        {"name": "solve_256cube", "kind": "solve", "shape": "256x256x256", "medium": "layers", "M": 12, "Mt": 4, "rhs": 1,
         "prec": 1, "restart": 40, "width": 24, "ppw": 8.0, "alpha": 0.3, "graphs": False, "steps": 95},
        # four requests on media of their own, from host arrays to host arrays, set-up included
        {"name": "serve_256", "kind": "serve", "shape": "256x256", "medium": "bumps", "M": 6, "Mt": 2, "rhs": 2,
         "prec": 1, "restart": 40, "width": 16, "ppw": 10.0, "alpha": 0.1, "graphs": True, "steps": 45, "requests": 4},
    ]


LENGTHS_2D = (48, 64, 96, 120, 128, 180, 192, 240, 256, 360, 480, 512, 720, 960, 1024, 1440, 1920, 2048)
LENGTHS_3D = (24, 32, 40, 48, 60, 64, 96, 120, 128, 180, 192, 240, 256)
SOLVE_2D = (120, 128, 180, 192, 240, 256, 360, 480, 512, 720)
SOLVE_3D = (60, 64, 96, 120, 128)


def _near(rng, lengths, target):
    """A length near target on a logarithmic scale (the three nearest alike)."""
    return rng.choice(sorted(lengths, key=lambda v: abs(math.log(v / target)))[:3])


def draw(rng):
    what = rng.random()
    if what < 0.55:
        # apply: 3e3 ... 1.6e7 points over all right-hand sides
        prec = 1 if rng.random() < 0.7 else 0
        points = math.exp(rng.uniform(math.log(4e3), math.log(1.2e7 if prec else 1e6)))
        rhs = rng.choice((1, 1, 1, 2, 3, 5, 8))
        points = max(points / rhs, 3e3)
        planes = rng.choice(((4, 2), (6, 2), (8, 0), (9, 3), (12, 4)))
        if rng.random() < 0.6:
            y = _near(rng, LENGTHS_2D, math.sqrt(points) * rng.uniform(0.6, 1.7))
            shape = "%dx%d" % (y, _near(rng, LENGTHS_2D, points / y))
        else:
            z = _near(rng, LENGTHS_3D, points ** (1 / 3) * rng.uniform(0.7, 1.4))
            y = _near(rng, LENGTHS_3D, math.sqrt(points / z))
            shape = "%dx%dx%d" % (z, y, _near(rng, LENGTHS_3D, points / z / y))
        return {"kind": "apply", "shape": shape, "M": planes[0], "Mt": planes[1], "rhs": rhs, "prec": prec}
    if what < 0.7:
        points = math.exp(rng.uniform(math.log(4e3), math.log(8e6)))
        rhs = rng.choice((1, 1, 2, 4))
        if rng.random() < 0.5:
            y = _near(rng, LENGTHS_2D, math.sqrt(points))
            shape = "%dx%d" % (y, _near(rng, LENGTHS_2D, points / y))
        else:
            z = _near(rng, LENGTHS_3D, points ** (1 / 3))
            shape = "%dx%dx%d" % (z, z, _near(rng, LENGTHS_3D, points / z / z))
        return {"kind": "operator", "shape": shape, "rhs": rhs, "prec": rng.choice((0, 1)), "damped": rng.random() < 0.5}
    case = {"kind": "solve", "rhs": rng.choice((1, 1, 2, 3, 4)), "prec": 1 if rng.random() < 0.8 else 0,
            "restart": rng.choice((20, 30, 40)), "width": 16, "ppw": round(rng.uniform(8.0, 11.0), 2),
            "graphs": rng.random() < 0.5}
    if rng.random() < 0.6:
        n = rng.choice(SOLVE_2D)
        case.update(shape="%dx%d" % (n, n), medium=rng.choice(("bumps", "gradient")), M=12, Mt=4,
                    alpha=0.15, steps=60)
    else:
        n = rng.choice(SOLVE_3D)
        case.update(shape="%dx%dx%d" % (n, n, n), medium=rng.choice(("bumps", "layers")), M=12, Mt=4,
                    alpha=0.2, steps=50)
        case["width"] = 12
    return case


def _shape(case):
    return tuple(int(v) for v in case["shape"].split("x"))


def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + 77 + salt)
    return g


def _medium(shape, kind, width, seed):
    """Wave speed and layer profile (float64 device tensors) in the unit box:
    smooth bumps on 1 ("bumps"), bumps on a gradient mapped to [1, 2]
    ("gradient"), or smoothed horizontal layers with spherical inclusions
    ("layers"), blended to C_O towards a layer of `width` cells."""
    rng = np.random.Generator(np.random.PCG64([20260, int(seed)]))
    d, h = len(shape), 1.0 / shape[-1]
    X = []
    for ax, n in enumerate(shape):
        b = [1] * d
        b[ax] = n
        X.append((torch.arange(n, device="cuda", dtype=torch.float64) / n - 0.5).reshape(b))
    inner = max(0.5 - (width + TAPER) * h, 0.05)
    if kind == "layers":
        speeds = rng.uniform(1.0, 3.0, 6)
        depths = np.sort(rng.uniform(-inner, inner, 5))
        c = torch.full(shape, float(speeds[0]), device="cuda", dtype=torch.float64)
        for i in range(5):
            c = c + (speeds[i + 1] - speeds[i]) * torch.sigmoid((X[0] - depths[i]) / (2 * h))
        for _ in range(10):
            r = rng.uniform(8, 20) / 256.0
            ctr = rng.uniform(-1, 1, d) * max(inner - r, 0.0)
            dist = torch.sqrt(sum((X[ax] - ctr[ax]) ** 2 for ax in range(d)))
            c = c * (1.0 + (0.2 if rng.uniform() < 0.5 else -0.2) * torch.sigmoid((r - dist) / (2 * h)))
    else:
        count, amp, sig = (3, (0.3, 0.3), (0.1, 0.1)) if kind == "bumps" else (20, (0.0, 1.0), (0.02, 0.1))
        c = torch.zeros(shape, device="cuda", dtype=torch.float64)
        for _ in range(count):
            a, s = rng.uniform(*amp), rng.uniform(*sig)
            ctr = rng.uniform(-1, 1, d) * max(inner - 2 * s, 0.02)
            c = c + a * torch.exp(-sum((X[ax] - ctr[ax]) ** 2 for ax in range(d)) / (2 * s * s))
        if kind == "gradient":
            c = c + 0.5 * (X[-1] + 0.5)
            c = 1.0 + (c - c.min()) / (c.max() - c.min())
        else:
            c = 1.0 + c
    dist = None
    for ax, n in enumerate(shape):
        i = torch.arange(n, device="cuda", dtype=torch.float64)
        b = [1] * d
        b[ax] = n
        di = torch.minimum(i, n - 1 - i).reshape(b)
        dist = di if dist is None else torch.minimum(dist, di)
    dist = dist.expand(shape)
    s = ((dist - width + 1) / (TAPER + 1)).clamp(0.0, 1.0)
    tau = torch.where(dist < width, 0.0, 0.5 * (1.0 - torch.cos(math.pi * s)))
    c = torch.where(dist < width, C_O, C_O + tau * (c - C_O))
    zeta = torch.where(dist < width, ZETA_MAX * (width - dist) / max(width, 1), 0.0)
    return c.contiguous(), zeta.contiguous(), dist


def _sources(dist, rhs, width, seed):
    """Unit point sources away from the layer, one per right-hand side."""
    rng = np.random.Generator(np.random.PCG64([20261, int(seed)]))
    f = torch.zeros((rhs,) + tuple(dist.shape), dtype=torch.complex128, device="cuda")
    for b in range(rhs):
        at = []
        for n in dist.shape:
            lo = min(width + TAPER, n // 2 - 1)
            at.append(int(rng.integers(lo, n - lo)))
        f[(b,) + tuple(at)] = 1.0
    return f


def _vector(shape, rhs, seed):
    return torch.randn((rhs,) + shape, dtype=torch.complex128, device="cuda", generator=_gen(seed))


def _field(case, seed):
    """The medium of an apply or operator case: (c, zeta, omega, alpha)."""
    shape = _shape(case)
    layer = case.get("Mt", 4) > 0
    width = max(2, min(24, min(shape) // 10)) if layer else 0
    c, zeta, _ = _medium(shape, "bumps", width, seed)
    return c, zeta if layer else None, 2.0 * math.pi * float(c.min()) * min(shape) / 8.0, 0.15


def prepare(case, seed):
    from paper_2409_16172_gb300 import hz
    shape, kind = _shape(case), case["kind"]
    if kind in ("apply", "operator"):
        c, zeta, omega, alpha = _field(case, seed)
        a = None
        if case.get("damped"):
            a = (20.0 + 10.0 * torch.rand(shape, dtype=torch.float64, device="cuda", generator=_gen(seed, 5))).cpu().numpy()
        med = hz.Medium(c.cpu().numpy(), None if zeta is None else zeta.cpu().numpy(), a, omega=omega,
                        M=case.get("M", 8), Mt=case.get("Mt", 4), c_o=C_O, alpha=alpha)
        x = _vector(shape, case["rhs"], seed)
        if kind == "operator" and case["prec"] == 1:
            x = x.to(torch.complex64)
        plan = hz.Plan(med, precision=case["prec"], restart=4, max_nrhs=case["rhs"])
        return {"case": case, "plan": plan, "x": x, "out": torch.empty(x.shape, dtype=torch.complex128, device="cuda")}
    if kind == "serve":
        reqs = []
        for i in range(case["requests"]):
            c, zeta, dist = _medium(shape, case["medium"], case["width"], int(seed) * 64 + i)
            f = _sources(dist, case["rhs"], case["width"], int(seed) * 64 + i)
            omega = 2.0 * math.pi * float(c.min()) * min(shape) / case["ppw"]
            reqs.append((c.cpu().numpy(), zeta.cpu().numpy(), f.cpu().numpy(), omega))
        return {"case": case, "server": hz.Server(max_slots=4, autotune=-1), "requests": reqs}
    c, zeta, dist = _medium(shape, case["medium"], case["width"], seed)
    omega = 2.0 * math.pi * float(c.min()) * min(shape) / case["ppw"]
    f = _sources(dist, case["rhs"], case["width"], seed)
    med = hz.Medium(c.cpu().numpy(), zeta.cpu().numpy(), omega=omega, M=case["M"], Mt=case["Mt"], c_o=C_O,
                    alpha=case["alpha"])
    plan = hz.Plan(med, precision=case["prec"], restart=case["restart"], tol=1e-6, maxit=400,
                   max_nrhs=case["rhs"], graphs=case["graphs"])
    return {"case": case, "plan": plan, "f": f, "u": torch.empty_like(f)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "apply":
        y = state["plan"].apply_preconditioner(state["x"], precision=case["prec"], out=state["out"])
        # a flexible Krylov method keeps what the complex64 preconditioner
        # gives it in complex64, as the library's own FGMRES does
        return [y.to(torch.complex64) if case["prec"] == 1 else y]
    if kind == "operator":
        return [state["plan"].apply_operator(state["x"], out=state["out"])]
    if kind == "solve":
        u, _ = state["plan"].solve(state["f"], state["u"].zero_())
        return [u]
    srv = state["server"]
    tickets = [srv.submit(c, f, omega=w, M=case["M"], Mt=case["Mt"], zeta=z, c_o=C_O, alpha=case["alpha"],
                          precision=case["prec"], restart=case["restart"], tol=1e-6, maxit=400, graphs=case["graphs"])
               for c, z, f, w in state["requests"]]
    return [srv.result(t)[1] for t in tickets]


def work(case):
    shape = _shape(case)
    n = math.prod(shape)
    b = case["rhs"] * case.get("requests", 1)
    s = 8.0 if case["prec"] == 1 else 16.0
    planes = case.get("M", 0) + case.get("Mt", 0)
    transform = 5.0 * n * math.log2(n)
    apply_flops = (planes + 1) * transform + 14.0 * n * planes
    op_flops = (30.0 if len(shape) == 3 else 26.0) * n
    if case["kind"] == "apply":
        # input, output, interpolation record
        return {"bytes": n * (b * (16.0 + s) + s / 2), "flops": b * apply_flops}
    if case["kind"] == "operator":
        return {"bytes": n * (b * (s + 16.0) + 16.0 + (8.0 if case["damped"] else 0.0)), "flops": b * op_flops}
    # Arnoldi steps: at step j the vector is orthogonalised twice against
    # j + 1 basis vectors (the basis is larger than a cache: read once each
    # time), and one preconditioner apply and one operator apply are made
    m = case["restart"]
    bytes_, flops = 0.0, 0.0
    for k in range(case["steps"]):
        j = k % m + 1
        bytes_ += n * (2 * 16.0 * j + 16.0 + 3 * s + 32.0)
        flops += 2 * 16.0 * n * j + apply_flops + op_flops
    return {"bytes": b * bytes_, "flops": b * flops}


# ---------------------------------------------------------------------------
# The same numbers in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _real_nodes(lo, hi, m, split):
    if m == 1 or hi - lo <= 1e-12 * hi:
        return [C_O if m == 1 and split else lo]
    if split and lo < C_O < hi:
        s1 = min(max(int(math.floor((m - 1) * (C_O - lo) / (hi - lo) + 0.5)), 1), m - 2)
        s2 = m - 1 - s1
        return [lo + (C_O - lo) * i / s1 for i in range(s1)] + [C_O + (hi - C_O) * i / s2 for i in range(s2)] + [hi]
    return [lo + (hi - lo) * i / (m - 1) for i in range(m - 1)] + [hi]


def _hats(x, nodes):
    """Hat functions of increasing nodes at x, one tensor per node."""
    if len(nodes) == 1:
        return [torch.ones_like(x)]
    x = x.clamp(nodes[0], nodes[-1])
    out = []
    for i, v in enumerate(nodes):
        w = torch.zeros_like(x)
        if i > 0:
            w = torch.where((x >= nodes[i - 1]) & (x <= v), (x - nodes[i - 1]) / (v - nodes[i - 1]), w)
        if i + 1 < len(nodes):
            w = torch.where((x >= v) & (x <= nodes[i + 1]), (nodes[i + 1] - x) / (nodes[i + 1] - v), w)
        out.append(w)
    return out


def _exact_apply(case, seed):
    shape = _shape(case)
    c, zeta, omega, alpha = _field(case, seed)
    x = _vector(shape, case["rhs"], seed)
    layer = zeta is not None
    lo, hi = float(c.min()), float(c.max())
    if layer:
        lo, hi = min(lo, C_O), max(hi, C_O)
    real = _real_nodes(lo, hi, case["M"], layer)
    weights = _hats(c, real)
    gammas = [complex(v) for v in real]
    if layer:
        inside = zeta > 0
        zn = [i * float(zeta.max()) / case["Mt"] for i in range(case["Mt"])] + [float(zeta.max())]
        wz = _hats(zeta, zn)
        at = real.index(C_O)
        weights = [torch.where(inside, wz[0] if k == at else torch.zeros_like(w), w) for k, w in enumerate(weights)]
        weights += [torch.where(inside, w, 0.0) for w in wz[1:]]
        gammas += [C_O * (1.0 - 1j * z) for z in zn[1:]]
    d = len(shape)
    xi2 = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for ax, n in enumerate(shape):
        b = [1] * d
        b[ax] = n
        k = torch.arange(n, device="cuda", dtype=torch.float64)
        k = torch.where(k <= (n - 1) // 2, k, k - n)
        xi2 = xi2 + ((2.0 * math.pi * k) ** 2).reshape(b)
    out = torch.empty_like(x)
    for r in range(case["rhs"]):
        xhat = torch.fft.fftn(x[r])
        acc = torch.zeros_like(x[r])
        for g, w in zip(gammas, weights):
            q = 1.0 / (complex(omega * omega, omega * alpha * omega) - g * g * xi2)
            acc += w * torch.fft.ifftn(q * xhat)
        out[r] = acc
    return [out]


def _exact_operator(case, seed):
    shape = _shape(case)
    c, zeta, omega, _ = _field(case, seed)
    x = _vector(shape, case["rhs"], seed)
    if case["prec"] == 1:
        x = x.to(torch.complex64).to(torch.complex128)
    g = (c * (1.0 - 1j * zeta)) ** 2
    lap = torch.zeros_like(x)
    for ax, n in enumerate(shape):
        lap += (torch.roll(x, 1, ax + 1) - 2.0 * x + torch.roll(x, -1, ax + 1)) * float(n) ** 2
    a = 0.0
    if case["damped"]:
        a = 20.0 + 10.0 * torch.rand(shape, dtype=torch.float64, device="cuda", generator=_gen(seed, 5))
    return [g * lap + (omega * omega + 1j * omega * a) * x]


def exact(case, seed):
    if case["kind"] == "apply":
        return _exact_apply(case, seed)
    if case["kind"] == "operator":
        return _exact_operator(case, seed)
    # a solve stops at its tolerance: what it returns has no value in 64 bits
    return None
