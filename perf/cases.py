"""Timing cases: the work a user has this library do, through its Python entry points.

Four groups, each from the smallest call to the largest mesh the configurations use:
flat Poisson solves (cold, warm-started, FP64, forward + gradient), moving-mesh solves
(19-point curvilinear operator: forward, forward + gradient, the symmetric variant, a
mesh-motion step), batches of independent solves, and a particle-mesh force evaluation.

Sources are seeded Gaussian random fields with P(k) ~ k^-2, deformation potentials are
Gaussian-smoothed fields scaled to a bounded Hessian, particles are a displaced lattice;
all are made on the GPU from the seed.  `exact` evaluates the same quantities in FP64 with
plain torch: FFT solves of the 7-point operator, preconditioned BiCGStab solves of the
curvilinear one, autograd for the gradient through the geometry.
"""
import math

import torch

import paper_2607_10983_gb300 as gb

TOL = 1e-6


# ------------------------------------------------------------------ cases


def listed():
    return [
        # the plain method's configuration: FP64 V-cycles on 32^3 to 1e-10 (smallest call; latency)
        {"name": "fp64_32", "kind": "flat", "shape": "32x32x32", "prec": "fp64", "warm": False, "tol": 1e-10,
         "degree": 3},
        # one small field-level-inference sample, solved alone
        {"name": "cold_64", "kind": "flat", "shape": "64x64x64", "prec": "mixed", "warm": False, "tol": TOL,
         "degree": 3},
        # a time step of a ragged box, warm-started from the previous step
        {"name": "warm_ragged", "kind": "flat", "shape": "160x128x224", "prec": "mixed", "warm": True, "tol": TOL,
         "degree": 3},
        # first step of a large box with three different sides
        {"name": "cold_ragged_large", "kind": "flat", "shape": "320x448x384", "prec": "mixed", "warm": False,
         "tol": TOL, "degree": 3},
        # the benchmark's time step: 512^3, warm-started (recycled) from the previous solution
        {"name": "warm_512", "kind": "flat", "shape": "512x512x512", "prec": "mixed", "warm": True, "tol": TOL,
         "degree": 3},
        # differentiable solve: loss = sum(w . grad4 phi), forward and backward
        {"name": "grad_256", "kind": "flat_grad", "shape": "256x256x256", "tol": TOL},
        # moving mesh: new geometry and one forward solve on a ragged box
        {"name": "mesh_ragged", "kind": "mesh", "shape": "160x128x192", "sym": False, "tol": TOL},
        # moving mesh: forward solve and the gradient with respect to source and geometry
        {"name": "mesh_grad_256", "kind": "mesh_grad", "shape": "256x256x256", "sym": False, "tol": TOL},
        # the symmetric discretisation of the same operator
        {"name": "mesh_sym_128", "kind": "mesh", "shape": "128x128x128", "sym": True, "tol": TOL},
        # one mesh-motion step: smoothed source, solve for the rate, advance the potential
        {"name": "motion_128", "kind": "motion", "shape": "128x128x128", "tol": TOL},
        # 48 independent samples of three sizes in one persistent launch under a CUDA graph
        {"name": "batch_48", "kind": "batch", "shapes": "64x64x64 96x96x96 128x128x128", "each": 16, "tol": TOL},
        # one force evaluation of a particle-mesh step: paint, warm solve, force at the particles
        {"name": "pm_256", "kind": "pm", "shape": "256x256x256", "tol": TOL},
    ]


def _side(rng, lo, hi):
    """A side m 2^k in [lo, hi], m in 4..7, the sizes spread over their logarithm."""
    sides = sorted({m << k for m in (4, 5, 6, 7) for k in range(1, 8) if lo <= m << k <= hi})
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(sides, key=lambda s: abs(math.log(s / t)))


def _levels_ok(s):
    """The coarsest level (halved while all sides are even and >= 8) has at most 6^3 cells (96^3's
    hierarchy; set-up inverts that level's operator on the host)."""
    while all(v % 2 == 0 and v >= 8 for v in s):
        s = [v // 2 for v in s]
    return s[0] * s[1] * s[2] <= 216


def _shape(rng, lo, hi, cells):
    """Three sides in [lo, hi], equal in a third of the cases, at most `cells` cells."""
    while True:
        if rng.random() < 0.33:
            s = [_side(rng, lo, hi)] * 3
        else:
            s = [_side(rng, lo, hi) for _ in range(3)]
        if s[0] * s[1] * s[2] <= cells and _levels_ok(list(s)):
            return "x".join(str(v) for v in s)


def draw(rng):
    kind = rng.choice(["flat", "flat", "flat", "fp64", "flat_grad", "mesh", "mesh", "mesh_grad", "motion", "batch",
                       "pm"])
    if kind == "flat":
        return {"kind": "flat", "shape": _shape(rng, 32, 512, 1 << 26), "prec": "mixed",
                "warm": rng.random() < 0.5, "tol": rng.choice([1e-5, 1e-6, 1e-8]), "degree": rng.choice([2, 3, 3, 4])}
    if kind == "fp64":
        return {"kind": "flat", "shape": _shape(rng, 16, 128, 1 << 21), "prec": "fp64", "warm": rng.random() < 0.5,
                "tol": rng.choice([1e-8, 1e-10]), "degree": 3}
    if kind == "flat_grad":
        return {"kind": "flat_grad", "shape": _shape(rng, 32, 256, 1 << 24), "tol": TOL}
    if kind == "mesh":
        return {"kind": "mesh", "shape": _shape(rng, 32, 224, 1 << 23), "sym": rng.random() < 0.3, "tol": TOL}
    if kind == "mesh_grad":
        return {"kind": "mesh_grad", "shape": _shape(rng, 32, 224, 1 << 23), "sym": rng.random() < 0.3, "tol": TOL}
    if kind == "motion":
        return {"kind": "motion", "shape": _shape(rng, 32, 192, 1 << 22), "tol": TOL}
    if kind == "batch":
        return {"kind": "batch", "shapes": " ".join(_shape(rng, 32, 128, 1 << 21) for _ in range(rng.choice([1, 2, 3]))),
                "each": rng.choice([3, 5, 8, 12]), "tol": TOL}
    return {"kind": "pm", "shape": _shape(rng, 48, 256, 1 << 24), "tol": TOL}


# ------------------------------------------------------------------ inputs


def _dims(text):
    return tuple(int(v) for v in text.split("x"))


def _gen(seed, stream=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _waves(shape, half=True):
    def f(n, real):
        fr = torch.fft.rfftfreq(n, device="cuda", dtype=torch.float64) if real else torch.fft.fftfreq(
            n, device="cuda", dtype=torch.float64)
        return 2 * math.pi * fr
    nz, ny, nx = shape
    return f(nz, False)[:, None, None], f(ny, False)[None, :, None], f(nx, half)[None, None, :]


def _grf(shape, g, index=-2.0):
    """Zero-mean, unit-variance Gaussian random field with P(k) ~ k^index."""
    w = torch.fft.rfftn(torch.randn(shape, generator=g, device="cuda", dtype=torch.float64))
    kz, ky, kx = _waves(shape)
    k2 = kz * kz + ky * ky + kx * kx
    k2[0, 0, 0] = 1.0
    w *= k2.pow_(index / 4.0)
    w[0, 0, 0] = 0.0
    f = torch.fft.irfftn(w, s=shape)
    f -= f.mean()
    f /= f.std(unbiased=False)
    return f


def _psi(shape, g, sigma=4.0, rowsum=0.5):
    """Deformation potential: a smoothed field, the Gershgorin row sum of its Hessian at most `rowsum`."""
    b = torch.fft.rfftn(_grf(shape, g))
    k = _waves(shape)
    b *= torch.exp(-0.5 * sigma * sigma * (k[0] ** 2 + k[1] ** 2 + k[2] ** 2))
    worst = 0.0
    for a in range(3):
        acc = 0.0
        for c in range(3):
            acc = acc + torch.fft.irfftn(k[a] * k[c] * b, s=shape).abs_()
        worst = max(worst, float(acc.max()))
    psi = torch.fft.irfftn(b, s=shape) * (rowsum / worst)
    return psi - psi.mean()


def _symbol(shape):
    kz, ky, kx = _waves(shape)
    return -(4 * torch.sin(kz / 2) ** 2 + 4 * torch.sin(ky / 2) ** 2 + 4 * torch.sin(kx / 2) ** 2)


def _fft_solve(F):
    """Zero-mean FP64 solution of the 7-point equation for F - mean(F)."""
    s = _symbol(F.shape)
    s[0, 0, 0] = 1.0
    w = torch.fft.rfftn(F) / s
    w[0, 0, 0] = 0.0
    return torch.fft.irfftn(w, s=F.shape)


def _particles(shape, g, rms=2.0):
    """One particle per cell: a lattice displaced along the gradient of a smooth potential, twice:
    this step's positions and the previous step's (95% of the displacement)."""
    w = torch.fft.rfftn(torch.randn(shape, generator=g, device="cuda", dtype=torch.float64))
    k = _waves(shape)
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    k2[0, 0, 0] = 1.0
    w *= k2 ** -1.5
    w[0, 0, 0] = 0.0
    disp = torch.stack([torch.fft.irfftn(1j * k[a] * w, s=shape) for a in (2, 1, 0)], -1)
    disp *= rms / (disp ** 2).sum(-1).mean().sqrt()
    q = torch.stack(torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.float64) + 0.5 for n in shape],
                                   indexing="ij")[::-1], -1)
    n = torch.tensor(shape[::-1], device="cuda", dtype=torch.float64)
    return [((q + s * disp) % n).reshape(-1, 3).float().contiguous() for s in (1.0, 0.95)]


def _paint(shape, pos):
    """FP64 cloud-in-cell density, mass 1 per particle."""
    nz, ny, nx = shape
    x = pos.double()
    i = torch.floor(x)
    f = x - i
    i = i.long()
    rho = torch.zeros(nz * ny * nx, dtype=torch.float64, device="cuda")
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                w = (f[:, 0] if dx else 1 - f[:, 0]) * (f[:, 1] if dy else 1 - f[:, 1]) * (
                    f[:, 2] if dz else 1 - f[:, 2])
                at = (((i[:, 2] + dz) % nz) * ny + (i[:, 1] + dy) % ny) * nx + (i[:, 0] + dx) % nx
                rho.index_add_(0, at, w)
    return rho.view(shape)


def _inputs(case, seed):
    """The tensors a case starts from, from the seed alone."""
    kind = case["kind"]
    if kind == "batch":
        shapes = [_dims(s) for s in case["shapes"].split() for _ in range(case["each"])]
        return {"F": [_grf(s, _gen(seed, j)) for j, s in enumerate(shapes)], "shapes": shapes}
    shape = _dims(case["shape"])
    d = {"shape": shape}
    if kind == "flat":
        d["F"] = _grf(shape, _gen(seed))
        if case["warm"]:
            d["prev"] = _fft_solve(d["F"])
            d["F"] += 0.05 * _grf(shape, _gen(seed, 1))
    elif kind == "flat_grad":
        d["F"] = _grf(shape, _gen(seed))
        d["w"] = torch.randn((3,) + shape, generator=_gen(seed, 1), device="cuda", dtype=torch.float32)
    elif kind in ("mesh", "mesh_grad"):
        d["F"] = _grf(shape, _gen(seed))
        d["psi"] = _psi(shape, _gen(seed, 1))
        if kind == "mesh_grad":
            d["w"] = torch.randn((3,) + shape, generator=_gen(seed, 2), device="cuda", dtype=torch.float32)
    elif kind == "motion":
        d["rho"] = 1.0 + 0.3 * _grf(shape, _gen(seed))
        d["psi"] = _psi(shape, _gen(seed, 1), rowsum=0.3)
    elif kind == "pm":
        d["pos"], before = _particles(shape, _gen(seed))
        d["prev"] = _fft_solve(_paint(shape, before))
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    d["case"] = case
    if kind == "batch":
        d["batch"] = gb.Batch(d["shapes"])
        d["batch"].use_graph(True)
        d["phi"] = [torch.empty_like(f) for f in d["F"]]
        return d
    op = "curv" if kind in ("mesh", "mesh_grad", "motion") else "flat"
    d["solver"] = gb.Solver(d["shape"], op=op, prec=case.get("prec", "mixed"), degree=case.get("degree", 3),
                            curv_sym=case.get("sym", False))
    if kind in ("flat", "pm"):
        d["phi"] = torch.empty(d["shape"], dtype=torch.float64, device="cuda")
    if kind == "pm":
        d["rho"] = torch.empty(d["shape"], dtype=torch.float64, device="cuda")
    return d


# ------------------------------------------------------------------ one pass

MOTION = {"kappa": 1.0, "m_init": 1.0, "dtau": 0.1}


def run(d):
    case = d["case"]
    kind, tol = case["kind"], case["tol"]
    if kind == "flat":
        s = d["solver"]
        if case["warm"]:  # recycling: the previous solution is the initial guess
            s.predict([d["prev"]], order=0, growth=1.0, out=d["phi"])
        else:
            d["phi"].zero_()
        return s.solve(d["F"], d["phi"], tol=tol)[0]
    if kind == "flat_grad":
        F = d["F"].detach().requires_grad_(True)
        phi = gb.MGSolve.apply(F, d["solver"], tol, 50)
        loss = gb.GradDotLoss.apply(phi, d["w"], d["solver"], 4)
        loss.backward()
        return {"phi": phi.detach(), "loss": loss.detach(), "F_bar": F.grad}
    if kind == "mesh":
        return d["solver"].solve(d["F"], tol=tol, max_vcycles=100, psi=d["psi"])[0]
    if kind == "mesh_grad":
        F, psi = d["F"].detach().requires_grad_(True), d["psi"].detach().requires_grad_(True)
        phi = gb.CurvMGSolve.apply(F, psi, d["solver"], tol, 100)
        loss = gb.GradDotLoss.apply(phi, d["w"], d["solver"], 2)
        loss.backward()
        return {"phi": phi.detach(), "loss": loss.detach(), "F_bar": F.grad, "psi_bar": psi.grad}
    if kind == "motion":
        psi, dot, _ = d["solver"].mesh_motion(d["rho"], d["psi"].clone(), MOTION["kappa"], MOTION["m_init"],
                                              MOTION["dtau"], tol=tol)
        return {"psi": psi, "psidot": dot}
    if kind == "batch":
        for p in d["phi"]:
            p.zero_()
        d["batch"].solve(d["F"], d["phi"], tol=tol)
        n = case["each"]
        return [torch.stack(d["phi"][k:k + n]) for k in range(0, len(d["phi"]), n)]
    s = d["solver"]
    rho = s.cic_paint(d["pos"], out=d["rho"])
    s.predict([d["prev"]], order=0, growth=1.0, out=d["phi"])
    phi, _ = s.solve(rho, d["phi"], tol=tol)
    return {"rho": rho, "phi": phi, "force": s.force(phi, d["pos"])}


def work(case):
    """Bytes of inputs and outputs; operations of the V-cycles a solve of that tolerance takes
    (a factor of about 9 per flat and 3 per curvilinear cycle)."""
    kind = case["kind"]
    if kind == "batch":
        n = sum(math.prod(_dims(s)) for s in case["shapes"].split()) * case["each"]
    else:
        n = math.prod(_dims(case["shape"]))
    flat = math.ceil(math.log(1 / case["tol"]) / math.log(9.0)) * 100.0
    curv = math.ceil(math.log(1 / case["tol"]) / math.log(3.0)) * 400.0
    per = {"flat": (24 if case.get("warm") else 16, flat),
           "flat_grad": (8 + 12 + 8 + 8, 2 * flat + 40),
           "mesh": (16 + 8, curv + 100),
           "mesh_grad": (16 + 12 + 8 + 16, 2 * curv + 500),
           "motion": (16 + 16, curv + 150),
           "batch": (16, flat),
           "pm": (12 + 8 + 8 + 8 + 12, flat + 150)}[kind]
    return {"bytes": per[0] * n, "flops": per[1] * n}


# ------------------------------------------------------------------ the same in FP64


def _sh(u, a, s):
    """u displaced: value at the cell + s e_a (a = 0 x, 1 y, 2 z)."""
    return torch.roll(u, -s, 2 - a)


def _geometry(psi):
    def second(a):
        return _sh(psi, a, 1) + _sh(psi, a, -1) - 2 * psi + 1

    def mixed(a, b):
        return 0.25 * (_sh(_sh(psi, a, 1), b, 1) - _sh(_sh(psi, a, 1), b, -1) - _sh(_sh(psi, a, -1), b, 1)
                       + _sh(_sh(psi, a, -1), b, -1))
    a, b, c = second(0), second(1), second(2)
    d, e, f = mixed(0, 1), mixed(0, 2), mixed(1, 2)
    j00, j11, j22 = b * c - f * f, a * c - e * e, a * b - d * d
    j01, j02, j12 = e * f - d * c, d * f - b * e, d * e - a * f
    J = a * j00 + d * j01 + e * j02
    B = {(0, 0): (j00 * j00 + j01 * j01 + j02 * j02) / J, (1, 1): (j01 * j01 + j11 * j11 + j12 * j12) / J,
         (2, 2): (j02 * j02 + j12 * j12 + j22 * j22) / J, (0, 1): (j00 * j01 + j01 * j11 + j02 * j12) / J,
         (0, 2): (j00 * j02 + j01 * j12 + j02 * j22) / J, (1, 2): (j01 * j02 + j11 * j12 + j12 * j22) / J}
    return J, B


def _op(u, B, sym):
    """The flux divergence M u (sym False) or its symmetric variant."""
    out = 0.0
    for a in range(3):
        fl = 0.5 * (B[a, a] + _sh(B[a, a], a, 1)) * (_sh(u, a, 1) - u)
        if not sym:
            for b in range(3):
                if b != a:
                    k = (min(a, b), max(a, b))
                    t = _sh(u, b, 1) - _sh(u, b, -1)
                    fl = fl + 0.5 * (B[k] + _sh(B[k], a, 1)) * 0.25 * (t + _sh(t, a, 1))
        out = out + fl - _sh(fl, a, -1)
    if sym:
        for a in range(3):
            for b in range(a + 1, 3):
                c = B[a, b] + _sh(B[a, b], a, 1)
                C = 0.25 * (c + _sh(c, b, 1))

                def E(v, p, q):
                    t = _sh(v, p, 1) - v
                    return 0.5 * (t + _sh(t, q, 1))

                def ET(v, p, q):
                    t = 0.5 * (v + _sh(v, q, -1))
                    return _sh(t, p, -1) - t
                out = out - ET(C * E(u, b, a), a, b) - ET(C * E(u, a, b), b, a)
    return out


def _krylov(op, b, tol=1e-12, most=300):
    """BiCGStab for op(x) = b on zero-mean fields, preconditioned by the FFT solve."""
    x = torch.zeros_like(b)
    r = b - b.mean()
    r0, p = r.clone(), r.clone()
    rho = (r0 * r).sum()
    stop = tol * r.norm()
    for _ in range(most):
        y = _fft_solve(p)
        v = op(y)
        alpha = rho / (r0 * v).sum()
        s = r - alpha * v
        z = _fft_solve(s)
        t = op(z)
        omega = (t * s).sum() / (t * t).sum()
        x += alpha * y + omega * z
        r = s - omega * t
        if r.norm() <= stop:
            break
        new = (r0 * r).sum()
        p = r + (new / rho) * (alpha / omega) * (p - omega * v)
        rho = new
    return x - x.mean()


def _mesh_solve(F, J, B, sym):
    return _krylov(lambda u: _op(u, B, sym), J * (F - (J * F).sum() / J.sum()))


def _grad(u, order):
    """Components x, y, z of the centred gradient of the given order."""
    if order == 2:
        return [0.5 * (_sh(u, a, 1) - _sh(u, a, -1)) for a in range(3)]
    return [(8 * (_sh(u, a, 1) - _sh(u, a, -1)) - (_sh(u, a, 2) - _sh(u, a, -2))) / 12 for a in range(3)]


def _grad_t(w, order):
    """Transpose of _grad applied to w (3 components)."""
    if order == 2:
        return sum(0.5 * (_sh(w[a], a, -1) - _sh(w[a], a, 1)) for a in range(3))
    return sum((8 * (_sh(w[a], a, -1) - _sh(w[a], a, 1)) - (_sh(w[a], a, -2) - _sh(w[a], a, 2))) / 12
               for a in range(3))


def _read(fields, pos):
    nz, ny, nx = fields[0].shape
    x = pos.double()
    i = torch.floor(x)
    f = x - i
    i = i.long()
    out = torch.zeros((pos.shape[0], len(fields)), dtype=torch.float64, device="cuda")
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                w = (f[:, 0] if dx else 1 - f[:, 0]) * (f[:, 1] if dy else 1 - f[:, 1]) * (
                    f[:, 2] if dz else 1 - f[:, 2])
                at = (((i[:, 2] + dz) % nz) * ny + (i[:, 1] + dy) % ny) * nx + (i[:, 0] + dx) % nx
                for c, g in enumerate(fields):
                    out[:, c] += w * g.reshape(-1)[at]
    return out


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        n = case["each"]
        phi = [_fft_solve(f) for f in d["F"]]
        return [torch.stack(phi[k:k + n]) for k in range(0, len(phi), n)]
    if kind == "flat":
        return _fft_solve(d["F"])
    if kind == "flat_grad":
        phi, w = _fft_solve(d["F"]), d["w"].double()
        loss = sum((w[a] * g).sum() for a, g in enumerate(_grad(phi, 4)))
        return {"phi": phi, "loss": loss, "F_bar": _fft_solve(_grad_t(w, 4))}
    if kind == "mesh":
        J, B = _geometry(d["psi"])
        return _mesh_solve(d["F"], J, B, case["sym"])
    if kind == "mesh_grad":
        sym = case["sym"]
        psi = d["psi"].requires_grad_(True)
        J, B = _geometry(psi)
        Jc, Bc = J.detach(), {k: v.detach() for k, v in B.items()}
        F, w = d["F"], d["w"].double()
        phi = _mesh_solve(F, Jc, Bc, sym)
        loss = sum((w[a] * g).sum() for a, g in enumerate(_grad(phi, 2)))
        bar = _grad_t(w, 2)

        def op_t(y):
            with torch.enable_grad():
                u = torch.zeros_like(y).requires_grad_(True)
                return torch.autograd.grad(_op(u, Bc, sym), u, y)[0]
        lam = _krylov(op_t, bar - bar.mean())
        F_bar = Jc * (lam - (Jc * lam).sum() / Jc.sum())
        b = J * (F - (J * F).sum() / J.sum())
        psi_bar = torch.autograd.grad((lam * (b - _op(phi, B, sym))).sum(), psi)[0]
        return {"phi": phi, "loss": loss, "F_bar": F_bar, "psi_bar": psi_bar}
    if kind == "motion":
        J, B = _geometry(d["psi"])
        f = MOTION["kappa"] * (MOTION["m_init"] - J * d["rho"])
        for _ in range(2):
            for a in range(3):
                f = 0.5 * f + 0.25 * (_sh(f, a, 1) + _sh(f, a, -1))
        dot = _mesh_solve(f, J, B, False)
        psi = d["psi"] + MOTION["dtau"] * dot
        return {"psi": psi - psi.mean(), "psidot": dot}
    rho = _paint(d["shape"], d["pos"])
    phi = _fft_solve(rho)
    return {"rho": rho, "phi": phi, "force": -_read(_grad(phi, 4), d["pos"])}
