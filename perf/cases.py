"""What the framework is timed on: the calls its users make, over the range of
sizes and options they make them with.

A user has a lattice cell (an octet truss, its voxels' solid fractions between
0 and 1) and asks for the strain and stress fields under one macro strain, or
under the six unit strains the effective stiffness needs; under mixed control;
for several cells at once; in FP64; with the displacement solver; or for an
elastoplastic increment.  Around the solves stand the allocation-free operator
of small cells and the convolution layers of the network that proposes
starting fields.

Grid sizes are 2^a 3^b 5^c.  Cells, offsets in the cell, loads and layer data
are drawn from the seed.  A solve runs to its tolerance or its budget of
iterations, so that a pass is the same work whatever the cell, and returns its
stress fields, which carry the mean stresses and the effective stiffness; FP64
solves return the strain fields too (in FP32 a strain in empty space, which no
stiffness holds, is noise).
"""
import math

import numpy as np
import torch

from paper_2110_00733_gb300 import hom
from paper_2110_00733_gb300 import net as hnet

E_M, NU_M = 110e9, 0.3               # the metal of the linear workloads
E_P, NU_P, Y_P = 1.7e9, 0.4, 70e6    # the polymer of the elastoplastic ones
MASK_LATERAL = 0b111110              # mean stress prescribed but for component 11
SMOOTH = sorted(2 ** a * 3 ** b * 5 ** c for a in range(10) for b in range(6) for c in range(4)
                if 2 ** a * 3 ** b * 5 ** c <= 512)
SQ2 = math.sqrt(2.0)


def _solve(name, grid, strains=1, precision="f32", control="strain", scheme="rotated", rho=0.10, max_it=50):
    d = {"kind": "solve", "n1": grid[0], "n2": grid[1], "n3": grid[2], "strains": strains, "precision": precision,
         "control": control, "scheme": scheme, "rho": rho, "max_it": max_it}
    return dict(d, name=name) if name else d


def listed():
    return [
        # the smallest call: the operator in a loop that may not allocate
        {"name": "apply_noalloc_32", "kind": "noalloc", "n1": 32, "n2": 32, "n3": 32, "scheme": "rotated"},
        # effective stiffness of a coarse cell, as a parameter study asks for by the thousand
        _solve("stiffness_32", (32, 32, 32), strains=6, max_it=50),
        # effective stiffness at the resolution the paper's compression study uses (108 = 2^2 3^3)
        _solve("stiffness_108", (108, 108, 108), strains=6, rho=0.20, max_it=100),
        # an elongated cell: three different lengths, none a power of two, continuous frequencies
        _solve("solve_240x100x90", (240, 100, 90), scheme="continuous", rho=0.15, max_it=60),
        # a fine cell between the power-of-two sizes
        _solve("solve_192", (192, 192, 192), max_it=120),
        # the headline cell
        _solve("solve_256", (256, 256, 256), max_it=150),
        # Young's modulus and Poisson's ratio from one uniaxial solve
        _solve("uniaxial_128", (128, 128, 128), control="uniaxial", rho=0.15, max_it=60),
        # the same fields where FP32 is not enough
        _solve("solve_f64_96", (96, 96, 96), precision="f64", max_it=60),
        # a study of cells of several densities and sizes in one call
        {"name": "batch_64_96_128", "kind": "batch", "grids": "64,96,128", "rho": 0.12, "max_it": 80},
        # the displacement solver
        {"name": "modbfft_128", "kind": "modbfft", "n1": 128, "n2": 128, "n3": 128, "rho": 0.15,
         "max_it": 80},
        # an increment of a compression test on the edge of yield, a bounded number of Newton steps
        {"name": "j2_increment_48", "kind": "j2", "n1": 48, "n2": 48, "n3": 48, "rho": 0.30, "max_newton": 3,
         "max_lin": 60},
        # a layer of the warm-start network in training: forward, input gradient, weight gradient
        {"name": "conv_layer_64_16", "kind": "conv", "batch": 8, "n1": 64, "n2": 64, "n3": 64, "cin": 16, "cout": 16},
    ]


def _grid_near(rng, lo, hi, cap):
    """Three smooth lengths between lo and hi, alike to a factor of two, at most cap voxels."""
    while True:
        edge = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        g = [rng.choice([n for n in SMOOTH if lo <= n <= hi and 0.7 * edge <= n <= 1.4 * edge] or [lo]) for _ in range(3)]
        if rng.random() < 0.4:
            g = [g[0]] * 3
        if g[0] * g[1] * g[2] <= cap:
            return g


def draw(rng):
    kind = rng.choice(["solve"] * 7 + ["noalloc", "batch", "modbfft", "j2", "conv"])
    scheme = "rotated" if rng.random() < 0.8 else "continuous"
    rho = round(rng.uniform(0.08, 0.30), 3)
    if kind == "solve":
        control = "uniaxial" if rng.random() < 0.2 else "strain"
        precision = "f64" if rng.random() < 0.2 else "f32"
        strains = 6 if control == "strain" and rng.random() < 0.35 else 1
        cap = (0.3e6 if precision == "f64" else 3.5e6) / strains / (2 if control == "uniaxial" else 1)
        g = _grid_near(rng, 16, 256, cap)
        return _solve(None, g, strains, precision, control, scheme, rho)
    if kind == "batch":
        gs = [rng.choice([n for n in SMOOTH if 32 <= n <= 80]) for _ in range(rng.randint(2, 4))]
        return {"kind": "batch", "grids": ",".join(map(str, gs)), "rho": rho, "max_it": 60}
    if kind == "noalloc":
        g = [rng.choice([n for n in SMOOTH if 4 <= n <= 32]) for _ in range(3)]
        return {"kind": "noalloc", "n1": g[0], "n2": g[1], "n3": g[2], "scheme": scheme}
    if kind == "modbfft":
        g = _grid_near(rng, 24, 128, 1.0e6)
        return {"kind": "modbfft", "n1": g[0], "n2": g[1], "n3": g[2], "rho": rho, "max_it": 60}
    if kind == "j2":
        g = _grid_near(rng, 16, 60, 1.2e5)
        return {"kind": "j2", "n1": g[0], "n2": g[1], "n3": g[2], "rho": max(rho, 0.15), "max_newton": rng.randint(1, 3),
                "max_lin": 60}
    g = [rng.choice([8, 12, 16, 20, 24, 32, 40, 48, 64]) for _ in range(3)]
    b = max(1, min(rng.randint(1, 8), int(1.5e6 / (g[0] * g[1] * g[2]))))
    return {"kind": "conv", "batch": b, "n1": g[0], "n2": g[1], "n3": g[2], "cin": 16 * rng.randint(1, 4),
            "cout": 16 * rng.randint(1, 4)}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _grid(case):
    return case["n1"], case["n2"], case["n3"]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _octet(grid, rho, seed, dtype=torch.float32):
    """Octet-truss cell of density rho, its origin drawn from the seed: the
    struts' axes run along the face diagonals through the face-centred cubic
    points; phi is linear in the distance to the strut surface over one voxel."""
    shift = np.random.default_rng(seed).random(3)
    ax = [(torch.arange(n, device="cuda", dtype=torch.float32) + 0.5) / n + float(s) for n, s in zip(grid, shift)]
    x = torch.meshgrid(*ax, indexing="ij")
    near = lambda t: t - torch.round(t)  # noqa: E731
    d2 = torch.full(tuple(grid), 1e9, device="cuda")
    for a, b, c in ((0, 1, 2), (0, 2, 1), (1, 2, 0)):
        for s in (1.0, -1.0):
            u = x[a] - s * x[b]
            for off in (0.0, 0.5):
                d2 = torch.minimum(d2, near(x[c] - off) ** 2 + 0.5 * near(u - off) ** 2)
    d = d2.sqrt()
    width = (1.0 / (grid[0] * grid[1] * grid[2])) ** (1.0 / 3.0)
    phi_at = lambda r: (0.5 + (r - d) / width).clamp(0.0, 1.0)  # noqa: E731
    lo, hi = 0.0, 0.5
    for _ in range(20):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if float(phi_at(mid).mean(dtype=torch.float64)) < rho else (lo, mid)
    return phi_at(0.5 * (lo + hi)).to(dtype).contiguous()


def _unit_strain(seed):
    """A macro strain on the unit sphere of the Mandel norm, tensor components."""
    m = np.random.default_rng(seed + 77).standard_normal(6)
    m /= np.linalg.norm(m)
    m[3:] /= SQ2
    return 1e-3 * m


def _fields_for(grid, strains, dtype):
    new = lambda: torch.empty((6,) + tuple(grid), dtype=dtype, device="cuda")  # noqa: E731
    return [{"stress": new(), "strain": new()} if dtype == torch.float64 else {"stress": new()} for _ in range(strains)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        g = _grid(case)
        phi = _octet(g, 0.2, seed)
        eps = torch.randn((6,) + g, generator=_gen(seed), device="cuda")
        st = {"phi": phi, "eps": eps, "out": torch.empty_like(eps)}
    elif kind == "conv":
        g, B, ci, co = _grid(case), case["batch"], case["cin"], case["cout"]
        gen = _gen(seed)
        rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
        x = rnd(B, *g, ci).relu().bfloat16()
        W = (rnd(27, co, ci) / math.sqrt(27 * ci / 2)).bfloat16()
        st = {"x": x, "W": W, "bias": 0.1 * rnd(co), "dy": rnd(B, *g, co).bfloat16(),
              "Wt": W.flip(0).transpose(1, 2).contiguous(),
              "y": torch.empty(B, *g, co, dtype=torch.bfloat16, device="cuda"), "dx": torch.empty_like(x),
              "dW": torch.empty(27, co, ci, device="cuda")}
    elif kind == "batch":
        grids = [(int(n),) * 3 for n in case["grids"].split(",")]
        phis = [_octet(g, case["rho"] * (1 + 0.3 * k), seed + 1000 * k) for k, g in enumerate(grids)]
        torch.cuda.synchronize()
        st = {"ctxs": [hom.hom_create(g, p, hom.HOM_INPUT_FRACTION_F32, E_M, NU_M, device_ptrs=True)
                       for g, p in zip(grids, phis)],
              "macro": np.eye(6), "fields": [_fields_for(g, 6, torch.float32) for g in grids]}
    elif kind == "j2":
        g = _grid(case)
        phi = _octet(g, case["rho"], seed, torch.float64)
        torch.cuda.synchronize()
        st = {"ctx": hom.hom_create(g, phi, hom.HOM_INPUT_FRACTION_F64, E_P, NU_P, device_ptrs=True,
                                    precision=hom.HOM_PREC_FP64),
              "e11": -0.04 * (1 + 0.1 * float(np.random.default_rng(seed).random())),
              "strain": torch.empty((6,) + g, dtype=torch.float64, device="cuda"),
              "plastic": torch.empty((6,) + g, dtype=torch.float64, device="cuda"),
              "alpha": torch.empty(g, dtype=torch.float64, device="cuda")}
    else:
        g = _grid(case)
        f64 = case.get("precision") == "f64"
        dt = torch.float64 if f64 else torch.float32
        phi = _octet(g, case["rho"], seed, dt)
        rotated = case.get("scheme", "continuous") == "rotated"
        torch.cuda.synchronize()
        ctx = hom.hom_create(g, phi, hom.HOM_INPUT_FRACTION_F64 if f64 else hom.HOM_INPUT_FRACTION_F32, E_M, NU_M,
                             device_ptrs=True, precision=hom.HOM_PREC_FP64 if f64 else hom.HOM_PREC_FP32_FIELDS,
                             derivative=hom.HOM_DERIV_ROTATED if rotated else hom.HOM_DERIV_CONTINUOUS,
                             solver=hom.HOM_SOLVER_MODBFFT_CG if kind == "modbfft" else hom.HOM_SOLVER_GALERKIN_MINRES)
        strains = case.get("strains", 1)
        macro = np.eye(6) if strains == 6 else _unit_strain(seed)
        stress = None
        if case.get("control") == "uniaxial":
            macro, stress = np.zeros(6), np.zeros(6)
            stress[seed % 3] = 1e6
        st = {"ctx": ctx, "phi": phi, "macro": macro, "stress": stress, "fields": _fields_for(g, strains, dt)}
    st["case"] = case
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "noalloc":
        deriv = hom.HOM_DERIV_ROTATED if case["scheme"] == "rotated" else hom.HOM_DERIV_CONTINUOUS
        return hom.hom_apply_noalloc(_grid(case), st["phi"], st["eps"], st["out"], 1.0, NU_M, deriv,
                                     stream=torch.cuda.current_stream().cuda_stream)
    if kind == "conv":
        g, s = _grid(case), torch.cuda.current_stream().cuda_stream
        hnet.conv3d(g, st["x"], st["W"], case["cout"], bias=st["bias"], relu=True, out=st["y"], stream=s)
        hnet.conv3d(g, st["dy"], st["Wt"], case["cin"], out=st["dx"], stream=s)
        hnet.conv3d_wgrad(g, st["dy"], st["x"], st["dW"], stream=s)
        return {"y": st["y"], "dx": st["dx"], "dW": st["dW"]}
    if kind == "batch":
        hom.hom_solve_batch(st["ctxs"], st["macro"], tol=1e-6, max_it=case["max_it"])
        return [_read(c, f) for c, f in zip(st["ctxs"], st["fields"])]
    if kind == "j2":
        hom.hom_j2_begin(st["ctx"], Y_P, 0.0)
        hom.hom_j2_increment(st["ctx"], [st["e11"], 0, 0, 0, 0, 0], np.zeros(6), MASK_LATERAL,
                             max_newton=case["max_newton"], max_lin=case["max_lin"])
        hom.hom_j2_state(st["ctx"], st["strain"], st["plastic"], st["alpha"])
        return {"strain": st["strain"], "plastic": st["plastic"], "alpha": st["alpha"]}
    if st["stress"] is not None:
        hom.hom_solve_mixed(st["ctx"], st["macro"], st["stress"], 63, tol=1e-6, max_it=case["max_it"])
    else:
        hom.hom_solve(st["ctx"], st["macro"], tol=1e-6, max_it=case["max_it"])
    return _read(st["ctx"], st["fields"])


def _read(ctx, fields):
    for k, f in enumerate(fields):
        hom.hom_fields(ctx, k, want=tuple(f), **f)
    return fields


def work(case):
    kind = case["kind"]
    if kind == "conv":
        v = case["batch"] * case["n1"] * case["n2"] * case["n3"]
        ci, co = case["cin"], case["cout"]
        # y = conv x, dx = conv dy, dW from x and dy: x and dy in, y and dx out, weights in and out
        return {"bytes": 4.0 * v * (ci + co) + 27 * ci * co * 8.0, "flops": 3 * 2.0 * 27 * v * ci * co}

    def operator(v, n):   # two transforms of six real components, law and projector
        return v * (2 * 6 * 2.5 * math.log2(n) + 40 + 75)

    if kind == "batch":
        vs = [int(n) ** 3 for n in case["grids"].split(",")]
        return {"bytes": sum(6.0 * v * (196 * case["max_it"] + 24) for v in vs),
                "flops": sum(6.0 * operator(v, v) * case["max_it"] for v in vs)}
    v = case["n1"] * case["n2"] * case["n3"]
    if kind == "noalloc":
        return {"bytes": 52.0 * v, "flops": operator(v, v)}
    if kind == "j2":
        its = case["max_newton"] * case["max_lin"]
        # a MINRES iteration reads five fields and the 36 tangent coefficients and writes three
        return {"bytes": v * ((8 * 48 + 288.0) * its + 104), "flops": (operator(v, v) + 72 * v) * its}
    # a MINRES iteration reads five fields and phi and writes three; PCG on
    # displacements reads and writes fields of half as many components
    word = 2 if case.get("precision") == "f64" else 1
    per = (4 + 8 * 12) if kind == "modbfft" else 196
    n = case.get("strains", 1)
    return {"bytes": float(n * v * word * (per * case["max_it"] + 24)), "flops": n * operator(v, v) * case["max_it"]}


# ---------------------------------------------------------------------------
# The same results in 64 bits, from the equations
# ---------------------------------------------------------------------------
def _frequency_directions(grid, rotated):
    """Unit frequency vectors on the half spectrum and where the projector is nonzero."""
    n1, n2, n3 = grid
    k = [np.fft.fftfreq(n1, 1 / n1), np.fft.fftfreq(n2, 1 / n2), np.arange(n3 // 2 + 1, dtype=float)]
    shape = [(-1, 1, 1), (1, -1, 1), (1, 1, -1)]
    D, M, keep = [], [], True
    for p, n in enumerate(grid):
        q = torch.tensor(2 * np.pi * k[p] / n, device="cuda").reshape(shape[p])
        e = torch.exp(1j * q)
        D.append(n * (e - 1) if rotated else 1j * q * n)
        M.append((e + 1) / 2 if rotated else torch.ones_like(e))
        nyq = torch.tensor((n % 2 == 0) & (np.abs(2 * k[p]) == n), device="cuda").reshape(shape[p])
        keep = ~nyq & keep
    xi = torch.stack([D[0] * M[1] * M[2], M[0] * D[1] * M[2], M[0] * M[1] * D[2]])
    norm = xi.abs().square().sum(0).sqrt()
    keep = keep & (norm > 0)
    return torch.where(keep, xi / torch.where(keep, norm, 1.0), torch.zeros_like(xi)), keep


class _Galerkin:
    """A(e) = P(C : e) on Mandel fields; mask: stress-controlled components."""

    def __init__(self, grid, phi, rotated, mask=()):
        self.grid, self.phi, self.mask = tuple(grid), phi.double(), list(mask)
        self.e, _ = _frequency_directions(grid, rotated)
        self.lam, self.mu = NU_M / ((1 + NU_M) * (1 - 2 * NU_M)), 0.5 / (1 + NU_M)

    def law(self, e):
        t = 2 * self.mu * e
        t[:3] += self.lam * e[:3].sum(0)
        return self.phi * t

    def project(self, t):
        f = torch.fft.rfftn(t, dim=(1, 2, 3))
        mean, (e0, e1, e2) = f[:, 0, 0, 0].clone(), self.e
        c0, c1, c2 = self.e.conj()
        f[3:] /= SQ2
        v0 = f[0] * c0 + f[5] * c1 + f[4] * c2
        v1 = f[5] * c0 + f[1] * c1 + f[3] * c2
        v2 = f[4] * c0 + f[3] * c1 + f[2] * c2
        s = c0 * v0 + c1 * v1 + c2 * v2
        u0, u1, u2 = 2 * v0 - e0 * s, 2 * v1 - e1 * s, 2 * v2 - e2 * s
        f[0], f[1], f[2] = u0 * e0, u1 * e1, u2 * e2
        f[3], f[4], f[5] = ((u1 * e2 + u2 * e1) / SQ2, (u0 * e2 + u2 * e0) / SQ2, (u0 * e1 + u1 * e0) / SQ2)
        for c in self.mask:
            f[c, 0, 0, 0] = mean[c]
        return torch.fft.irfftn(f, s=self.grid, dim=(1, 2, 3))

    def minres(self, b, tol, max_it):
        dot = lambda a, c: float((a * c).sum())  # noqa: E731
        x, v0, w0, w1 = (torch.zeros_like(b) for _ in range(4))
        beta = beta1 = math.sqrt(dot(b, b))
        if beta1 == 0:
            return x
        v = b / beta
        c, s, dbar, eps, phi = -1.0, 0.0, 0.0, 0.0, beta1
        for _ in range(max_it):
            p = self.project(self.law(v))
            alpha = dot(v, p)
            p -= alpha * v + beta * v0
            beta_next = math.sqrt(dot(p, p))
            delta, gbar = c * dbar + s * alpha, s * dbar - c * alpha
            eps_next, dbar = s * beta_next, -c * beta_next
            gamma = max(math.hypot(gbar, beta_next), 1e-300)
            c, s = gbar / gamma, beta_next / gamma
            w0, w1 = w1, (v - delta * w1 - eps * w0) / gamma
            x += (c * phi) * w1
            phi, eps = s * phi, eps_next
            if phi <= tol * beta1 or beta_next == 0:
                break
            v0, v, beta = v, p / beta_next, beta_next
        return x


def _exact_fields(op, macro, sbar, max_it, strain=False):
    m = torch.tensor(macro, device="cuda", dtype=torch.float64)
    m = torch.cat([m[:3], SQ2 * m[3:]])
    for c in op.mask:
        m[c] = 0.0
    ebar = m.reshape(6, 1, 1, 1)
    t = op.law(ebar.expand((6,) + op.grid).clone())
    if sbar is not None:
        t = t - torch.tensor(sbar / E_M, device="cuda").reshape(6, 1, 1, 1)
    e = ebar + op.minres(-op.project(t), 5e-7, max_it)
    s = E_M * op.law(e.clone())
    scale = torch.tensor([1, 1, 1, 1 / SQ2, 1 / SQ2, 1 / SQ2], device="cuda", dtype=torch.float64).reshape(6, 1, 1, 1)
    return {"stress": s * scale, "strain": e * scale} if strain else {"stress": s * scale}


def exact(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        g = _grid(case)
        op = _Galerkin(g, _octet(g, 0.2, seed), case["scheme"] == "rotated")
        return op.project(op.law(torch.randn((6,) + g, generator=_gen(seed), device="cuda").double()))
    if kind == "conv":
        st = prepare(case, seed)
        x, W, dy = st["x"].double(), st["W"].double(), st["dy"].double()
        y, dx, dW = st["bias"].double().expand(dy.shape).clone(), torch.zeros_like(x), torch.zeros_like(W)
        for t in range(27):
            d = (t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1)
            xs = torch.roll(x, tuple(-k for k in d), (1, 2, 3))
            y += xs @ W[t].T
            dx += torch.roll(dy @ W[t], d, (1, 2, 3))
            dW[t] = dy.reshape(-1, dy.shape[-1]).T @ xs.reshape(-1, x.shape[-1])
        return {"y": y.relu(), "dx": dx, "dW": dW}
    if kind == "solve":
        g = _grid(case)
        if g[0] * g[1] * g[2] * case["strains"] > 8e6:   # over 20 seconds in 64 bits
            return None
        f64 = case["precision"] == "f64"
        phi = _octet(g, case["rho"], seed, torch.float64 if f64 else torch.float32)
        mixed = case["control"] == "uniaxial"
        op = _Galerkin(g, phi, case["scheme"] == "rotated", range(6) if mixed else ())
        sbar = None
        if mixed:
            sbar = np.zeros(6)
            sbar[seed % 3] = 1e6
        loads = np.eye(6) if case["strains"] == 6 else [np.zeros(6) if mixed else _unit_strain(seed)]
        return [_exact_fields(op, m, sbar, case["max_it"], f64) for m in loads]
    if kind == "batch":
        out = []
        for k, n in enumerate(case["grids"].split(",")):
            g = (int(n),) * 3
            op = _Galerkin(g, _octet(g, case["rho"] * (1 + 0.3 * k), seed + 1000 * k), True)
            out.append([_exact_fields(op, m, None, case["max_it"]) for m in np.eye(6)])
        return out
    # displacement solver, elastoplastic increment: over 20 seconds in 64 bits
    return None
