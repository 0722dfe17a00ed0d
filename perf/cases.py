"""Performance cases of the complex-coordinate FMM: what a program that solves integral equations
with this library asks of it, through the package's public entry points.

The geometries are the complexified curve (2D) and the complexified plane with a bump (3D) of the
repository's workloads, drawn from the seed. Most passes are one application of a resident plan (the
matvec of an iterative solver); some build the plan as well (a geometry that is used once), and two
are the differentiated apply and the direct sum.
"""
import math

import numpy as np
import torch

import paper_2509_05458_gb300 as cf


def _case(name, do, dim, kernel, layers, n, **more):
    c = {"name": name, "do": do, "dim": dim, "kernel": kernel, "layers": layers, "n": n, "targets": 0, "kappa": 0.0,
         "eps": 1e-6, "leaf": 64, "sep": 1 if dim == 2 else 2, "precision": "fp64", "nrhs": 1, "matvecs": 1}
    c.update(more)
    return c


def listed():
    return [
        # the smallest solves: a 2D electrostatics matvec, where launches and latency are the cost
        _case("lap2d_n4000", "apply", 2, "laplace", "s", 4000, leaf=32),
        # the matvec of GMRES on the 2D complex-scaled half-space equation (double layer, Green's constant)
        _case("bie2d_n3001", "apply", 2, "helmholtz", "d", 3001, kappa=5.0, eps=1e-10),
        # a short-lived request of a mixed stream: plan a small surface, apply it a few times, drop it
        _case("request_lap3d_n2500", "request", 3, "laplace", "s", 2500, eps=1e-3, precision="auto", matvecs=5),
        # the 2D Helmholtz workload as one step on a new geometry: plan and apply, combined field
        _case("helm2d_step_n100000", "step", 2, "helmholtz", "sd", 100000, kappa=20.0, precision="mixed"),
        # the same operator at the tighter accuracy, whole in FP64, on a resident plan
        _case("helm2d_fp64_n100000", "apply", 2, "helmholtz", "sd", 100000, kappa=20.0, eps=1e-9),
        # a long 2D line at moderate accuracy
        _case("lap2d_mixed_n700001", "apply", 2, "laplace", "sd", 700001, precision="mixed"),
        # the 3D Helmholtz surface matvec, mixed precision: the headline workload
        _case("helm3d_mixed_n1000000", "apply", 3, "helmholtz", "s", 1000000, kappa=10.0, leaf=256, precision="mixed"),
        # the same family in FP64
        _case("helm3d_fp64_n100003", "apply", 3, "helmholtz", "s", 100003, kappa=10.0, leaf=128),
        # several right-hand sides on one surface at a higher wavenumber
        _case("helm3d_rhs8_n20011", "apply", 3, "helmholtz", "s", 20011, kappa=15.0, leaf=128, precision="mixed", nrhs=8),
        # 3D Laplace potential of a surface at separate targets above it, FP64
        _case("lap3d_targets_n200000", "targets", 3, "laplace", "sd", 200000, targets=50007, leaf=128),
        # normal derivatives on a surface: potential and gradient
        _case("helm3d_grad_n30000", "grad", 3, "helmholtz", "s", 30000, kappa=6.0),
        # field of a solved 2D density at points off the curve: the direct sum
        _case("direct2d_n20000", "direct", 2, "helmholtz", "d", 20000, targets=3001, kappa=20.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    dim = rng.choice([2, 3])
    kernel = rng.choice(["laplace", "helmholtz"])
    do = rng.choice(["apply", "apply", "apply", "step", "request", "targets", "grad", "direct"])
    layers = "s" if do == "grad" else rng.choice(["s", "d", "sd"])
    eps = rng.choice([1e-3, 1e-6, 1e-6, 1e-9])
    precision = rng.choice(["fp64", "mixed"]) if eps > 1e-8 and do not in ("grad", "direct") else "fp64"
    kappa = 0.0 if kernel == "laplace" else round(rng.uniform(1.0, 30.0 if dim == 2 else 12.0), 3)
    leaf = rng.choice([32, 64, 100] if dim == 2 else [64, 128, 256])
    nrhs = rng.choice([1, 1, 1, 2, 5]) if do == "apply" else 1
    # sizes over the range that a pass of this kind has in use; FP64 and 3D ones end earlier
    top = {(2, "mixed"): 400000, (2, "fp64"): 150000, (3, "mixed"): 200000, (3, "fp64"): 60000}[dim, precision]
    if do in ("grad", "direct"):
        top = 30000
    if dim == 3 and eps < 1e-8:
        top = min(top, 30000)
    n = _log(rng, 1000, top // nrhs)
    targets = _log(rng, 500, max(1000, n)) if do in ("targets", "direct") else 0
    return {"do": do, "dim": dim, "kernel": kernel, "layers": layers, "n": n, "targets": targets, "kappa": kappa, "eps": eps,
            "leaf": leaf, "sep": 1 if dim == 2 else 2, "precision": precision, "nrhs": nrhs,
            "matvecs": rng.randint(2, 6) if do == "request" else 1}


# ---- inputs -----------------------------------------------------------------

def _halton(n, base, start):
    i = np.arange(start, start + n, dtype=np.int64)
    out, f = np.zeros(n), 1.0
    while i.any():
        f /= base
        out += f * (i % base)
        i //= base
    return out


def _curve(case, n, rng):
    """t -> (t + i 0.5 sign(t) max(|t| - 4, 0), h e^{-t^2}) and its normal (gamma_2', -gamma_1')."""
    half = 40.0 if case["n"] >= 20000 else 10.0
    h = rng.uniform(0.3, 1.0)
    t = rng.uniform(-half, half, n)
    y = h * np.exp(-t * t)
    zero = np.zeros(n)
    re, im = np.stack([t, y], 1), np.stack([0.5 * np.sign(t) * np.maximum(np.abs(t) - 4.0, 0.0), zero], 1)
    nr, ni = np.stack([-2.0 * t * y, zero - 1.0], 1), np.stack([zero, -0.5 * (np.abs(t) > 4.0)], 1)
    return re, im, nr, ni


def _surface(n, rng, height=0.0):
    """The plane over [-20, 20]^2 with a Gaussian bump, (x, y) complexified with slope 0.4 beyond rho = 6."""
    start = int(rng.integers(1, 100000))
    x, y = 40.0 * _halton(n, 2, start) - 20.0, 40.0 * _halton(n, 3, start) - 20.0
    z = 0.5 * np.exp(-(x * x + y * y))
    rho = np.maximum(np.hypot(x, y), 1e-300)
    f = 0.4 * np.maximum(rho - 6.0, 0.0) / rho
    re, im = np.stack([x, y, z + height], 1), np.stack([f * x, f * y, np.zeros(n)], 1)
    nr = np.stack([2.0 * x * z, 2.0 * y * z, np.ones(n)], 1)
    return re, im, nr, np.zeros((n, 3))


def _inputs(case, seed):
    """Sources, normals, separate targets and densities [matvecs][nrhs][ncomp][n], on the GPU."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n, m = case["n"], case["targets"]
    src = _curve(case, n, rng) if case["dim"] == 2 else _surface(n, rng)
    if not m:
        trg = (None, None)
    elif case["dim"] == 2:   # real points above the undeformed part of the curve
        re = np.stack([rng.uniform(-4.0, 4.0, m), rng.uniform(1.2, 4.0, m)], 1)
        trg = (re, np.zeros((m, 2)))
    else:                    # a parallel surface
        trg = _surface(m, rng, height=0.7)[:2]
    d = rng.standard_normal((case["matvecs"], case["nrhs"], len(case["layers"]), n, 2)).view(np.complex128)[..., 0]
    gpu = [None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*src, *trg, d)]
    return dict(zip(("re", "im", "nr", "ni", "tre", "tim", "dens"), gpu))


def _options(case):
    kernel = cf.HELMHOLTZ if case["kernel"] == "helmholtz" else cf.LAPLACE
    kernel |= (cf.SLP if "s" in case["layers"] else 0) | (cf.DLP if "d" in case["layers"] else 0)
    if case["layers"] == "d":
        kernel |= cf.GREEN_SCALE
    precision = {"fp64": cf.FP64, "mixed": cf.MIXED, "auto": cf.AUTO}[case["precision"]]
    return kernel, dict(leaf_size=case["leaf"], sep=case["sep"], precision=precision, top_level=cf.TOP_FIT)


def _plan(case, s):
    kernel, opts = _options(case)
    normals = (s["nr"], s["ni"]) if "d" in case["layers"] else (None, None)
    if case["do"] == "targets":
        return cf.plan_targets(case["dim"], kernel, case["kappa"], case["eps"], s["re"], s["im"], s["tre"], s["tim"],
                               *normals, **opts)
    return cf.plan(case["dim"], kernel, case["kappa"], case["eps"], s["re"], s["im"], *normals, **opts)


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    if case["do"] in ("apply", "targets", "grad"):
        s["plan"] = _plan(case, s)
    return s


def run(s):
    case, dens = s["case"], s["dens"]
    if case["do"] in ("apply", "targets"):
        return s["plan"].apply(dens[0])
    if case["do"] == "grad":
        return s["plan"].apply_grad(dens[0])
    if case["do"] == "direct":
        normals = (s["nr"], s["ni"]) if "d" in case["layers"] else (None, None)
        return cf.direct(case["dim"], _options(case)[0], case["kappa"], s["re"], s["im"], s["tre"], s["tim"], dens[0], *normals)
    p = _plan(case, s)       # step, request: the geometry is new
    return [p.apply(d) for d in dens]


# ---- work -------------------------------------------------------------------

def work(case):
    """Inputs read and outputs written once; the operations of the method: near pairs at the cost of one
    kernel value each, List-2 translations at the order of their level."""
    dim, n, m, k, leaf = case["dim"], case["n"], case["targets"], case["sep"], case["leaf"]
    ncomp, nrhs, passes = len(case["layers"]), case["nrhs"], case["matvecs"]
    out = m or n
    grad = 1 + dim if case["do"] == "grad" else 1
    points = (n + m) * 2 * dim + (n * 2 * dim if "d" in case["layers"] else 0)
    moved = 8 * points + passes * nrhs * 16 * (ncomp * n + grad * out)
    pair = {(2, "laplace"): 40, (2, "helmholtz"): 200, (3, "laplace"): 35, (3, "helmholtz"): 70}[dim, case["kernel"]]
    pair += 10 * (ncomp - 1) + (20 * dim if grad > 1 else 0) + 8 * ncomp * (nrhs - 1)
    if case["do"] == "direct":
        return {"bytes": moved, "flops": float(n) * m * pair}
    fill = 0.6 * leaf                                    # mean points of a leaf
    flops = passes * out * min(n, (2 * k + 1) ** (dim - 1) * fill) * pair
    width = 80.0 if dim == 2 and n >= 20000 else 20.0 if dim == 2 else 40.0
    ratio = (math.sqrt(dim) / 2.0) / (k + 0.5)
    base = math.log(10.0 / case["eps"]) / -math.log(ratio)
    boxes = 2 ** (dim - 1)
    while boxes * fill <= n + m:
        w = width / boxes ** (1.0 / (dim - 1))
        order = max(base, 0.7 * base + case["kappa"] * w)
        if order <= 63 or dim == 2:
            one = 8.0 * (2 * order + 1) ** 2 * (1 if case["kernel"] == "helmholtz" else 0.5) if dim == 2 else 17.0 * order ** 3
            flops += passes * nrhs * boxes * (2 ** (dim - 1) - 1) * (2 * k + 1) ** (dim - 1) * one
        boxes *= 2 ** (dim - 1)
    return {"bytes": moved, "flops": flops}


# ---- the direct sums in 64 bits ------------------------------------------------

_GAUSS = np.polynomial.hermite.hermgauss(96)


def _hankel(z):
    """H_0^(1), H_1^(1) of complex z, Re z > 0: the power series for |z| <= 5, beyond it
    K_nu(w) = sqrt(pi/(2w)) e^{-w} / Gamma(nu + 1/2) int e^{-u} u^{nu-1/2} (1 + u/(2w))^{nu-1/2} du at w = -iz,
    u = v^2, by Gauss-Hermite quadrature."""
    h0, h1 = torch.empty_like(z), torch.empty_like(z)
    small = z.abs() <= 5.0
    y = z[small]
    q, t = -0.25 * y * y, torch.ones_like(y)
    j0, a0, j1, a1, hk = t.clone(), torch.zeros_like(y), t.clone(), t.clone(), 0.0
    for i in range(1, 36):
        t = t * q / (i * i)                              # (-z^2/4)^i / (i!)^2
        hk += 1.0 / i
        j0 += t
        a0 += hk * t
        j1 += t / (i + 1)
        a1 += (2.0 * hk + 1.0 / (i + 1)) * t / (i + 1)
    lg = torch.log(0.5 * y) + np.euler_gamma
    h0[small] = j0 + 2j / math.pi * (lg * j0 - a0)
    h1[small] = 0.5 * y * j1 + 1j * (-2.0 / (math.pi * y) + 2.0 / math.pi * lg * 0.5 * y * j1 - y / (2.0 * math.pi) * a1)
    w = -1j * z[~small]
    k0, k1 = torch.zeros_like(w), torch.zeros_like(w)
    for x, g in zip(*_GAUSS):
        if x < 0.0 or g < 1e-30:
            continue
        root = torch.sqrt(1.0 + x * x / (2.0 * w))
        k0 += 2.0 * g / root
        k1 += 4.0 * g * x * x * root
    front = torch.sqrt(math.pi / (2.0 * w)) * torch.exp(-w) / math.sqrt(math.pi)
    h0[~small] = front * k0 * (2.0 / (math.pi * 1j))
    h1[~small] = front * k1 * (-2.0 / math.pi)
    return h0, h1


def _kernel(case, r2):
    """K(r) and K'(r)/r."""
    if case["kernel"] == "laplace":
        if case["dim"] == 2:
            return 0.5 * torch.log(r2), 1.0 / r2
        inv = 1.0 / torch.sqrt(r2)
        return inv, -inv / r2
    r = torch.sqrt(r2)
    kap = case["kappa"]
    if case["dim"] == 2:
        h0, h1 = _hankel(kap * r)
        return h0, -kap * h1 / r
    k = torch.exp(1j * kap * r) / r
    return k, k * (1j * kap * r - 1.0) / r2


def exact(case, seed):
    s = None
    pairs = case["n"] * (case["targets"] or case["n"])
    if pairs > (1.5e8 if case["dim"] == 2 and case["kernel"] == "helmholtz" else 1.1e10):
        return None
    s = _inputs(case, seed)
    x = torch.complex(s["re"], s["im"])
    t = x if s["tre"] is None else torch.complex(s["tre"], s["tim"])
    nu = torch.complex(s["nr"], s["ni"])
    scale = 1.0
    if case["layers"] == "d":
        scale = 1.0 / (4.0 * math.pi) if case["dim"] == 3 else 0.25j if case["kernel"] == "helmholtz" else -1.0 / (2.0 * math.pi)
    grad = case["do"] == "grad"
    u = [torch.zeros((case["nrhs"], t.shape[0]), dtype=torch.complex128, device="cuda") for _ in s["dens"]]
    g = torch.zeros((case["nrhs"], case["dim"], t.shape[0]), dtype=torch.complex128, device="cuda")
    rows = max(1, 20000000 // case["n"])
    for a in range(0, t.shape[0], rows):
        at = slice(a, a + rows)
        d = [t[at, i, None] - x[None, :, i] for i in range(case["dim"])]
        r2 = sum(v * v for v in d)
        same = sum(v.abs() for v in d) == 0
        r2[same] = 1.0
        k0, k1 = _kernel(case, r2)
        k0[same], k1[same] = 0.0, 0.0
        ops = ([k0] if "s" in case["layers"] else []) + \
              ([-k1 * sum(v * nu[None, :, i] for i, v in enumerate(d))] if "d" in case["layers"] else [])
        for out, dens in zip(u, s["dens"]):
            out[:, at] = scale * sum(dens[:, c] @ op.T for c, op in enumerate(ops))
        if grad:
            for i, v in enumerate(d):
                g[:, i, at] = s["dens"][0][:, 0] @ (k1 * v).T
    return (u[0], g) if grad else u if case["do"] in ("step", "request") else u[0]
