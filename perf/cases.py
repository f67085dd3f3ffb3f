"""What a user of this library has it do, as cases that can be timed.

A case is one call sequence through the public entry points on one body:

  step      build + solve + |E| on a new conductivity model (the headline step)
  solve     solve + |E| for another source on a body whose context is kept
  flux      facet fluxes -> edge potentials (tree-cotree), solve, |E|
  batch     several sources on one body in one batched solve
  group     bodies of different sizes solved by one group call
  gradient  the differentiable field energy, forward and backward
  post      |E| and its per-tissue 99th percentiles from a given potential
  host      build + solve + |E| between pinned host arrays in one call

Bodies are the ellipsoid phantom of ``spfd_inputs`` (the same ellipsoids in
fractions of the box, Voronoi tissues, log-uniform conductivities), made on
the GPU from the seed, homogeneous spheres, or random voxels with air between
(many separate components).  Sources are current loops outside the body, or a
uniform flux density for the largest grid.
"""

from __future__ import annotations

import math
import random
from fractions import Fraction

import numpy as np
import torch

import paper_2010_12879_gb300 as spfd
from paper_2010_12879_gb300.autograd import field_energy
from spfd_inputs.phantoms import BODY_ELLIPSOIDS
from spfd_inputs.sources_torch import loop_potential_t

OMEGA = 2.0 * math.pi * 85e3
BODY_HEIGHT = 1.792   # m: the body's box, 896 voxels of 2 mm
N_TISSUES, N_BLOBS = 40, 200
SIGMA_RANGE = (0.02, 2.0)
DEV = "cuda"
F64 = torch.float64


def _case(op, nx, ny, nz, body="body", precision="fp64", tol=1e-8, n=1, source="loop", name=None):
    c = {"op": op, "nx": nx, "ny": ny, "nz": nz, "body": body, "precision": precision,
         "tol": tol, "n": n, "source": source}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one more source on the 32^3 validation sphere; latency and launches
        _case("solve", 32, 32, 32, body="sphere", tol=1e-12, name="sphere_32_solve_fp64"),
        # a coarse body from scratch, as a parameter study on a coarse model runs it
        _case("step", 32, 20, 112, name="body_16mm_step_fp64"),
        # ragged grid with air between the voxels: many components, odd sizes on every level
        _case("solve", 45, 37, 29, body="random", tol=1e-12, name="random_islands_solve_fp64"),
        # measured fluxes to the field at the double-precision accuracy of 1e-12
        _case("flux", 128, 80, 448, tol=1e-12, name="body_4mm_flux_fp64"),
        # conductivity and source gradients for an inverse problem, forward and backward
        _case("gradient", 128, 96, 448, tol=1e-10, name="body_4mm_gradient_fp64"),
        # the headline workload, every operation in FP64
        _case("step", 256, 160, 896, name="body_2mm_step_fp64"),
        # the same with FP64 refinement around an FP32 solve
        _case("step", 256, 160, 896, precision="mixed", name="body_2mm_step_mixed"),
        # the largest grid: the body at 1 mm
        _case("step", 512, 320, 1792, precision="mixed", source="uniform", name="body_1mm_step_mixed"),
        # coil positions and orientations on one body
        _case("batch", 128, 80, 448, precision="mixed", n=8, name="body_4mm_batch8_mixed"),
        # twelve bodies of different sizes in one call
        _case("group", 192, 128, 640, precision="mixed", n=12, name="group_12_bodies_mixed"),
        # exposure assessment: |E| and the 99th percentile of every tissue
        _case("post", 256, 160, 896, name="body_2mm_percentiles"),
        # end to end between host arrays
        _case("host", 128, 80, 448, name="body_4mm_host_fp64"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _box(rng, lo, hi):
    """A body box of lo..hi voxels in height, its other sides near the body's proportions."""
    nz = int(round(_log(rng, lo, hi)))
    return (max(8, int(nz * 256 / 896 * rng.uniform(0.8, 1.1))),
            max(8, int(nz * 160 / 896 * rng.uniform(0.8, 1.1))), nz)


def draw(rng: random.Random):
    op = rng.choice(["step", "step", "solve", "solve", "flux", "batch", "group", "gradient",
                     "post", "host"])
    precision = rng.choice(["fp64", "mixed"])
    tol = rng.choice([1e-8, 1e-10, 1e-12] if op in ("step", "solve", "flux") else [1e-8, 1e-10])
    if op == "solve":
        kind = rng.choice(["sphere", "random", "body"])
        if kind == "sphere":
            n = int(round(_log(rng, 12, 80)))
            return _case(op, n, n, n, body="sphere", precision=precision, tol=tol)
        if kind == "random":
            d = [int(round(_log(rng, 6, 64))) for _ in range(3)]
            return _case(op, *d, body="random", precision="fp64", tol=1e-12)
    if op == "group":
        return _case(op, *_box(rng, 96, 480), precision=precision, tol=tol, n=rng.randint(2, 8))
    if op == "batch":
        return _case(op, *_box(rng, 64, 448), precision=precision, tol=tol, n=rng.randint(2, 12))
    if op in ("gradient", "host", "flux"):
        return _case(op, *_box(rng, 64, 448), precision=precision, tol=tol)
    if op == "post":
        return _case(op, *_box(rng, 64, 896))
    return _case(op, *_box(rng, 64, 896), precision=precision, tol=tol)


# ------------------------------------------------------------------ inputs
def _h(case):
    if case["body"] == "body":
        return BODY_HEIGHT / case["nz"]
    return 2e-3


def _origin(case, dims, h):
    nx, ny, nz = dims
    return (nx * h / 2, ny * h / 2, 0.0 if case["body"] == "body" else nz * h / 2)


def _centres(n):
    """Voxel centres as fractions of the box."""
    return (torch.arange(n, dtype=F64, device=DEV) + 0.5) / n


def _body(dims, rng):
    """sigma [nz][ny][nx] and int32 tissue labels (-1: air) of the ellipsoid body in its box."""
    nx, ny, nz = dims
    x, y, z = _centres(nx), _centres(ny), _centres(nz)
    wx, wy, wz = 0.512, 0.320, BODY_HEIGHT   # the box of the ellipsoids, m
    mask = torch.zeros((nz, ny, nx), dtype=torch.bool, device=DEV)
    for cx, cy, cz, a, b, c in BODY_ELLIPSOIDS:
        tx = (((x - 0.5) * wx - cx) / a) ** 2
        ty = (((y - 0.5) * wy - cy) / b) ** 2
        tz = ((z * wz - cz) / c) ** 2
        mask |= (tz[:, None, None] + ty[None, :, None] + tx[None, None, :]) <= 1.0
    # Voronoi tissues: blob centres among the body's voxels, the nearest one's tissue
    table = torch.from_numpy(np.exp(rng.uniform(math.log(SIGMA_RANGE[0]), math.log(SIGMA_RANGE[1]),
                                                N_TISSUES))).to(DEV)
    tissue = rng.integers(0, N_TISSUES, N_BLOBS)
    idx = mask.reshape(-1).nonzero().reshape(-1)
    pick = idx[torch.from_numpy((rng.random(N_BLOBS) * int(idx.numel())).astype(np.int64)).to(DEV)]
    blobs = torch.stack([(pick % nx + 0.5) / nx * wx, (pick // nx % ny + 0.5) / ny * wy,
                         (pick // (nx * ny) + 0.5) / nz * wz], 1).float()
    labels = torch.full((nz, ny, nx), -1, dtype=torch.int32, device=DEV)
    flat = labels.reshape(-1)
    tt = torch.from_numpy(tissue.astype(np.int32)).to(DEV)
    for part in idx.split(1 << 21):
        p = torch.stack([(part % nx + 0.5) / nx * wx, (part // nx % ny + 0.5) / ny * wy,
                         (part // (nx * ny) + 0.5) / nz * wz], 1).float()
        flat[part] = tt[(p @ blobs.t() * -2 + (blobs * blobs).sum(1)).argmin(1)]
    sigma = torch.where(labels >= 0, table[labels.clamp(min=0).long()], 0.0)
    return sigma.contiguous(), labels


def _sphere(dims, rng):
    r = [2 * _centres(n) - 1 for n in dims]
    inside = (r[2][:, None, None] ** 2 + r[1][None, :, None] ** 2 + r[0][None, None, :] ** 2
              <= (28.0 / 32.0) ** 2)
    return torch.where(inside, float(rng.uniform(0.1, 0.5)), 0.0).to(F64).contiguous(), None


def _random(dims, rng):
    nx, ny, nz = dims
    air = rng.random((nz, ny, nx)) < 0.9   # past percolation: hundreds of separate islands
    s = np.exp(rng.uniform(math.log(SIGMA_RANGE[0]), math.log(SIGMA_RANGE[1]), (nz, ny, nx)))
    s[air] = 0.0
    s[0, 0, 0] = 1.0
    return torch.from_numpy(s).to(DEV), None


def _sigma(case, dims, rng):
    return {"body": _body, "sphere": _sphere, "random": _random}[case["body"]](dims, rng)


def _uniform(dims, h, origin, B, out=None):
    """Edge potentials of the uniform flux density B in the symmetric gauge, B x r / 2."""
    nx, ny, nz = dims
    x, y, z = (torch.arange(n + 1, dtype=F64, device=DEV) * h - o for n, o in zip(dims, origin))
    X, Y, Z = x[None, None, :], y[None, :, None], z[:, None, None]
    a = torch.empty((3, nz + 1, ny + 1, nx + 1), dtype=F64, device=DEV) if out is None else out
    a[0] = 0.5 * h * (B[1] * Z - B[2] * Y)
    a[1] = 0.5 * h * (B[2] * X - B[0] * Z)
    a[2] = 0.5 * h * (B[0] * Y - B[1] * X)
    a[0, :, :, nx] = 0.0
    a[1, :, ny, :] = 0.0
    a[2, nz] = 0.0
    return a


def _potential(case, dims, h, rng, out=None):
    origin = _origin(case, dims, h)
    if case["body"] != "body" or case["source"] == "uniform":
        B = 27e-6 * rng.normal(size=3)
        return _uniform(dims, h, origin, [float(v) for v in B], out)
    centre = (float(rng.uniform(-0.5, 0.5)), float(rng.uniform(-0.5, 0.5)),
              float(rng.uniform(-0.6, -0.3)))
    normal = rng.normal(size=3)
    return loop_potential_t(dims, h, origin, center=centre, normal=[float(v) for v in normal],
                            device=DEV, out=out)


def _curl(a):
    """Facet fluxes b = C a, [3][nz+1][ny+1][nx+1] (facets that leave the grid: 0)."""
    b = torch.zeros_like(a)
    ax, ay, az = a
    b[0, :-1, :-1, :] = ay[:-1, :-1] + az[:-1, 1:] - ay[1:, :-1] - az[:-1, :-1]
    b[1, :-1, :, :-1] = az[:-1, :, :-1] + ax[1:, :, :-1] - az[:-1, :, 1:] - ax[:-1, :, :-1]
    b[2, :, :-1, :-1] = ax[:, :-1, :-1] + ay[:, :-1, 1:] - ax[:, 1:, :-1] - ay[:, :-1, :-1]
    return b


def _group_dims(case):
    """n boxes from 64 x 64 x 128 up to the case's, interpolated; a small case's start lower."""
    n, big = case["n"], (case["nx"], case["ny"], case["nz"])
    lo = tuple(min(s, max(8, b // 2)) for s, b in zip((64, 64, 128), big))
    return [tuple(int(round(s + i / max(1, n - 1) * (b - s))) for s, b in zip(lo, big))
            for i in range(n)]


def _precision(case):
    return spfd.SPFD_MIXED if case["precision"] == "mixed" else spfd.SPFD_FP64


def prepare(case, seed):
    rng = np.random.default_rng([int(seed), 2010])
    op, h = case["op"], _h(case)
    dims = (case["nx"], case["ny"], case["nz"])
    s = {"case": case, "h": h, "prec": _precision(case)}
    if op == "group":
        solvers, s["a"] = [], []
        for d in _group_dims(case):
            hd = BODY_HEIGHT / d[2]
            sigma, _ = _sigma(case, d, rng)
            solvers.append(spfd.Solver(sigma, hd, precision=s["prec"]))
            s["a"].append(_potential(case, d, hd, rng))
        s["solvers"], s["group"] = solvers, spfd.Group(solvers)
        return s
    sigma, labels = _sigma(case, dims, rng)
    if op == "batch":
        shape = (case["n"], 3, dims[2] + 1, dims[1] + 1, dims[0] + 1)
        s["a"] = torch.empty(shape, dtype=F64, device=DEV)
        for j in range(case["n"]):
            _potential(case, dims, h, rng, out=s["a"][j])
        s["solver"] = spfd.Solver(sigma, h, precision=s["prec"])
        return s
    a = _potential(case, dims, h, rng)
    if op == "flux":
        s["b"] = _curl(a)
    else:
        s["a"] = a
    if op == "step":
        s["sigma"] = sigma
    elif op in ("solve", "flux"):
        s["solver"] = spfd.Solver(sigma, h, precision=s["prec"])
    elif op == "gradient":
        s["sigma"] = sigma.requires_grad_()
        s["a"] = a.requires_grad_()
    elif op == "post":
        s["solver"] = spfd.Solver(sigma, h)
        s["labels"] = labels
        # a smooth node potential of the induced field's size
        nx, ny, nz = dims
        x, y, z = (torch.linspace(0, 1, n + 1, dtype=F64, device=DEV) for n in dims)
        k = [float(v) for v in rng.uniform(1, 6, 3)]
        psi = (torch.sin(k[2] * z)[:, None, None] + torch.cos(k[1] * y)[None, :, None]
               + torch.sin(k[0] * x)[None, None, :]) * float(s["a"].abs().max())
        s["psi"] = psi.contiguous()
    elif op == "host":
        def pinned(t):
            p = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
            p.copy_(t)
            return p
        nx, ny, nz = dims
        s["sigma"], s["a"] = pinned(sigma), pinned(a)
        s["psi"] = torch.empty((nz + 1, ny + 1, nx + 1), dtype=F64, pin_memory=True)
        s["E"] = torch.empty((nz, ny, nx), dtype=F64, pin_memory=True)
        s["opts"] = spfd.spfd_opts_default()
        s["opts"].precision = s["prec"]
    return s


# -------------------------------------------------------------------- pass
def run(s):
    case = s["case"]
    op, tol = case["op"], case["tol"]
    if op == "step":
        with spfd.Solver(s["sigma"], s["h"], precision=s["prec"]) as S:
            psi, _, _ = S.solve(s["a"], tol)
            return {"psi": psi, "E": S.efield(s["a"], psi, OMEGA)}
    if op == "solve":
        psi, _, _ = s["solver"].solve(s["a"], tol)
        return {"psi": psi, "E": s["solver"].efield(s["a"], psi, OMEGA)}
    if op == "flux":
        a = spfd.tree_cotree(s["b"])
        psi, _, _ = s["solver"].solve(a, tol)
        return {"a": a, "psi": psi, "E": s["solver"].efield(a, psi, OMEGA)}
    if op == "batch":
        psi, _, _ = s["solver"].solve_batch(s["a"], tol)
        return {"psi": psi}
    if op == "group":
        psis, _, _ = s["group"].solve(s["a"], tol)
        return {"psi": list(psis)}
    if op == "gradient":
        s["sigma"].grad = s["a"].grad = None
        J = field_energy(s["sigma"], s["a"], s["h"], OMEGA, tol, precision=s["prec"])
        J.backward()
        return {"J": J.detach(), "dsigma": s["sigma"].grad, "da": s["a"].grad}
    if op == "post":
        E = s["solver"].efield(s["a"], s["psi"], OMEGA)
        values, counts = s["solver"].percentile(E, s["labels"], N_TISSUES, 0.99)
        return {"E": E, "values": np.array(values), "counts": np.array(counts)}
    spfd.pipeline_host(s["sigma"], s["a"], s["h"], tol, OMEGA, s["psi"], s["E"], opts=s["opts"])
    return {"psi": s["psi"], "E": s["E"]}


# -------------------------------------------------------------------- work
def work(case):
    """Inputs read once and outputs written once; for a solve, one application of
    the 7-point operator (13 operations a node) for each decimal digit of tol."""
    def sizes(d):
        return d[0] * d[1] * d[2], (d[0] + 1) * (d[1] + 1) * (d[2] + 1)
    op = case["op"]
    nv, nn = sizes((case["nx"], case["ny"], case["nz"]))
    digits = -math.log10(case["tol"])
    if op == "group":
        nn = sum(sizes(d)[1] for d in _group_dims(case))
        return {"bytes": 32.0 * nn, "flops": 13.0 * nn * digits}
    if op == "batch":
        return {"bytes": 32.0 * nn * case["n"], "flops": 13.0 * nn * digits * case["n"]}
    if op == "gradient":
        return {"bytes": 48.0 * nn + 16.0 * nv, "flops": 26.0 * nn * digits}
    if op == "post":
        return {"bytes": 32.0 * nn + 12.0 * nv, "flops": 40.0 * nv}
    b = 32.0 * nn + 8.0 * nv
    if op == "flux":
        b += 24.0 * nn
    if op in ("step", "host"):
        b += 8.0 * nv
    return {"bytes": b, "flops": 13.0 * nn * digits}


# ------------------------------------------------- the same in plain 64 bits
def _conductances(sigma, h):
    """Edge conductances [3][nz+1][ny+1][nx+1]: h/4 times the sum of the voxels around an edge."""
    nz, ny, nx = sigma.shape
    s = torch.zeros((nz + 2, ny + 2, nx + 2), dtype=F64, device=sigma.device)
    s[1:-1, 1:-1, 1:-1] = sigma
    g = torch.zeros((3, nz + 1, ny + 1, nx + 1), dtype=F64, device=sigma.device)
    g[0, :, :, :nx] = (s[:-1, :-1, 1:-1] + s[:-1, 1:, 1:-1] + s[1:, :-1, 1:-1] + s[1:, 1:, 1:-1])
    g[1, :, :ny, :] = (s[:-1, 1:-1, :-1] + s[:-1, 1:-1, 1:] + s[1:, 1:-1, :-1] + s[1:, 1:-1, 1:])
    g[2, :nz] = (s[1:-1, :-1, :-1] + s[1:-1, :-1, 1:] + s[1:-1, 1:, :-1] + s[1:-1, 1:, 1:])
    return g * (h / 4)


def _grad(p):
    """G p: head minus tail on every edge slot (0 past the last node)."""
    u = torch.zeros((3,) + tuple(p.shape), dtype=F64, device=p.device)
    u[0, :, :, :-1] = p[:, :, 1:] - p[:, :, :-1]
    u[1, :, :-1] = p[:, 1:] - p[:, :-1]
    u[2, :-1] = p[1:] - p[:-1]
    return u


def _div(w):
    """G^T w: entering minus leaving edges of every node."""
    d = -(w[0] + w[1] + w[2])
    d[:, :, 1:] += w[0, :, :, :-1]
    d[:, 1:] += w[1, :, :-1]
    d[1:] += w[2, :-1]
    return d


class _System:
    """The discrete Poisson system on the node grid, solved by plain Jacobi-CG."""

    def __init__(self, sigma, h):
        self.g = _conductances(sigma, h)
        self.diag = self.g.sum(0)
        self.diag[:, :, 1:] += self.g[0, :, :, :-1]
        self.diag[:, 1:] += self.g[1, :, :-1]
        self.diag[1:] += self.g[2, :-1]
        self.on = self.diag > 0
        lab = torch.arange(self.diag.numel(), device=sigma.device).reshape(self.diag.shape)
        lab = torch.where(self.on, lab, -1)
        while True:  # each component takes its smallest node number
            old = lab.clone()
            for d, ax in ((0, 2), (1, 1), (2, 0)):
                n = lab.shape[ax]
                lo, hi = lab.narrow(ax, 0, n - 1), lab.narrow(ax, 1, n - 1)
                link = self.g[d].narrow(ax, 0, n - 1) > 0
                m = torch.minimum(lo, hi)
                lo.copy_(torch.where(link, m, lo))
                hi.copy_(torch.where(link, torch.minimum(m, hi), hi))
            flat = lab.reshape(-1)
            jump = torch.where(flat >= 0, flat[flat.clamp(min=0)], -1)
            lab = jump.reshape(lab.shape)
            if torch.equal(lab, old):
                break
        ids, inv = torch.unique(lab[self.on], return_inverse=True)
        self.comp = inv
        self.size = torch.bincount(inv, minlength=ids.numel()).to(F64)

    def project(self, v):
        x = v[self.on]
        mean = torch.zeros_like(self.size).index_add_(0, self.comp, x) / self.size
        out = torch.zeros_like(v)
        out[self.on] = x - mean[self.comp]
        return out

    def apply(self, p):
        return _div(self.g * _grad(p))

    def solve(self, b):
        b = self.project(b)
        dinv = torch.where(self.on, 1.0 / self.diag.clamp(min=1e-300), 0.0)
        bb = float(b.norm())
        x = torch.zeros_like(b)
        if bb == 0.0:
            return x
        # restarted from its true residual, so that it ends at rounding level
        for target in (1e-10, 1e-4, 1e-2):
            r = self.project(b - self.apply(x))
            r0 = float(r.norm())
            if r0 <= 1e-15 * bb:
                break
            z = dinv * r
            p = z.clone()
            rz = (r * z).sum()
            dx = torch.zeros_like(x)
            for it in range(1, 40000):
                q = self.apply(p)
                alpha = rz / (p * q).sum()
                dx += alpha * p
                r -= alpha * q
                z = dinv * r
                new = (r * z).sum()
                if it % 25 == 0 and float(r.norm()) <= target * r0:
                    break
                p = z + (new / rz) * p
                rz = new
            x = self.project(x + dx)
        return x


def _field(sigma, h, u):
    """The three voxel-averaged components of omega u / h."""
    c = OMEGA / (4 * h)
    ex = u[0, :-1, :-1, :-1] + u[0, 1:, :-1, :-1] + u[0, :-1, 1:, :-1] + u[0, 1:, 1:, :-1]
    ey = u[1, :-1, :-1, :-1] + u[1, 1:, :-1, :-1] + u[1, :-1, :-1, 1:] + u[1, 1:, :-1, 1:]
    ez = u[2, :-1, :-1, :-1] + u[2, :-1, 1:, :-1] + u[2, :-1, :-1, 1:] + u[2, :-1, 1:, 1:]
    return torch.where(sigma > 0, torch.stack([ex, ey, ez]) * c, 0.0)


def _gauge(b, j0, k0):
    """The potentials with a = 0 on the comb tree of root line (j0, k0), by prefix sums."""
    a = torch.zeros_like(b)
    bx, by, bz = b
    row = torch.zeros_like(a[0, k0])
    row[j0 + 1:, :-1] = -torch.cumsum(bz[k0, j0:-1, :-1], 0)
    row[:j0, :-1] = torch.cumsum(bz[k0, :j0, :-1].flip(0), 0).flip(0)
    a[0, k0] = row
    a[0, k0 + 1:, :, :-1] = row[None, :, :-1] + torch.cumsum(by[k0:-1, :, :-1], 0)
    a[0, :k0, :, :-1] = row[None, :, :-1] - torch.cumsum(by[:k0, :, :-1].flip(0), 0).flip(0)
    a[1, k0 + 1:, :-1] = -torch.cumsum(bx[k0:-1, :-1], 0)
    a[1, :k0, :-1] = torch.cumsum(bx[:k0, :-1].flip(0), 0).flip(0)
    return a


def exact(case, seed):
    op, h = case["op"], _h(case)
    dims = (case["nx"], case["ny"], case["nz"])
    nn = (dims[0] + 1) * (dims[1] + 1) * (dims[2] + 1)
    # plain CG on more than this takes over 20 seconds
    if op == "group" or (op != "post" and nn * (2 if op == "gradient" else case["n"]) > 12_000_000):
        return None
    rng = np.random.default_rng([int(seed), 2010])
    sigma, labels = _sigma(case, dims, rng)
    if op == "batch":
        sources = [_potential(case, dims, h, rng) for _ in range(case["n"])]
        A = _System(sigma, h)
        return {"psi": torch.stack([A.solve(_div(A.g * a).neg()) for a in sources])}
    a = _potential(case, dims, h, rng)
    if op == "post":
        s = prepare(case, seed)
        E = _field(sigma, h, s["a"] + _grad(s["psi"])).square().sum(0).sqrt()
        e, lab = E[sigma > 0], labels[sigma > 0]
        values, counts = [], []
        for t in range(N_TISSUES + 1):
            v = torch.sort(e[lab == t] if t < N_TISSUES else e).values
            n = int(v.numel())
            counts.append(n)
            values.append(float(v[max(1, math.ceil(Fraction(0.99) * n)) - 1]) if n else math.nan)
        return {"E": E, "values": np.array(values), "counts": np.array(counts)}
    A = _System(sigma, h)
    out = {}
    if op == "flux":
        a = _gauge(_curl(a), dims[1] // 2, dims[2] // 2)
        out["a"] = a
    psi = A.solve(_div(A.g * a).neg())
    if op != "gradient":
        out["psi"] = psi
        out["E"] = _field(sigma, h, a + _grad(psi)).square().sum(0).sqrt()
        return out
    u = (a + _grad(psi)).requires_grad_()
    J = _field(sigma, h, u).square().sum() / (sigma > 0).sum()
    (gJ,) = torch.autograd.grad(J, u)
    for d, ax in ((0, 2), (1, 1), (2, 0)):  # slots past the last node hold no edge
        gJ[d].narrow(ax, gJ.shape[ax + 1] - 1, 1).zero_()
    lam = _grad(A.solve(_div(gJ)))
    sig = sigma.clone().requires_grad_()
    (ds,) = torch.autograd.grad(-(_conductances(sig, h) * lam * u.detach()).sum(), sig)
    return {"J": J.detach(), "dsigma": torch.where(sigma > 0, ds, 0.0), "da": gJ - A.g * lam}
