"""The performance cases of libclusterspec: what a Kohn-Sham program has it do, through the
package's public calls.

A case is one call (or the few calls that always go together) on one basis, grid and block
size. `listed()` holds the standing ones, `draw()` makes more over the same ranges, `exact()`
restates each result in plain 64-bit torch.

Inputs follow the library's own workloads: clusters of pseudo-atoms -4 erf(r/0.8)/r placed at
random with a minimum separation of 3.5 bohr, Gaussian s and p projectors, blocks of states
whose coefficients fall off with their kinetic energy as those of a filtered block do.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1404_3773_gb300 as cs

DEVICE = "cuda:0"
PRECISION = {"fp64": cs.CS_FP64, "fp32": cs.CS_FP32, "mixed": cs.CS_MIXED_BF16,
             "df64": cs.CS_DF64, "sliced": cs.CS_FP64_SLICED}
F32 = ("fp32", "mixed")

# basis R / lmax / nmax / grid n_r x n_theta x n_phi of the library's standing workloads
BALL = dict(R=8.0, lmax=10, nmax=16, n_r=32, n_theta=22, n_phi=42, natoms=2)
CLUSTER = dict(R=14.0, lmax=30, nmax=48, n_r=96, n_theta=60, n_phi=120, natoms=32)
LARGE = dict(R=26.0, lmax=60, nmax=96, n_r=192, n_theta=120, n_phi=240, natoms=120)


def listed():
    return [
        # One H X of the smallest basis: a solver's inner call, all launches and latency.
        dict(name="apply_fp64_ball", op="apply", prec="fp64", n_s=16, pad=0, kb=False, **BALL),
        # The reference precision (the library's default) on an ordinary cluster block.
        dict(name="apply_fp64_cluster", op="apply", prec="fp64", n_s=80, pad=0, kb=False,
             **CLUSTER),
        # FP64-class H X on the FP32 pipe: what Rayleigh-Ritz projects in production.
        dict(name="apply_df64_cluster", op="apply", prec="df64", n_s=80, pad=0, kb=False,
             **CLUSTER),
        # Mixed-precision H X, one step of the production filter.
        dict(name="apply_mixed_cluster", op="apply", prec="mixed", n_s=80, pad=0, kb=False,
             **CLUSTER),
        # The same at scale: one 128-state chunk of a large cluster with projectors.
        dict(name="apply_mixed_large_kb", op="apply", prec="mixed", n_s=128, pad=0, kb=True,
             **LARGE),
        # A whole Chebyshev filter pass in FP32.
        dict(name="filter_fp32_cluster", op="filter", prec="fp32", n_s=80, pad=0, kb=False,
             degree=16, **CLUSTER),
        # A whole filter pass in mixed precision on an odd, ragged basis with a padded block.
        dict(name="filter_mixed_odd", op="filter", prec="mixed", n_s=53, pad=5, kb=False,
             degree=8, R=12.5, lmax=23, nmax=42, n_r=84, n_theta=47, n_phi=92, natoms=21),
        # Orthonormalisation of a filtered block.
        dict(name="cholqr_cluster", op="cholqr", dense="df64", n_s=80, pad=0, **CLUSTER),
        # Rayleigh-Ritz of a cluster block: H X, projection, eigensolve, rotations, residuals.
        dict(name="ritz_cluster", op="ritz", prec="df64", dense="df64", n_s=80, pad=0, kb=False,
             **CLUSTER),
        # Rayleigh-Ritz of a large cluster's whole block, slice-product dense steps.
        dict(name="ritz_large", op="ritz", prec="df64", dense="sliced", n_s=880, pad=0, kb=False,
             **LARGE),
        # Many small clusters of uneven size filtered together.
        dict(name="batch_fp32", op="batch", prec="fp32", count=10, sizes=4000, degree=8),
        # What an SCF iteration does after the eigensolve: density, Hartree, LDA.
        dict(name="fields_cluster", op="fields", n_s=80, pad=0, **CLUSTER),
    ]


# ---------------------------------------------------------------------- drawn cases
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# cost of one flop of each arithmetic relative to FP64 (only bounds the drawn sizes)
_WEIGHT = {"fp64": 1.0, "df64": 0.3, "fp32": 0.04, "mixed": 0.02}
_MOST = 1.5e11


def draw(rng):
    op = rng.choice(["apply"] * 5 + ["filter"] * 3 + ["cholqr", "ritz", "ritz", "batch", "fields"])
    if op == "batch":
        return dict(op=op, prec=rng.choice(["fp32", "fp32", "mixed"]), count=rng.randint(4, 10),
                    sizes=rng.randint(5000, 9999), degree=rng.choice([6, 8, 10]))
    lmax = _log_int(rng, 6, 60)
    nmax = min(96, max(8, int(round(lmax * rng.uniform(1.4, 2.0)))))
    natoms = max(1, int(round(0.035 * lmax * lmax * rng.uniform(0.6, 1.0))))
    R = round(6.0 + lmax / 3.0 + rng.uniform(0.0, 2.0), 3)
    n_theta = lmax + 2 + rng.randint(lmax // 2, lmax)
    n_phi = 2 * (lmax + 1 + rng.randint(lmax // 2, lmax))
    if lmax > 31:  # the large bases are run on grids whose phi count is a multiple of four
        n_phi += n_phi % 4
        n_theta = min(n_theta, 127)
    c = dict(op=op, n_s=_log_int(rng, 3, 200), pad=rng.choice([0, 0, 1, 8]), R=R, lmax=lmax,
             nmax=nmax, n_r=2 * nmax + rng.randint(-2, 3), n_theta=n_theta, n_phi=n_phi,
             natoms=natoms)
    if op in ("apply", "filter"):
        c["prec"] = rng.choice(["fp64", "df64", "fp32", "mixed", "mixed"])
        c["kb"] = c["prec"] != "df64" and natoms <= 40 and rng.random() < 0.25
    if op == "filter":
        c["degree"] = rng.randint(4, 16) if c["prec"] != "mixed" else rng.randint(4, 8)
    if op == "ritz":
        c["prec"], c["dense"] = rng.choice([("df64", "df64"), ("df64", "sliced"), ("fp64", "fp64")])
        c["kb"] = False
    if op == "cholqr":
        c["dense"] = rng.choice(["fp64", "df64", "sliced"])
    if op in ("cholqr", "ritz"):
        c["n_s"] = min(c["n_s"], (lmax + 1) ** 2 * nmax // 8)
    while c["n_s"] > 1 and _cost(c) > _MOST:
        c["n_s"] = max(1, c["n_s"] * 2 // 3)
    return c


def _cost(c):
    return work(c)["flops"] * _WEIGHT.get(c.get("prec", "fp64"), 1.0)


# ---------------------------------------------------------------------- inputs
def _clusters(case):
    """The uneven clusters of a batch: sizes from the case, as the library's batch workload."""
    out = []
    for i in range(case["count"]):
        rng = random.Random(case["sizes"] * 1000 + i)
        natoms = rng.randint(4, 48)
        r_place = 1.75 * (natoms / 0.15) ** (1.0 / 3.0) - 1.75
        rmin = max(8.0, r_place + 6.0)
        R = rng.uniform(rmin, 16.0) if rmin < 16.0 else 16.0
        lmax = int(round(12 + 20 * (R - 8.0) / 8.0))
        nmax = int(round(24 + 32 * (R - 8.0) / 8.0))
        out.append(dict(R=R, lmax=lmax, nmax=nmax, n_r=2 * nmax, n_theta=2 * lmax,
                        n_phi=4 * lmax, natoms=natoms, n_s=min(128, math.ceil(2.4 * natoms)),
                        pad=0, kb=False, prec=case["prec"], degree=case["degree"]))
    return out


def _atoms(c, seed):
    """natoms points in the ball, at least 3.5 bohr apart (less where they would not fit)."""
    rng = np.random.default_rng(seed * 7919 + 1)
    r_place = max(1.0, c["R"] - 6.0 if c["R"] < 20.0 else c["R"] - 8.0)
    sep = min(3.5, 1.1 * r_place / c["natoms"] ** (1.0 / 3.0))
    kept = np.zeros((0, 3))
    while len(kept) < c["natoms"]:
        p = rng.normal(size=3)
        p *= r_place * rng.random() ** (1.0 / 3.0) / np.linalg.norm(p)
        if not len(kept) or np.min(np.sum((kept - p) ** 2, axis=1)) >= sep * sep:
            kept = np.vstack([kept, p])
    return kept


def _points(r, t, phi):
    """(n_r, n_theta, n_phi, 3) Cartesian grid points on the device."""
    r, t, phi = (torch.as_tensor(np.asarray(v), dtype=torch.float64, device=DEVICE)
                 for v in (r, t, phi))
    s = torch.sqrt(1.0 - t * t)
    x = r[:, None, None] * s[None, :, None] * torch.cos(phi)
    y = r[:, None, None] * s[None, :, None] * torch.sin(phi)
    z = (r[:, None, None] * t[None, :, None]).expand_as(x)
    return torch.stack([x, y, z], dim=-1)


def _potential(xyz, atoms):
    v = torch.zeros(xyz.shape[:3], dtype=torch.float64, device=DEVICE)
    for a in torch.as_tensor(atoms, device=DEVICE):
        r = torch.linalg.vector_norm(xyz - a, dim=-1).clamp_min(1e-6)
        v -= 4.0 * torch.erf(r / 0.8) / r
    return v


def _projector_values(xyz, atom):
    """Gaussian s, px, py, pz functions of one atom (width 1, unit norm): (4, grid)."""
    dx = xyz - torch.as_tensor(atom, device=DEVICE)
    g = torch.exp(-0.5 * torch.sum(dx * dx, dim=-1))
    s, p = math.pi ** -0.75, (math.pi ** 1.5 / 2.0) ** -0.5
    return torch.stack([s * g] + [p * dx[..., i] * g for i in range(3)])


def _couplings(natoms):
    return np.tile(np.array([1.0, 0.5, 0.5, 0.5]), natoms)


def _bounds(c, half_lambda, v):
    """Filter interval [a, b] and scaling point a0, as a program's first pass sets them."""
    a0 = 0.5 * float(v.min())
    b = float(half_lambda.max()) + (4.0 if c["kb"] else 1.0)
    return a0 + (b - a0) / 10.0, b, a0


def _block(c, half_lambda, seed, dtype=torch.float64):
    """(n_s, d + pad) block: Gaussian coefficients that fall off with kinetic energy, each
    state with a range of its own (0.5 to 8 Hartree), normalised."""
    g = torch.Generator(device=DEVICE).manual_seed(seed * 2 + 1)
    n_s, d = c["n_s"], half_lambda.numel()
    X = torch.zeros((n_s, d + c["pad"]), dtype=torch.float64, device=DEVICE)
    for s in range(n_s):
        e = 0.5 * 16.0 ** (s / max(1, n_s - 1))
        X[s, :d] = torch.randn(d, dtype=torch.float64, device=DEVICE, generator=g) \
            / (1.0 + half_lambda / e)
    X /= torch.linalg.vector_norm(X, dim=1, keepdim=True)
    return X.to(dtype)


def _orthonormal(X, d):
    """One Cholesky-QR pass of rows (a well-conditioned block) in plain torch."""
    A = X[:, :d]
    L = torch.linalg.cholesky(A @ A.T)
    X[:, :d] = torch.linalg.solve_triangular(L, A, upper=False)
    return X


def _context(c, seed):
    """Context with its potential (and projectors), and what the inputs need of it."""
    ctx = cs.cs_basis_init(c["R"], c["lmax"], c["nmax"], c["n_r"], c["n_theta"], c["n_phi"])
    r, _, t, _, phi = cs.cs_grid(ctx)
    atoms = _atoms(c, seed)
    xyz = _points(r, t, phi)
    v = _potential(xyz, atoms)
    cs.cs_set_potential(ctx, v)
    if c.get("kb"):
        P = torch.empty((4 * len(atoms), ctx.d), dtype=torch.float64, device=DEVICE)
        for i in range(0, len(atoms), 4):
            g = torch.cat([_projector_values(xyz, a) for a in atoms[i:i + 4]])
            cs.cs_forward_transform(ctx, g, P[4 * i:4 * i + len(g)])
        cs.cs_set_projectors(ctx, P, _couplings(len(atoms)))
    hl = torch.as_tensor(cs.cs_kinetic(ctx), device=DEVICE)
    return ctx, v, hl


def prepare(case, seed):
    c, op = case, case["op"]
    if op == "batch":
        ctxs, X0, bounds = [], [], []
        for i, k in enumerate(_clusters(c)):
            ctx, v, hl = _context(k, seed + 97 * i)
            ctxs.append(ctx)
            X0.append(_block(k, hl, seed + 97 * i, torch.float32))
            bounds.append(_bounds(k, hl, v))
        batch = cs.cs_batch_create(ctxs, [x.shape[0] for x in X0], c["degree"])
        cs.cs_batch_set_variant(batch, "concurrent")
        if c["prec"] == "mixed":
            cs.cs_batch_set_precision(batch, cs.CS_MIXED_BF16)
        return dict(op=op, batch=batch, X0=X0, X=[torch.empty_like(x) for x in X0],
                    bounds=tuple(zip(*bounds)))
    ctx, v, hl = _context(c, seed)
    s = dict(op=op, ctx=ctx, case=dict(c))
    if op in ("cholqr", "ritz"):
        cs.cs_set_dense_precision(ctx, PRECISION[c["dense"]])
    if op in ("apply", "filter"):
        s["X0"] = _block(c, hl, seed, torch.float32 if c["prec"] in F32 else torch.float64)
        s["out"] = torch.zeros_like(s["X0"])
        if op == "filter":
            s["bounds"] = _bounds(c, hl, v)
    elif op == "cholqr":
        s["X0"] = _block(c, hl, seed)
        s["out"] = torch.empty_like(s["X0"])
    elif op == "ritz":
        cs.cs_set_rr_precision(ctx, PRECISION[c["prec"]])
        s["X0"] = _orthonormal(_block(c, hl, seed), ctx.d)
        s["out"] = torch.empty_like(s["X0"])
        s["hx"] = torch.zeros_like(s["X0"])
        s["theta"] = torch.empty(c["n_s"], dtype=torch.float64, device=DEVICE)
        s["resid"] = torch.empty_like(s["theta"])
    elif op == "fields":
        s["X0"] = _block(c, hl, seed)
        s["occ"] = _occupations(c)
        shape = (c["n_r"], c["n_theta"], c["n_phi"])
        s.update({k: torch.empty(shape, dtype=torch.float64, device=DEVICE)
                  for k in ("rho", "vh", "exc", "vxc")})
    return s


def _occupations(c):
    i = torch.arange(c["n_s"], dtype=torch.float64, device=DEVICE)
    return 1.0 / (1.0 + torch.exp((i - 0.8 * c["n_s"]) / (0.05 * c["n_s"] + 0.5)))


def run(state):
    s, op = state, state["op"]
    if op == "batch":  # filters in place: the program's blocks are filled first
        torch._foreach_copy_(s["X"], s["X0"])
        a, b, a0 = s["bounds"]
        cs.cs_batch_cheb_filter(s["batch"], s["X"], a, b, a0)
        return s["X"]
    ctx, c = s["ctx"], s["case"]
    if op == "apply":
        cs.cs_apply_H(ctx, s["X0"], s["out"], PRECISION[c["prec"]])
        return s["out"][:, :ctx.d]
    if op == "fields":
        cs.cs_density(ctx, s["X0"], s["occ"], s["rho"])
        cs.cs_hartree(ctx, s["rho"], s["vh"])
        cs.cs_lda_xc(ctx, s["rho"], s["exc"], s["vxc"])
        return {k: s[k] for k in ("rho", "vh", "exc", "vxc")}
    s["out"].copy_(s["X0"])  # the calls below work in place
    if op == "filter":
        a, b, a0 = s["bounds"]
        cs.cs_cheb_filter(ctx, s["out"], c["degree"], a, b, a0, PRECISION[c["prec"]])
        return s["out"][:, :ctx.d]
    if op == "cholqr":
        cs.cs_cholqr(ctx, s["out"])
        return s["out"][:, :ctx.d]
    cs.cs_rayleigh_ritz(ctx, s["out"], s["theta"], s["resid"], s["hx"])
    return {"theta": s["theta"], "resid": s["resid"], "X": s["out"][:, :ctx.d],
            "HX": s["hx"][:, :ctx.d]}


# ---------------------------------------------------------------------- work
def _apply_flops(c, n_s):
    """H X of n_s states: radial products, parity-folded Legendre sums, real-FFT phi
    transforms, the potential and the projector pair."""
    L2, grid = (c["lmax"] + 1) ** 2, c["n_r"] * c["n_theta"] * c["n_phi"]
    one = 2 * c["n_r"] * c["nmax"] * L2 + c["n_theta"] * L2 * c["n_r"] \
        + 2.5 * math.log2(c["n_phi"]) * grid
    kb = 4.0 * L2 * c["nmax"] * 4 * c["natoms"] if c.get("kb") else 0.0
    return n_s * (2.0 * one + grid + kb)


def work(case):
    c, op = case, case["op"]
    if op == "batch":
        parts = [work(dict(k, op="filter")) for k in _clusters(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    d = (c["lmax"] + 1) ** 2 * c["nmax"]
    grid = c["n_r"] * c["n_theta"] * c["n_phi"]
    n = c["n_s"]
    size = 4 if c.get("prec") in F32 else 8
    if op in ("apply", "filter"):
        pairs = 4 * c["natoms"] * d if c["kb"] else 0
        return {"bytes": float(size * (2 * d * n + grid + pairs)),
                "flops": float(_apply_flops(c, n) * c.get("degree", 1))}
    if op == "cholqr":  # two passes of a symmetric Gram matrix and a triangular rotation
        return {"bytes": float(8 * 2 * d * n), "flops": 4.0 * d * n * n}
    if op == "ritz":  # H X, symmetric projection, two rotations
        return {"bytes": float(8 * (3 * d * n + grid)),
                "flops": _apply_flops(c, n) + 5.0 * d * n * n}
    half = 0.5 * _apply_flops(c, 1)  # fields: one synthesis per state, one H X for Hartree
    return {"bytes": float(8 * (d * n + 4 * grid)),
            "flops": n * (half + 3.0 * grid) + 2.0 * half}


# ---------------------------------------------------------------------- 64-bit restatement
def _sph_jn(l, x):
    """Spherical Bessel function j_l (numpy or torch array x > 0): upward recurrence above the
    turning point, Miller's downward recurrence normalised by j_0 or j_1 below it."""
    lib = torch if isinstance(x, torch.Tensor) else np
    up = lib.clip(x, max(l, 1e-3), None)
    a, b = lib.sin(up) / up, lib.sin(up) / up ** 2 - lib.cos(up) / up
    for i in range(1, l):
        a, b = b, (2 * i + 1) / up * b - a
    high = a if l == 0 else b
    if l == 0:
        return lib.sin(x) / x
    low_x = lib.clip(x, 1e-8, max(l, 1e-3))
    f1, f0 = lib.zeros_like(x), lib.ones_like(x) * 1e-200
    keep = lib.zeros_like(x)
    for i in range(l + 60, 0, -1):  # f0 holds order i
        if i == l:
            keep = f0
        if i == 1:
            one = f0
        f1, f0 = f0, (2 * i + 1) / low_x * f0 - f1
        big = lib.abs(f0) > 1e150
        scale = lib.where(big, lib.ones_like(x) * 1e-150, lib.ones_like(x))
        f1, f0, keep = f1 * scale, f0 * scale, keep * scale
        if i == 1:
            one = one * scale
    j0 = lib.sin(low_x) / low_x
    j1 = lib.sin(low_x) / low_x ** 2 - lib.cos(low_x) / low_x
    use0 = (lib.abs(j0) >= lib.abs(j1)) | (low_x < 1.0)
    low = lib.where(use0, keep * (j0 / lib.where(use0, f0, lib.ones_like(x))),
                    keep * (j1 / lib.where(use0, lib.ones_like(x), one)))
    return lib.where(x > l, high, low)


def _bessel_zeros(lmax, nmax):
    """z[l, n], the zeros of j_l, by bisection between the interlacing zeros of j_(l-1)."""
    z = math.pi * np.arange(1, nmax + lmax + 1)
    out = [z[:nmax]]
    for l in range(1, lmax + 1):
        lo, hi = z[:-1].copy(), z[1:].copy()
        s = np.sign(_sph_jn(l, lo + 1e-9))
        for _ in range(24):
            mid = 0.5 * (lo + hi)
            left = np.sign(_sph_jn(l, mid)) == s
            lo, hi = np.where(left, mid, lo), np.where(left, hi, mid)
        z = 0.5 * (lo + hi)
        for _ in range(3):
            f = _sph_jn(l, z)
            z = z - f / (_sph_jn(l - 1, z) - (l + 1) / z * f)
        out.append(z[:nmax])
    return np.stack(out)


class _Exact:
    """Basis tables and H X of one case in 64-bit torch."""

    def __init__(self, c, seed):
        self.c, R, lmax = c, c["R"], c["lmax"]
        f64 = lambda v: torch.as_tensor(v, dtype=torch.float64, device=DEVICE)  # noqa: E731
        x, w = np.polynomial.legendre.leggauss(c["n_r"])
        r = 0.5 * R * (1.0 + x)
        t, wt = np.polynomial.legendre.leggauss(c["n_theta"])
        phi = 2.0 * math.pi * np.arange(c["n_phi"]) / c["n_phi"]
        z = _bessel_zeros(lmax, c["nmax"])
        self.rad, rows, self.k = [], [], z / R
        for l in range(lmax + 1):
            norm = math.sqrt(2.0 / R ** 3) / f64(_sph_jn(l + 1, z[l]))
            self.rad.append(_sph_jn(l, f64(r)[:, None] * f64(self.k[l])[None, :]) * norm)
            rows.append(np.repeat(0.5 * self.k[l][None, :] ** 2, 2 * l + 1, axis=0).ravel())
        self.r, self.half_lambda = f64(r), f64(np.concatenate(rows))
        self.d = self.half_lambda.numel()
        # normalised Theta_lm(t), no Condon-Shortley phase
        s, self.theta = np.sqrt(1.0 - t * t), []
        mm = np.full_like(t, math.sqrt(0.5 / (2.0 * math.pi)))
        for m in range(lmax + 1):
            if m:
                mm = mm * s * math.sqrt((2 * m + 1) / (2.0 * m))
            p = [mm, math.sqrt(2 * m + 3) * t * mm]
            for l in range(m + 2, lmax + 1):
                a = math.sqrt((4.0 * l * l - 1) / (l * l - m * m))
                b = math.sqrt(((l - 1.0) ** 2 - m * m) / (4.0 * (l - 1) ** 2 - 1))
                p.append(a * (t * p[-1] - b * p[-2]))
            self.theta.append(f64(np.stack(p[:lmax + 1 - m], axis=1)))
        m = np.arange(-lmax, lmax + 1)
        ang = np.abs(m)[:, None] * phi[None, :]
        tri = np.where(m[:, None] < 0, np.sin(ang), np.cos(ang))
        self.tri = f64(tri * np.where(m == 0, 1.0, math.sqrt(2.0))[:, None])
        self.weights = f64(w * 0.5 * R * r * r)[:, None, None] * f64(wt)[None, :, None] \
            * (2.0 * math.pi / c["n_phi"]) * torch.ones(c["n_phi"], device=DEVICE)
        self.lm = [f64([l * l + l + k for l in range(abs(k), lmax + 1)]).long() for k in m]
        xyz = _points(r, t, phi)
        atoms = _atoms(c, seed)
        self.v = _potential(xyz, atoms)
        self.chunk = max(1, int(4e8 // self.v.numel()))
        self.P = None
        if c.get("kb"):
            self.P = torch.cat([self.adjoint(_projector_values(xyz, a) * self.weights)
                                for a in atoms])
            self.h = f64(_couplings(len(atoms)))

    def synthesis(self, X, rad=None):
        """(S, d) coefficients to (S, n_r, n_theta, n_phi) values."""
        c, rad, S = self.c, rad or self.rad, X.shape[0]
        N, L = c["nmax"], c["lmax"] + 1
        G = torch.cat([X[:, l * l * N:(l + 1) ** 2 * N].reshape(S, 2 * l + 1, N) @ rad[l].T
                       for l in range(L)], dim=1)
        F = torch.empty((S, c["n_r"], c["n_theta"], 2 * L - 1), dtype=torch.float64,
                        device=DEVICE)
        for i, lm in enumerate(self.lm):
            F[..., i] = torch.einsum("jl,slk->skj", self.theta[abs(i - L + 1)], G[:, lm])
        return F @ self.tri

    def adjoint(self, g):
        """(S, n_r, n_theta, n_phi) weighted values to (S, d) coefficients."""
        c, S = self.c, g.shape[0]
        L = c["lmax"] + 1
        A = g @ self.tri.T
        G = torch.empty((S, L * L, c["n_r"]), dtype=torch.float64, device=DEVICE)
        for i, lm in enumerate(self.lm):
            G[:, lm] = torch.einsum("jl,skj->slk", self.theta[abs(i - L + 1)], A[..., i])
        return torch.cat([(G[:, l * l:(l + 1) ** 2] @ self.rad[l]).reshape(S, -1)
                          for l in range(L)], dim=1)

    def apply(self, X):
        out, wv = torch.empty_like(X), self.weights * self.v
        for i in range(0, X.shape[0], self.chunk):
            x = X[i:i + self.chunk]
            out[i:i + self.chunk] = self.adjoint(self.synthesis(x) * wv)
        out += X * self.half_lambda
        if self.P is not None:
            out += ((X @ self.P.T) * self.h) @ self.P
        return out

    def filter(self, X, bounds):
        a, b, a0 = bounds
        mid, e = 0.5 * (a + b), 0.5 * (b - a)
        s1 = e / (a0 - mid)
        prev, cur, sig = X, (self.apply(X) - mid * X) * (s1 / e), s1
        for _ in range(1, self.c["degree"]):
            new = 1.0 / (2.0 / s1 - sig)
            prev, cur = cur, (self.apply(cur) - mid * cur) * (2.0 * new / e) - sig * new * prev
            sig = new
        return cur


def _exact_filter(c, seed):
    e = _Exact(c, seed)
    X = _block(c, e.half_lambda, seed, torch.float32 if c["prec"] in F32 else torch.float64)
    return e.filter(X[:, :e.d].double(), _bounds(c, e.half_lambda, e.v))


def _exact_fields(c, seed):
    e = _Exact(c, seed)
    X, occ = _block(c, e.half_lambda, seed)[:, :e.d], _occupations(c)
    rho = torch.zeros_like(e.v)
    for i in range(0, c["n_s"], e.chunk):
        f = e.synthesis(X[i:i + e.chunk])
        rho += 2.0 * torch.einsum("skjq,s->kjq", f * f, occ[i:i + e.chunk])
    tau, R, zeta, at = e.adjoint((rho * e.weights)[None]), c["R"], [], []
    for l in range(c["lmax"] + 1):
        k = torch.as_tensor(e.k[l], device=DEVICE)
        z = (2 * l + 1) / k ** 2 * e.rad[l] \
            + math.sqrt(2.0 / R ** 3) * R * ((e.r / R) ** l)[:, None] / k
        zeta.append(z * (4.0 * math.pi / (2 * l + 1)))
    vh = e.synthesis(tau, zeta)[0]
    pos = rho > 0
    n = torch.where(pos, rho, torch.ones_like(rho))
    rs = (3.0 / (4.0 * math.pi * n)) ** (1.0 / 3.0)
    ex = -0.75 * (3.0 * n / math.pi) ** (1.0 / 3.0)
    sq, lg = torch.sqrt(rs), torch.log(rs)
    den = 1.0 + 1.0529 * sq + 0.3334 * rs
    ec = torch.where(rs >= 1.0, -0.1423 / den, 0.0311 * lg - 0.048 + 0.002 * rs * lg - 0.0116 * rs)
    vc = torch.where(rs >= 1.0, -0.1423 / den ** 2 * (1.0 + 7.0 / 6.0 * 1.0529 * sq
                                                      + 4.0 / 3.0 * 0.3334 * rs),
                     0.0311 * lg + (-0.048 - 0.0311 / 3.0) + 2.0 / 3.0 * 0.002 * rs * lg
                     + (2.0 * -0.0116 - 0.002) / 3.0 * rs)
    zero = torch.zeros_like(rho)
    return {"rho": rho, "vh": vh, "exc": torch.where(pos, ex + ec, zero),
            "vxc": torch.where(pos, 4.0 / 3.0 * ex + vc, zero)}


def exact(case, seed):
    c, op = case, case["op"]
    if work(c)["flops"] > 2.0e13:
        return None
    if op == "batch":
        return [_exact_filter(k, seed + 97 * i) for i, k in enumerate(_clusters(c))]
    if op == "filter":
        return _exact_filter(c, seed)
    if op == "fields":
        return _exact_fields(c, seed)
    e = _Exact(c, seed)
    if op == "apply":
        X = _block(c, e.half_lambda, seed, torch.float32 if c["prec"] in F32 else torch.float64)
        return e.apply(X[:, :e.d].double())
    X = _block(c, e.half_lambda, seed)
    if op == "cholqr":  # X R^-1 with a positive diagonal of R is unique
        X = X[:, :e.d]
        for _ in range(2):
            X = torch.linalg.solve_triangular(torch.linalg.cholesky(X @ X.T), X, upper=False)
        return X
    # Ritz vectors have no sign of their own: only the values and residual norms are given
    X = _orthonormal(X, e.d)[:, :e.d]
    HX = e.apply(X)
    M = X @ HX.T
    theta, Q = torch.linalg.eigh(0.5 * (M + M.T))
    resid = torch.linalg.vector_norm(Q.T @ HX - theta[:, None] * (Q.T @ X), dim=1)
    return {"theta": theta, "resid": resid, "X": None, "HX": None}
