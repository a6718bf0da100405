"""Timed cases of the Helmholtz solver: the solves that programs make through
the package's public entry points, over the sizes, precisions, boundary
conditions and elements that its tests, benchmark and request server use.

A case is a dict of plain values:
  kind      "solve" (Plan.solve of one load), "many" (helm_solve_many of nrhs
            loads of one operator), "batch" (count mixed 2D problems as one
            Batch.solve) or "serve" (a request server with warm plans that
            takes requests of several operators and waits for them all)
  nx, ny, nz, lx, ly, lz   node counts and side lengths (nz = 0: 2D)
  ppw       nodes per wavelength at the largest spacing
  mode      "c128", "fp64" (complex64 solves refined on the FP64 residual) or
            "ff" (refined on the float-float residual)
  neumann   axes with Neumann faces, e.g. "x" (the others absorb)
  element   "q1" or "q1mod"
  rhs       "gaussian" or "bump" (times a Gaussian bump at the box's centre)
"batch" and "serve" draw their problems from `problems` (a seed) with sizes in
[lo, hi].
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1809_03808_gb300 as helm

TOL = 2e-11  # refinement tolerance of the benchmark, the batches and the server
_MODE = {"c128": helm.HELM_C128, "fp64": helm.HELM_C64_REFINED, "ff": helm.HELM_C64_REFINED}


def _one(name, kind, shape, lengths, ppw, mode, neumann="", element="q1", rhs="gaussian", nrhs=1):
    n, side = tuple(shape) + (0,) * (3 - len(shape)), tuple(lengths) + (0.0,) * (3 - len(lengths))
    return {"name": name, "kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "lx": side[0], "ly": side[1],
            "lz": side[2], "ppw": ppw, "mode": mode, "neumann": neumann, "element": element, "rhs": rhs, "nrhs": nrhs}


def listed():
    return [
        # a small 2D problem of an inner loop (16 nodes per wavelength), in FP64: launches and latency
        _one("2d_129_c128", "solve", (129, 129), (1.0, 1.0), 16.0, "c128"),
        # the same problem by the refined path that programs take by default for speed
        _one("2d_129_refined", "solve", (129, 129), (1.0, 1.0), 16.0, "fp64"),
        # an ordinary 2D duct with a prime transform length (Bluestein) and Neumann ends
        _one("2d_640x1021_refined_neumann", "solve", (640, 1021), (1.3, 0.8), 9.0, "fp64", neumann="x"),
        # the large 2D benchmark, refined and in FP64: a localised load on 33.5 M unknowns
        _one("2d_8192x4096_refined", "solve", (8192, 4096), (2.0, 1.0), 10.0, "fp64", rhs="bump"),
        _one("2d_8192x4096_c128", "solve", (8192, 4096), (2.0, 1.0), 10.0, "c128", rhs="bump"),
        # a mid-size 3D problem in FP64 with composite lengths
        _one("3d_201x150x175_c128", "solve", (201, 150, 175), (1.0, 0.75, 0.9), 10.0, "c128"),
        # a ragged 3D problem with prime lengths and the low-dispersion elements, FP64 residual
        _one("3d_190x223x127_refined_mod", "solve", (190, 223, 127), (0.9, 1.1, 0.7), 8.0, "fp64", element="q1mod"),
        # the 3D benchmark: 134 M unknowns refined on the FP64 residual
        _one("3d_512_refined", "solve", (512, 512, 512), (1.0, 1.0, 1.0), 10.0, "fp64"),
        # a large 3D problem on the float-float residual
        _one("3d_384x320x256_ff", "solve", (384, 320, 256), (1.2, 1.0, 0.8), 10.0, "ff"),
        # domain-decomposition sweeps: many loads of one small 3D operator
        _one("3d_96x80x72_many8", "many", (96, 80, 72), (1.0, 0.9, 0.8), 10.0, "ff", nrhs=8),
        # a parameter study: mixed 2D problems of any length as one launch
        {"name": "batch_48", "kind": "batch", "count": 48, "problems": 1000, "lo": 63, "hi": 511, "mode": "fp64"},
        # a server with its operators' plans cached takes a burst of requests
        {"name": "serve_6", "kind": "serve", "count": 6, "problems": 2000, "operators": 3, "lo": 31, "hi": 160,
         "most_rhs": 6, "mode": "ff"},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(("2d", "2d", "3d", "3d", "3d", "many", "batch", "serve"))
    if what == "batch":
        return {"kind": "batch", "count": rng.randint(8, 48), "problems": rng.randint(1, 10 ** 6), "lo": 63,
                "hi": rng.randint(200, 511), "mode": rng.choice(("fp64", "ff"))}
    if what == "serve":
        return {"kind": "serve", "count": rng.randint(2, 6), "problems": rng.randint(1, 10 ** 6), "operators": 3,
                "lo": 31, "hi": rng.randint(64, 160), "most_rhs": rng.randint(1, 6), "mode": rng.choice(("fp64", "ff"))}
    mode = rng.choice(("fp64", "fp64", "ff", "c128"))
    dim = 2 if what == "2d" else 3
    if dim == 2:
        shape = (size(63, 4096), size(63, 2048))
    elif what == "many":
        shape = (size(31, 128), size(31, 128), size(31, 128))
    else:
        top = 224 if mode == "c128" else 400
        shape = (size(31, top), size(31, top), size(31, top))
    c = _one("", "many" if what == "many" else "solve", shape, [round(rng.uniform(0.5, 2.0), 3) for _ in shape],
             round(rng.uniform(8.0, 16.0), 2), mode, neumann=rng.choice(("", "", "", "x", "y")),
             element=rng.choice(("q1", "q1", "q1mod")), rhs=rng.choice(("gaussian", "gaussian", "bump")),
             nrhs=rng.randint(2, 12) if what == "many" else 1)
    del c["name"]
    return c


# ---- the problems of a case --------------------------------------------------

def _problems(case):
    """[(shape, h, omega, bc, element, rhs, nrhs)] of the case's solves."""
    out = []
    if case["kind"] in ("solve", "many"):
        dim = 3 if case["nz"] else 2
        shape = (case["nx"], case["ny"], case["nz"])[:dim]
        h = tuple(side / (n - 1) for side, n in zip((case["lx"], case["ly"], case["lz"]), shape))
        bc = tuple("neumann" if a in case["neumann"] else "abc" for a in "xyz"[:dim])
        omega = 2.0 * math.pi / (case["ppw"] * max(h))
        return [(shape, h, omega, bc, case["element"], case["rhs"], case["nrhs"])]
    rng = random.Random(case["problems"])
    dim = 2 if case["kind"] == "batch" else 3
    pool = []
    for _ in range(case["count"] if dim == 2 else case["operators"]):
        shape = tuple(rng.randint(case["lo"], case["hi"]) for _ in range(dim))
        h = tuple(rng.uniform(0.5, 2.0) / (n - 1) for n in shape)
        omega = 2.0 * math.pi / (rng.uniform(8.0, 16.0) * max(h))
        pool.append((shape, h, omega, ("abc",) * dim, "q1", "gaussian"))
    for k in range(case["count"]):
        p = pool[k if dim == 2 else rng.randrange(len(pool))]
        out.append(p + (1 if dim == 2 else rng.randint(1, case["most_rhs"]),))
    return out


def _load(shape, rhs, nrhs, gen):
    """nrhs complex Gaussian nodal loads, "bump": times a Gaussian at the centre."""
    f = torch.randn((nrhs,) + tuple(shape), dtype=torch.complex128, device="cuda", generator=gen)
    if rhs == "bump":
        for k, n in enumerate(shape):
            x = torch.linspace(-1.0, 1.0, n, dtype=torch.float64, device="cuda")
            f *= torch.exp(-x * x / (2.0 * 0.2 ** 2)).reshape([n if j == k + 1 else 1 for j in range(len(shape) + 1)])
    return f


def _loads(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [_load(p[0], p[5], p[6], gen) for p in _problems(case)]


def _plan(p, mode):
    shape, h, omega, bc, element = p[:5]
    plan = helm.Plan(shape, h, omega, _MODE[mode], bc=bc if "neumann" in bc else None, element=element)
    if mode != "c128":
        helm.helm_set_refinement(plan.handle, TOL, 10)
        if mode == "ff":
            helm.helm_set_residual(plan.handle, helm.HELM_RESID_FF)
    return plan


def _submit_all(s):
    tickets = [s["server"].submit(p[0], p[1], p[2], f, u, residual=s["residual"], tol=TOL, nrhs=p[6])
               for p, f, u in zip(s["problems"], s["f"], s["u"])]
    for t in tickets:
        r = s["server"].wait(t)
        if r.status != helm.HELM_OK:
            raise RuntimeError(f"request failed: {s['server'].error(t)}")


def prepare(case, seed):
    ps, fs = _problems(case), _loads(case, seed)
    us = [torch.empty_like(f) for f in fs]
    s = {"kind": case["kind"], "problems": ps, "f": fs, "u": us}
    if case["kind"] == "serve":
        s["server"] = helm.Server(nslots=4, device_budget_bytes=16 << 30)
        s["residual"] = helm.HELM_RESID_FF if case["mode"] == "ff" else helm.HELM_RESID_FP64
        torch.cuda.synchronize()  # the server's streams read the loads
        _submit_all(s)            # plans cached, as in a server that has been up
    else:
        s["plans"] = [_plan(p, case["mode"]) for p in ps]
        if case["kind"] != "many":
            s["f"], s["u"] = [f[0] for f in fs], [u[0] for u in us]
        if case["kind"] == "batch":
            s["batch"] = helm.Batch(s["plans"])
    return s


def run(s):
    if s["kind"] == "solve":
        return s["plans"][0].solve(s["f"][0], s["u"][0])
    if s["kind"] == "many":
        h = s["plans"][0].handle
        helm.helm_set_stream(h, torch.cuda.current_stream().cuda_stream)
        helm.helm_solve_many(h, s["f"][0].shape[0], s["f"][0], s["u"][0])
        return s["u"][0]
    if s["kind"] == "batch":
        return s["batch"].solve(s["f"], s["u"])
    _submit_all(s)
    return s["u"]


def work(case):
    """Each load read and each solution written once (complex128); operations
    of one direct solve: the transforms there and back (5 n log2 n a line) and
    three complex tridiagonal sweeps (30 operations an unknown; 3D: for each
    of the three outer ones)."""
    byts = flops = 0.0
    for p in _problems(case):
        n = math.prod(p[0]) * p[6]
        byts += 32.0 * n
        flops += n * (10.0 * sum(math.log2(k) for k in p[0][1:]) + (90.0 if len(p[0]) == 2 else 270.0))
    return {"bytes": byts, "flops": flops}


# ---- the same solutions in 64 bits, without the package ----------------------

def _axis(n, h, omega, element):
    """Diagonals and off-diagonals of the 1D matrices K (with the faces' terms)
    and M of one axis; omega = 0: Neumann faces."""
    den = 12.0 if element == "q1mod" else 6.0
    kd = np.full(n, 2.0 / h, dtype=complex)
    md = np.full(n, (den - 2.0) * h / den, dtype=complex)
    kd[[0, -1]] = 1.0 / h - 1j * omega
    md[[0, -1]] *= 0.5
    return kd, -1.0 / h, md, h / den


def _eigen(n, ax):
    """V, lam with V^T K V = diag(lam), V^T M V = I, from the two parity halves
    of the axis (K and M are symmetric under reversal)."""
    kd, ko, md, mo = ax
    dense = [np.diag(d) + o * (np.eye(n, k=1) + np.eye(n, k=-1)) for d, o in ((kd, ko), (md, mo))]
    vs, lams = [], []
    for sign, half in ((1.0, (n + 1) // 2), (-1.0, n // 2)):
        q = np.zeros((n, half))
        for j in range(half):
            if j == n - 1 - j:
                q[j, j] = 1.0
            else:
                q[j, j], q[n - 1 - j, j] = math.sqrt(0.5), sign * math.sqrt(0.5)
        k2, m2 = q.T @ dense[0] @ q, q.T @ dense[1] @ q
        lam, v = np.linalg.eig(np.linalg.solve(m2, k2))
        v = v / np.sqrt(np.einsum("ij,ij->j", v, m2 @ v))
        vs.append(q @ v)
        lams.append(lam)
    return np.concatenate(vs, axis=1), np.concatenate(lams)


def _tri(ax, axis, u):
    """The tridiagonal matrices K u and M u of one axis applied along `axis`."""
    kd, ko, md, mo = ax
    n = u.shape[axis]
    s = torch.zeros_like(u)
    s.narrow(axis, 1, n - 1).add_(u.narrow(axis, 0, n - 1))
    s.narrow(axis, 0, n - 1).add_(u.narrow(axis, 1, n - 1))
    shape = [n if j == axis else 1 for j in range(u.dim())]
    dev = lambda d: torch.from_numpy(d).to(u.device).reshape(shape)  # noqa: E731
    return dev(kd) * u + ko * s, dev(md) * u + mo * s


def _apply(axes, w2, u):
    """A u = sum_j (K on axis j, M on the others) u - w^2 M...M u."""
    kp, mp = None, u  # kp: the terms with one K so far; mp: M on all axes so far
    for k, ax in enumerate(axes):
        knew, mnew = _tri(ax, k, mp)
        kp = knew if kp is None else knew + _tri(ax, k, kp)[1]
        mp = mnew
    return kp - w2 * mp


def _solve64(p, f):
    """u of A u = f by the eigenvectors of every axis but the longest and a
    tridiagonal solve along that one, refined twice on the residual."""
    shape, h, omega, bc, element = p[:5]
    axes = [_axis(n, hk, omega if b == "abc" else 0.0, element) for n, hk, b in zip(shape, h, bc)]
    line = max(range(len(shape)), key=lambda k: shape[k])
    rest = [k for k in range(len(shape)) if k != line]
    eig = {k: tuple(torch.from_numpy(x).cuda() for x in _eigen(shape[k], axes[k])) for k in rest}
    lam = -omega ** 2 + sum(eig[k][1].reshape([-1 if j == i else 1 for j in range(len(rest))])
                            for i, k in enumerate(rest))
    kd, ko, md, mo = axes[line]

    def to(v, k, m):
        return torch.movedim(torch.tensordot(v, m, dims=([k], [0])), -1, k)

    def solve(r):
        for k in rest:
            r = to(r, k, eig[k][0])
        r = torch.movedim(r, line, 0).contiguous()
        b = ko + lam * mo
        inv = []
        for i in range(shape[line]):
            d = complex(kd[i]) + lam * complex(md[i])
            if i:
                g = b * inv[-1]
                d = d - g * b
                r[i] -= g * r[i - 1]
            inv.append(1.0 / d)
        for i in reversed(range(shape[line])):
            if i + 1 < shape[line]:
                r[i] -= b * r[i + 1]
            r[i] *= inv[i]
        del inv
        r = torch.movedim(r, 0, line)
        for k in rest:
            r = to(r, k, eig[k][0].T)
        return r

    u = solve(f.clone())
    for _ in range(2):
        u = u + solve(f - _apply(axes, omega ** 2, u))
    return u.contiguous()


def exact(case, seed):
    ps = _problems(case)
    if any(sorted(p[0])[-2] > 1100 for p in ps):  # dense eigenvectors of every axis but the longest
        return None
    us = []
    for p, f in zip(ps, _loads(case, seed)):
        us.append(torch.stack([_solve64(p, f[i]) for i in range(f.shape[0])]))
    if case["kind"] == "solve":
        return us[0][0]
    if case["kind"] == "many":
        return us[0]
    return [u[0] for u in us] if case["kind"] == "batch" else us
