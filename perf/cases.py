"""Performance cases of the directional H^2 compression library.

A case is one pass that a program makes through the public entry points: a
compression of a matrix it holds (or of a kernel it names) followed by a product
with the result, or a product with a representation it made earlier.  The
product is what such a program needs the representation for, and it depends on
every basis, transfer matrix, coupling matrix and nearfield block, so it is the
output that is compared.

Inputs: collocation of the Helmholtz single-layer kernel exp(i kappa r)/(4 pi r)
(diagonal 1/(4 pi h), h the mean nearest-neighbour distance) or of 1/2 I + the
double-layer kernel, on a rotated Fibonacci lattice of the unit sphere, on
uniform random points of a 2:1:1 ellipsoid, or of the unit cube's surface.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1510_07087_gb300 as D

MODES = {"fp64": D.MODE_FP64, "fp32": D.MODE_FP32, "mixed": D.MODE_MIXED_BF16X3}
LITERAL = {"eta1": 2.0 * math.sqrt(2.0), "eta2": 1.0}
PAPER = {"eta1": 20.0, "eta2": 5.0}
# kappa * diameter of the surfaces of a batch
DIAMETER = {"sphere": 2.0, "ellipsoid": 2.0, "cube": math.sqrt(3.0)}


def _case(kind, surface, n, kappa, leaf, mode, eps=1e-4, nrhs=1, kernel="slp", paper=False):
    return {"kind": kind, "surface": surface, "n": n, "kappa": kappa, "leaf": leaf, "mode": mode, "eps": eps,
            "nrhs": nrhs, "kernel": kernel, **(PAPER if paper else LITERAL)}


def listed():
    return [
        # one product of an iterative solver on a small problem: launches and latency count
        dict(_case("product", "sphere", 1024, 2.0, 32, "fp32"), name="product-n1024"),
        # one product of an iterative solver at the benchmark's size
        dict(_case("product", "sphere", 32768, 32.0, 64, "mixed"), name="product-n32768"),
        # a block of right-hand sides (several incident waves) in double precision
        dict(_case("product", "sphere", 8192, 16.0, 32, "fp64", nrhs=8), name="product-fp64-n8192-r8"),
        # the adjoint product of a least-squares or BiCG iteration, double-layer matrix, odd size
        dict(_case("adjoint", "ellipsoid", 12289, 16.0, 64, "mixed", nrhs=3, kernel="dlp"), name="adjoint-dlp-n12289-r3"),
        # double-precision compression: the small sphere, and the middle one
        dict(_case("compress", "sphere", 2048, 4.0, 32, "fp64"), name="compress-fp64-n2048"),
        dict(_case("compress", "sphere", 8192, 16.0, 32, "fp64"), name="compress-fp64-n8192"),
        # mixed-precision compression: the middle sphere, and the benchmark's
        dict(_case("compress", "sphere", 8192, 16.0, 32, "mixed"), name="compress-mixed-n8192"),
        dict(_case("compress", "sphere", 32768, 32.0, 64, "mixed"), name="compress-mixed-n32768"),
        # single precision at the small tolerance
        dict(_case("compress", "sphere", 8192, 16.0, 32, "fp32", eps=1e-6), name="compress-fp32-n8192-eps1e-6"),
        # independent surfaces of uneven size in one call (a scene of scatterers)
        {"name": "batch-mixed-16", "kind": "batch", "count": 16, "lo": 1024, "hi": 6144, "leaf": 64, "mode": "mixed",
         "eps": 1e-4, "nrhs": 1, "shape_seed": 7, **LITERAL},
        # entries generated in the kernels, cube surface, kappa = 0.2 sqrt(n), the coarse tolerance
        dict(_case("free", "cube", 16384, 25.6, 64, "fp32", eps=1e-3), name="free-cube-n16384"),
        # a captured schedule replayed on a double-layer matrix of odd size, the paper's parameters
        dict(_case("plan", "ellipsoid", 8191, 16.0, 64, "mixed", kernel="dlp", paper=True), name="plan-dlp-paper-n8191"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product", "product", "adjoint", "compress", "compress", "compress", "batch", "free", "plan"])
    if kind == "batch":
        lo = _log_int(rng, 500, 2048)
        return {"kind": "batch", "count": rng.randint(3, 16), "lo": lo, "hi": rng.randint(2 * lo, 6144),
                "leaf": rng.choice([32, 48, 64]), "mode": rng.choice(["fp32", "mixed", "mixed"]), "eps": 1e-4,
                "nrhs": 1, "shape_seed": rng.randint(0, 10 ** 6), **LITERAL}
    surface = rng.choice(["sphere", "ellipsoid", "cube"])
    mode = rng.choice(["fp64", "fp32", "mixed", "mixed"])
    paper = kind in ("compress", "plan") and rng.random() < 0.3
    top = 32768
    if paper:
        top = 8192
    if kind == "free" or mode == "fp32":
        top = min(top, 16384)
    if mode == "fp64":
        top = min(top, 4096 if paper or kind == "free" else 8192)
    n = _log_int(rng, 1024, top)
    kappa = round(rng.uniform(0.09, 0.2) * math.sqrt(n), 2)
    if surface == "ellipsoid":
        kernel = rng.choice(["slp", "dlp"]) if kind != "free" else "slp"
    else:
        kernel = "slp"
    eps = rng.choice([1e-3, 1e-4, 1e-4]) if mode == "mixed" else rng.choice([1e-3, 1e-4, 1e-6 if not paper else 1e-5])
    nrhs = rng.choice([1, 1, 2, 3, 5, 8, 16]) if kind in ("product", "adjoint") else 1
    return _case(kind, surface, n, kappa, rng.choice([32, 48, 64]), mode, eps, nrhs, kernel, paper)


# ------------------------------------------------------------------ inputs

def _points(surface, n, rng):
    """(points, outward unit normals), float64 (n, 3); the cube's normals are not used."""
    if surface == "sphere":
        i = np.arange(n, dtype=np.float64)
        z = 1.0 - (2.0 * i + 1.0) / n
        r = np.sqrt(np.maximum(0.0, 1.0 - z * z))
        phi = i * (math.pi * (3.0 - math.sqrt(5.0)))
        q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
        p = np.ascontiguousarray(np.stack([r * np.cos(phi), r * np.sin(phi), z], axis=1) @ q)
        return p, p / np.linalg.norm(p, axis=1, keepdims=True)
    if surface == "ellipsoid":
        a = np.array([1.0, 0.5, 0.5])
        parts, have = [], 0
        while have < n:  # the sphere's uniform points kept by the map's area element, |a| |u / a|
            u = rng.standard_normal((2 * n, 3))
            u /= np.linalg.norm(u, axis=1, keepdims=True)
            u = u[rng.random(2 * n) * 2.0 <= np.linalg.norm(u / a, axis=1)]
            parts.append(u * a)
            have += len(u)
        p = np.ascontiguousarray(np.concatenate(parts)[:n])
        nrm = p / a ** 2
        return p, nrm / np.linalg.norm(nrm, axis=1, keepdims=True)
    face = rng.integers(0, 6, size=n)
    uv = rng.random((n, 2))
    p = np.empty((n, 3))
    for ax in range(3):
        s = face // 2 == ax
        o = [d for d in range(3) if d != ax]
        p[s, ax] = (face % 2)[s]
        p[s, o[0]], p[s, o[1]] = uv[s, 0], uv[s, 1]
    return p, np.zeros((n, 3))


def _spacing(pts):
    """Mean nearest-neighbour distance of device points."""
    total, n = 0.0, pts.shape[0]
    for s in range(0, n, 2048):
        d = pts[None, :, :] - pts[s:s + 2048, None, :]
        d2 = (d * d).sum(-1)
        d2[torch.arange(d2.shape[0], device=d2.device), torch.arange(s, s + d2.shape[0], device=d2.device)] = math.inf
        total += float(d2.min(1).values.sqrt().sum())
    return total / n


def _columns(pts, nrm, kappa, kernel, diag, s, e):
    """Columns [s, e) of G in complex128, one per row of the result."""
    d = pts[None, :, :] - pts[s:e, None, :]
    r = (d * d).sum(-1).sqrt()
    ph = kappa * r
    g = torch.complex(torch.cos(ph), torch.sin(ph))
    if kernel == "dlp":
        g = g * torch.complex(torch.ones_like(r), -ph) * ((d * nrm[s:e, None, :]).sum(-1) / (4.0 * math.pi * r ** 3))
    else:
        g = g / (4.0 * math.pi * r)
    g[torch.arange(e - s, device=g.device), torch.arange(s, e, device=g.device)] = diag
    return g


def _vectors(n, nrhs, dtype, rng):
    """Column-major (n, nrhs), or (n,) for one vector."""
    v = torch.from_numpy(rng.standard_normal((nrhs, n, 2))).cuda()
    v = torch.view_as_complex(v).to(dtype)
    return v[0].contiguous() if nrhs == 1 else v.t()


def _problem(c, rng, dense=True):
    """Points, tree, matrix (column-major view, the tree's order) and vectors of one surface."""
    host, hn = _points(c["surface"], c["n"], rng)
    tree = D.dh2_tree_build(host, c["leaf"], c["kappa"], c["eta1"], c["eta2"])
    perm = tree.perm()
    pts, nrm = torch.from_numpy(host[perm]).cuda(), torch.from_numpy(hn[perm]).cuda()
    dtype = torch.complex128 if c["mode"] == "fp64" else torch.complex64
    n = c["n"]
    diag = 0.5 if c["kernel"] == "dlp" else 1.0 / (4.0 * math.pi * _spacing(pts))
    p = {"tree": tree, "host": host, "pts": pts, "nrm": nrm, "diag": diag, "kappa": c["kappa"], "kernel": c["kernel"]}
    if dense:
        m = torch.empty((n, n), dtype=dtype, device="cuda")
        for s in range(0, n, 1024):
            e = min(n, s + 1024)
            m[s:e] = _columns(pts, nrm, c["kappa"], c["kernel"], diag, s, e)
        p["G"] = m.t()
    p["x"] = _vectors(n, c["nrhs"], dtype, rng)
    p["y"] = torch.zeros_like(p["x"])
    return p


def _members(c):
    """The surfaces of a batch: their kinds, sizes and wave numbers are the case's, their points the seed's."""
    r = np.random.default_rng(c["shape_seed"])
    out = []
    for i in range(c["count"]):
        surface = ("sphere", "ellipsoid", "cube")[i % 3]
        out.append({"surface": surface, "n": int(r.integers(c["lo"], c["hi"] + 1)),
                    "kappa": float(r.uniform(8.0, 40.0)) / DIAMETER[surface], "kernel": "slp",
                    **{k: c[k] for k in ("leaf", "mode", "eps", "nrhs", "eta1", "eta2")}})
    return out


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "batch":
        return {"case": case, "parts": [_problem(m, rng) for m in _members(case)]}
    p = _problem(case, rng, dense=case["kind"] != "free")
    opts = {"eps": case["eps"], "mode": MODES[case["mode"]]}
    if case["kind"] in ("product", "adjoint"):
        # the solver's program keeps the representation (it holds its own copy of the nearfield)
        p["M"] = D.dh2_compress(p["tree"], p["G"], **opts)
        p["M"]._G = None
        del p["G"]
    elif case["kind"] == "plan":
        p["plan"] = D.Plan([p["tree"]], [p["G"]], **opts)
    return {"case": case, "parts": [p]}


# ------------------------------------------------------------------ the pass

def run(state):
    c, parts = state["case"], state["parts"]
    p = parts[0]
    if c["kind"] == "product":
        D.dh2_matvec(p["M"], p["x"], p["y"])
        return p["y"]
    if c["kind"] == "adjoint":
        D.dh2_matvec_adjoint(p["M"], p["x"], p["y"])
        return p["y"]
    opts = {"eps": c["eps"], "mode": MODES[c["mode"]]}
    if c["kind"] == "compress":
        mats = [D.dh2_compress(p["tree"], p["G"], **opts)]
    elif c["kind"] == "free":
        mats = [D.dh2_compress_kernel(p["tree"], p["host"], p["kappa"], p["diag"], **opts)]
    elif c["kind"] == "plan":
        p["plan"].run([p["G"]])
        p["plan"].wait()
        mats = p["plan"].matrices()
    else:
        mats = D.dh2_compress_batched([q["tree"] for q in parts], [q["G"] for q in parts], **opts)
    for q, m in zip(parts, mats):
        D.dh2_matvec(m, q["x"], q["y"])
    return [q["y"] for q in parts]


# ------------------------------------------------------------------ floors and exact values

def work(case):
    """Compression: G read once (matrix-free: ~30 operations per entry instead), the nearfield entries of the
    representation written once, and read once by the product.  Product: the nearfield entries read once.  The
    vectors once each.  At least one complex multiply-add per dense entry and per nearfield entry and vector."""
    b = f = 0.0
    for c in _members(case) if case["kind"] == "batch" else [case]:
        host, _ = _points(c["surface"], c["n"], np.random.default_rng(1))
        adm = D.dh2_tree_build(host, c["leaf"], c["kappa"], c["eta1"], c["eta2"]).stats().adm_fraction
        size = 16 if c["mode"] == "fp64" else 8
        all_, near = float(c["n"]) ** 2, (1.0 - adm) * float(c["n"]) ** 2
        b += size * (near + 2.0 * c["n"] * c["nrhs"])
        f += 8.0 * near * c["nrhs"]
        if case["kind"] in ("compress", "batch", "plan"):
            b += size * (all_ + near)
            f += 8.0 * all_
        elif case["kind"] == "free":
            b += size * near + 24.0 * c["n"]
            f += 38.0 * all_
    return {"bytes": b, "flops": f}


def exact(case, seed):
    """G x (or G^* x) in 64 bits with the matrix that the pass is given."""
    rng = np.random.default_rng(seed)
    out = []
    for c in _members(case) if case["kind"] == "batch" else [case]:
        p = _problem(c, rng, dense=case["kind"] != "free")
        x = p["x"].to(torch.complex128)
        x = x[:, None] if x.dim() == 1 else x
        y = torch.zeros((c["n"], c["nrhs"]), dtype=torch.complex128, device="cuda")
        for s in range(0, c["n"], 1024):
            e = min(c["n"], s + 1024)
            if "G" in p:
                rows = p["G"].t()[s:e].to(torch.complex128)
            else:
                rows = _columns(p["pts"], p["nrm"], p["kappa"], p["kernel"], p["diag"], s, e)
            if case["kind"] == "adjoint":
                y[s:e] = rows.conj() @ x
            else:
                y += rows.t() @ x[s:e]
        y = y[:, 0] if c["nrhs"] == 1 else y
        out.append(y)
    return out[0] if case["kind"] in ("product", "adjoint") else out
