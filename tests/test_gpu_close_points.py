"""Entries of the matrix-free FP32 mode where differences of the points cancel.

All points lie in one leaf, so products with the unit vectors are the generated
entries themselves.  They are compared with the formula in extended precision on
the same FP64 points: pairs of points close beside the extent, points graded
towards one place, flat faces, and extents far from 1.  An entry's own FP32
roundings (sin and cos of the reduced phase 2 ulp each, the phase half an ulp of
1 times pi, scale, (1 - i kappa r) and product 1 ulp each) stay below 16 u,
u = 2^-24, of its modulus.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _entries(pts, nrm, kappa, diag):
    import paper_1510_07087_gb300 as D

    n = len(pts)
    T = D.dh2_tree_build(pts, 64, kappa)
    if nrm is None:
        M = D.dh2_compress_kernel(T, pts, kappa, diag, eps=1e-4, mode=D.MODE_FP32)
    else:
        M = D.dh2_compress_kernel_dlp(T, pts, nrm, kappa, eps=1e-4, mode=D.MODE_FP32)
    x = torch.eye(n, dtype=torch.complex64, device="cuda").t()
    y = torch.empty_like(x)
    D.dh2_matvec(M, x, y)
    perm = T.perm()
    out = np.empty((n, n), dtype=np.complex128)
    out[np.ix_(perm, perm)] = y.cpu().numpy()
    return out


def _formula(pts, nrm, kappa, diag):
    p = pts.astype(np.longdouble)
    d = p[:, None, :] - p[None, :, :]
    r = np.sqrt((d * d).sum(-1))
    np.fill_diagonal(r, 1.0)
    ph = np.longdouble(kappa) * r
    re, im, pi4 = np.cos(ph), np.sin(ph), 4 * np.arctan(np.longdouble(1)) * 4
    if nrm is None:
        re, im = re / (pi4 * r), im / (pi4 * r)
    else:
        s = (d * nrm.astype(np.longdouble)[None]).sum(-1) / (pi4 * r ** 3)
        re, im = (re + ph * im) * s, (im - ph * re) * s
    G = re.astype(np.float64) + 1j * im.astype(np.float64)
    np.fill_diagonal(G, diag)
    return G


def _sphere(n, rng):
    p = rng.standard_normal((n, 3))
    return p / np.linalg.norm(p, axis=1, keepdims=True)


def _twins(h):
    rng = np.random.default_rng(4)
    p = _sphere(24, rng)
    t = np.cross(p, _sphere(24, rng))
    q = p + h * t / np.linalg.norm(t, axis=1, keepdims=True)
    pts = np.concatenate([p, q / np.linalg.norm(q, axis=1, keepdims=True)])
    return pts, pts.copy()


def _graded():
    rng = np.random.default_rng(5)
    return _sphere(48, rng) * 10.0 ** -np.linspace(0, 14, 48)[:, None], _sphere(48, rng)


def _face():
    rng = np.random.default_rng(6)
    pts = np.concatenate([rng.random((24, 3)) * [1, 1, 0], rng.random((24, 3)) * [0, 1, 1]])
    nrm = np.repeat([[0.0, 0.0, -1.0], [-1.0, 0.0, 0.0]], 24, axis=0)
    return pts, nrm


CASES = [("twins", 1e-3), ("twins", 1e-5), ("twins", 1e-7), ("twins", 1e-9), ("twins", 1e-12), ("graded", 1.0),
         ("face", 1.0), ("scale", 1e-12), ("scale", 1e12), ("scale", 1e30)]


@pytest.mark.parametrize("kind,value", CASES)
@pytest.mark.parametrize("kernel", ["slp", "dlp"])
def test_entries(kernel, kind, value):
    if kind == "scale" and kernel == "dlp" and value > 1e15:
        pytest.skip("the entries themselves are below FP32's range")
    pts, nrm = _twins(value) if kind == "twins" else _graded() if kind == "graded" else _face() if kind == "face" \
        else tuple(v * s for v, s in zip(_twins(1e-4), (value, 1.0)))
    kappa = 3.0 / np.ptp(pts, axis=0).max()
    diag = 0.5 if kernel == "dlp" else 2.0
    nrm = nrm if kernel == "dlp" else None
    got, want = _entries(pts, nrm, kappa, diag), _formula(pts, nrm, kappa, diag)
    assert np.all(np.isfinite(got))
    # the FP64 scalar product <x - y, n> itself cancels: 4 of its roundings of r / (4 pi r^3)
    slack = 0.0
    if nrm is not None:
        r = np.linalg.norm(pts[:, None] - pts[None], axis=-1)
        np.fill_diagonal(r, np.inf)
        slack = 4 * 2.0 ** -53 / (4 * np.pi * r ** 2) * np.hypot(1.0, kappa * np.where(np.isinf(r), 0.0, r))
    assert np.all(np.abs(got - want) <= 16 * 2.0 ** -24 * np.abs(want) + slack)


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -20, 2.0 ** 37])
@pytest.mark.parametrize("kernel", ["slp", "dlp"])
def test_small_and_large_surfaces(kernel, scale):
    """Block norms far from 1 (at 2^37 the double layer's entries are of 1e-23, whose squares FP32
    cannot hold): scaled by a power of two, the same tree gets the same ranks."""
    import paper_1510_07087_gb300 as D
    from synth import fibonacci_sphere

    unit = fibonacci_sphere(3000)

    def compress(f):
        T = D.dh2_tree_build(unit * f, 32, 6.0 / f)
        if kernel == "slp":
            return T, D.dh2_compress_kernel(T, unit * f, 6.0 / f, 20.0 / f, eps=1e-4, mode=D.MODE_FP32)
        return T, D.dh2_compress_kernel_dlp(T, unit * f, unit, 6.0 / f, eps=1e-4, mode=D.MODE_FP32)

    (T0, M0), (T, M) = compress(1.0), compress(scale)
    assert T0.stats().adm_fraction > 0.1
    assert np.array_equal(T0.perm(), T.perm()) and np.array_equal(T0.blocks(), T.blocks())
    for s in (0, 1):
        assert max(M0.ranks(s)) > 4
        assert np.mean(M.ranks(s) != M0.ranks(s)) <= 0.01
    w, w0 = M.block_weights(), M0.block_weights()
    b = T.blocks()[:, 2] == 1
    factor = 1.0 / scale if kernel == "slp" else 1.0 / scale ** 2  # the entries'
    assert np.max(np.abs(w[b] * factor / w0[b] - 1.0)) <= 1e-6
