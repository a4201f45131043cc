"""The FP32 mode's Gram matrices in 64-bit integers, at the sizes where they can go wrong.

Leaf sizes at the edges of the 4 x 4 tiles and of the size classes, column counts
around the 64-column chunks, and matrices whose entries grow by 2^24 from the
first columns of a block to the last, so that later chunks raise a row's scale
and shift the sums.  Against the FP64 mode on the same complex64 values: a
singular value may differ by the fixed point's backward error (2^-24 of a row's
largest entry over at most 1500 columns, below 64 u_32 of the largest singular
value) and by the FP32 Cholesky factor and Jacobi rotations (p u_32): 2e-5 of the
largest covers both at 64 rows.
"""
import numpy as np
import pytest

from gpu_cases import colmajor, dev
from synth import helmholtz_matrix, random_cube_surface, random_ellipsoid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("leaf,eta1,eta2", [(3, 2.8284271247461903, 1.0), (21, 2.8284271247461903, 1.0),
                                            (33, 20.0, 5.0), (41, 2.8284271247461903, 1.0), (64, 20.0, 5.0)])
@pytest.mark.parametrize("grow", [False, True])
def test_singular_values_agree_with_fp64(leaf, eta1, eta2, grow):
    D = dev()
    n, kappa = (700, 5.0) if leaf < 10 else (2600, 8.0)
    pts = random_ellipsoid(n) if leaf % 2 else random_cube_surface(n)
    T = D.dh2_tree_build(pts, leaf, kappa, eta1, eta2)
    perm = T.perm()
    G = helmholtz_matrix(pts, kappa)[np.ix_(perm, perm)]
    if grow:
        g = 2.0 ** np.round(24.0 * np.arange(n) / n)
        G = G * g[None, :] * g[:, None]
    G = G.astype(np.complex64).astype(np.complex128)
    M64 = D.dh2_compress(T, colmajor(G, torch.complex128), eps=1e-4, mode=D.MODE_FP64)
    M = D.dh2_compress(T, colmajor(G, torch.complex64), eps=1e-4, mode=D.MODE_FP32)
    checked = 0
    for side in (0, 1):
        pairs = T.pairs(side)
        assert np.mean(M.ranks(side) != M64.ranks(side)) <= 0.02
        leafs, rest = np.flatnonzero(pairs["leaf"]), np.flatnonzero(pairs["leaf"] == 0)
        for q in list(leafs[:: max(1, len(leafs) // 60)]) + list(rest[:: max(1, len(rest) // 30)]):
            a, b = M.sigma(side, int(q)), M64.sigma(side, int(q))
            k = min(len(a), len(b))
            assert np.all(np.abs(a[:k] - b[:k]) <= 2e-5 * b[0]), (side, int(q))
            checked += k
    assert checked > 50
    x = torch.randn(n, dtype=torch.complex128, device="cuda")
    y, y64 = torch.empty(n, dtype=torch.complex64, device="cuda"), torch.empty_like(x)
    D.dh2_matvec(M, x.to(torch.complex64), y)
    D.dh2_matvec(M64, x, y64)
    assert float((y - y64).norm()) <= 2e-4 * float(np.linalg.norm(G)) * float(x.norm())
