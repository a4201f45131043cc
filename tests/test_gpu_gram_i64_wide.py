"""The FP32 mode's integer Gram matrices for leaf pairs of many columns.

The sums of a pair wider than 512 columns are taken to double-float before they
can overflow, so that the fixed point keeps 26 bits at any width.  (One 64-bit sum
over the whole width leaves 23 bits at 8193 to 32768 columns, and the noise
raises ranks until the level pairs pass the compiled row limit.)
"""
import numpy as np
import pytest

from synth import random_ellipsoid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _problem(n, leaf, kappa, eta1, eta2, dtype, flat=False):
    import paper_1510_07087_gb300 as D

    pts = random_ellipsoid(n)
    T = D.dh2_tree_build(pts, leaf, kappa, eta1, eta2)
    p = pts[T.perm()]
    m = torch.empty((n, n), dtype=dtype, device="cuda")
    q = torch.from_numpy(p).cuda()
    for s in range(0, n, 1024):  # column by column, the tree's order; diagonal 1
        r = (q[None] - q[s:s + 1024, None]).norm(dim=-1)
        r[torch.arange(r.shape[0]), torch.arange(s, s + r.shape[0])] = 1.0
        g = torch.polar(torch.ones_like(r) if flat else 1.0 / (4 * np.pi * r), kappa * r)
        g[torch.arange(r.shape[0]), torch.arange(s, s + r.shape[0])] = 1.0
        m[s:s + 1024] = g.to(dtype)
    leafs = [T.pairs(s)["ncols"][T.pairs(s)["leaf"] == 1] for s in (0, 1)]
    return D, T, m.t(), max(int(v.max()) for v in leafs)


def test_very_wide_pairs_stay_within_the_row_limit():
    """Leaf pairs of more than 16000 columns at eps 1e-6: compressed, with an error of the size of
    FP32's own rounding of the bases (128 u = 7.6e-6; twice that)."""
    D, T, G, widest = _problem(20000, 64, 1.0, 20.0, 5.0, torch.complex64)
    assert widest > 16384
    M = D.dh2_compress(T, G, eps=1e-6, mode=D.MODE_FP32)
    assert D.dh2_error(M, G) <= 2 * 128 * 2.0 ** -24


@pytest.mark.parametrize("flat", [False, True])
@pytest.mark.parametrize("n,leaf", [(1400, 5), (2600, 40), (6000, 64)])
def test_singular_values_across_flushes(n, leaf, flat):
    """Pairs on both sides of one and of several flushes (most of them where all entries have modulus
    1, so that the sums grow fastest), small and full tiles, against FP64: a
    singular value may differ by the norm of the fixed point's errors, 2^-27 sqrt(2 p N) of a row's
    largest entry, and by the FP32 factor and rotations, p u_32, relative to the largest."""
    D, T, G64, widest = _problem(n, leaf, 3.0, 20.0, 5.0, torch.complex128, flat)
    assert widest > 1024
    G = G64.t().to(torch.complex64).t()
    G64 = G.t().to(torch.complex128).t()
    M = D.dh2_compress(T, G, eps=1e-4, mode=D.MODE_FP32)
    M64 = D.dh2_compress(T, G64, eps=1e-4, mode=D.MODE_FP64)
    checked = 0
    for side in (0, 1):
        pr = T.pairs(side)
        assert np.mean(M.ranks(side) != M64.ranks(side)) <= 0.02
        leafs = np.flatnonzero(pr["leaf"])
        for q in leafs[np.argsort(-pr["ncols"][leafs])][:: max(1, len(leafs) // 80)]:
            a, b = M.sigma(side, int(q)), M64.sigma(side, int(q))
            k = min(len(a), len(b))
            tol = 2.0 ** -27 * np.sqrt(2.0 * leaf * pr["ncols"][q]) + leaf * 2.0 ** -24
            assert np.all(np.abs(a[:k] - b[:k]) <= tol * b[0]), (side, int(q))
            checked += k
    assert checked > 50
