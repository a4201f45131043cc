"""Launch counts by kernel class: they add up to the launches where every class launches its own
kernels, and a launch over several classes counts in each of them."""
import numpy as np
import pytest

from gpu_cases import colmajor, dev
from synth import helmholtz_matrix, random_ellipsoid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _compress(n, leaf, kappa, mode, **eta):
    D = dev()
    pts = random_ellipsoid(n)
    T = D.dh2_tree_build(pts, leaf, kappa, **eta)
    G = helmholtz_matrix(pts, kappa)[np.ix_(T.perm(), T.perm())]
    fp64 = mode == D.MODE_FP64
    M = D.dh2_compress(T, colmajor(G, torch.complex128 if fp64 else torch.complex64), eps=1e-4, mode=mode)
    size, rows = T.clusters()["size"], []
    for s in (0, 1):
        pr = T.pairs(s)
        rows.append(size[pr["cluster"][pr["leaf"] == 1]])
    cls = sorted(set(np.searchsorted([32, 40, 48, 64], np.concatenate(rows), side="left").tolist()))
    levels = {int(v) for s in (0, 1) for v in T.clusters()["level"][T.pairs(s)["cluster"][T.pairs(s)["leaf"] == 0]]}
    return D, M, M.class_launches(), cls, len(levels)


def test_fp64_counts_add_up():
    D, M, L, cls, levels = _compress(3000, 32, 8.0, dev().MODE_FP64)
    assert levels > 0 and L.sum() == M.launch_count()
    assert L[D.KC_LEVEL_GRAM] == 0


@pytest.mark.parametrize("mode", ["fp32", "mixed"])
def test_merged_launches_count_in_every_class(mode):
    m = dev().MODE_FP32 if mode == "fp32" else dev().MODE_MIXED_BF16X3
    D, M, L, cls, levels = _compress(4096, 64, 12.0, m, eta1=20.0, eta2=5.0)
    assert len(cls) > 1 and levels > 0
    for c in range(4):
        assert L[D.KC_LEAF_FACTOR + c] == L[D.KC_LEAF_GRAM + c] == L[D.KC_LEAF_JACOBI + c] == (c in cls)
    assert L[D.KC_LEVEL_GRAM] == levels
    # Cholesky and Jacobi of each level, in class 0 whatever the level's rows
    assert L[D.KC_LEVEL_FACTOR] == 2 * levels
    extra = (len(cls) - 1) + sum(int(L[D.KC_LEVEL_FACTOR + c]) for c in (0, 1))
    assert L.sum() == M.launch_count() + extra
