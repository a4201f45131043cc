"""Scratch memory of the FP32 and mixed modes' Gram matrices.

A level's segments are widened until there are at most 4096 beside one per pair,
the LQ's segment buffer holds one level's segments, and without room for
the Gram matrices the factors come from the LQ.
"""
import ctypes

import numpy as np
import pytest

from gpu_cases import dev
from synth import random_ellipsoid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _problem(n, leaf, kappa, **eta):
    D = dev()
    pts = random_ellipsoid(n)
    T = D.dh2_tree_build(pts, leaf, kappa, **eta)
    p = torch.from_numpy(pts[T.perm()]).cuda()
    G = torch.empty((n, n), dtype=torch.complex64, device="cuda")
    for s in range(0, n, 1024):
        r = (p[None] - p[s:s + 1024, None]).norm(dim=-1)
        r[torch.arange(r.shape[0]), torch.arange(s, s + r.shape[0])] = 0.02
        G[s:s + 1024] = torch.polar(1.0 / (4 * np.pi * r), kappa * r).to(torch.complex64)
    return D, T, G.t()


class _Pool:
    """Bytes in use in the device's stream-ordered pool, now and at most since the last reset."""

    NOW, HIGH = 7, 8  # cudaMemPoolAttrUsedMemCurrent, cudaMemPoolAttrUsedMemHigh

    def __init__(self):
        self.rt = ctypes.CDLL("libcudart.so.13")
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def reset(self):
        v = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolSetAttribute(self.pool, self.HIGH, ctypes.byref(v)) == 0

    def read(self, attr):
        v = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolGetAttribute(self.pool, attr, ctypes.byref(v)) == 0
        return v.value


def test_level_scratch_is_bounded_and_wide_segments_are_right():
    D, T, G = _problem(16384, 64, 16.0, eta1=20.0, eta2=5.0)
    level = T.clusters()["level"]
    pairs = [T.pairs(s) for s in (0, 1)]
    count, segs, lq = {}, {}, {}
    for pr in pairs:
        for q in np.flatnonzero(pr["leaf"] == 0):
            lv, n = int(level[pr["cluster"][q]]), int(pr["ncols"][q])
            count[lv] = count.get(lv, 0) + 1
            segs[lv] = segs.get(lv, 0) + -(-n // 256)
            lq[lv] = lq.get(lv, 0) + (-(-n // 1024) if n > 2048 else 0)
    assert max(segs.values()) > 8192 + max(count.values())  # 256 and 512 columns would be too many
    nleaf = sum(int(pr["leaf"].sum()) for pr in pairs)
    pool = _Pool()
    torch.cuda.synchronize()
    pool.reset()
    M = D.dh2_compress(T, G, eps=1e-4, mode=D.MODE_FP32)
    torch.cuda.synchronize()
    used = pool.read(pool.HIGH) - pool.read(pool.NOW)
    matrix = 64 * 64 * 16
    bound = matrix * (nleaf + max(count.values()) + 4096) + 128 * 128 * 8 * max(lq.values()) + (64 << 20)
    assert 0 < used <= bound
    # level pairs of segments of 1024 columns, several flushes wide, against FP64
    M64 = D.dh2_compress(T, G.t().to(torch.complex128).t(), eps=1e-4, mode=D.MODE_FP64,
                         rank_override=(M.ranks(0), M.ranks(1)))
    checked = 0
    for side, pr in enumerate(pairs):
        rest = np.flatnonzero(pr["leaf"] == 0)
        for q in rest[np.argsort(-pr["ncols"][rest])][::8]:
            a, b = M.sigma(side, int(q)), M64.sigma(side, int(q))
            k = min(len(a), len(b))
            # fixed point, FP32 factor and rotations (p u_32) of the pair and of its sons' R
            tol = 2.0 ** -27 * np.sqrt(2.0 * 64 * pr["ncols"][q]) + 3 * 64 * 2.0 ** -24
            assert np.all(np.abs(a[:k] - b[:k]) <= tol * b[0]), (side, int(q))
            checked += 1
    assert checked > 100


@pytest.mark.parametrize("mode", ["fp32", "mixed"])
def test_without_room_for_gram_matrices_the_lq_runs(mode):
    D, _, G = _problem(4096, 32, 12.0, eta1=20.0, eta2=5.0)
    m = D.MODE_FP32 if mode == "fp32" else D.MODE_MIXED_BF16X3
    pts = random_ellipsoid(4096)
    T = D.dh2_tree_build(pts, 32, 12.0, eta1=20.0, eta2=5.0)
    D.dh2_debug_fail_alloc(3)  # the tree's lists, the matrix, then the call's scratch
    try:
        M = D.dh2_compress(T, G, eps=1e-4, mode=m)
    finally:
        D.dh2_debug_fail_alloc(0)
    W = D.dh2_compress(T, G, eps=1e-4, mode=m)
    L, N = M.class_launches(), W.class_launches()
    if mode == "fp32":
        assert L[D.KC_LEAF_GRAM:D.KC_LEAF_GRAM + 4].sum() == 0 < N[D.KC_LEAF_GRAM:D.KC_LEAF_GRAM + 4].sum()
    assert not np.array_equal(L, N)
    for side in (0, 1):
        d = M.ranks(side) - W.ranks(side)
        assert np.mean(d != 0) <= 0.01 and np.abs(d).max() <= 1
    assert D.dh2_error(M, G) <= 1e-4
    assert D.dh2_error(M, G) <= 1.05 * D.dh2_error(W, G)
