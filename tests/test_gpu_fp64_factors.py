"""The parts of the FP64 factorisation that use less than FP64 on the way.

The reciprocal and reciprocal square root of dh2_scalar.cuh over their range
against the exact values, and the singular values and bases of full-rank leaf
matrices with close singular values (every column stays, so the FP32
preconditioner turns all of them) against LAPACK.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from gpu_cases import colmajor, dev
from synth import random_ellipsoid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1510_07087_gb300", "csrc")
SOURCE = """
#include "dh2_scalar.cuh"
__global__ void eval(const double* x, double* o, int n) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  o[i] = dh2::frsqrt(x[i]);
  o[n + i] = dh2::frcp(x[i]);
  // the start that the rotation scalars use, for arguments near 1
  o[2 * n + i] = x[i] >= 0.5 && x[i] <= 4.0 ? dh2::rsqrt_from(x[i], (double)rsqrtf((float)x[i])) : rsqrt(x[i]);
}
extern "C" void run(const double* x, double* o, int n) { eval<<<(n + 255) / 256, 256>>>(x, o, n); }
"""


def test_reciprocals_within_two_ulp(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src, lib = tmp_path / "s.cu", tmp_path / "s.so"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_103a,code=sm_103a", "-shared", "-Xcompiler",
                    "-fPIC", f"-I{CSRC}", str(src), "-o", str(lib)], check=True)
    rng = np.random.default_rng(0)
    m = np.concatenate([np.linspace(1.0, 4.0, 3001)[:-1], 1.0 + 3.0 * rng.random(20000),
                        np.nextafter([1.0, 2.0, 4.0], [9.0, 9.0, 0.0]), np.nextafter([2.0], [0.0])])
    # squared norms from Eps<double>::tiny (1e-280) to near overflow
    e = np.concatenate([np.arange(-928, 1020, 4), [-928, -2, 0, 2, 1018]])
    x = np.concatenate([np.ldexp(m[rng.integers(0, len(m), 2000)], int(k)) for k in e] + [m, np.ldexp(m, -1)])
    xd = torch.from_numpy(x).cuda()
    o = torch.empty((3, len(x)), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    fn = ctypes.CDLL(str(lib)).run
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    fn(xd.data_ptr(), o.data_ptr(), len(x))
    torch.cuda.synchronize()
    o = o.cpu().numpy()
    xl = x.astype(np.longdouble)
    assert np.finfo(np.longdouble).nmant > 60
    for got, want in ((o[0], 1 / np.sqrt(xl)), (o[1], 1 / xl), (o[2], 1 / np.sqrt(xl))):
        ulp = np.spacing(want.astype(np.float64))
        assert np.max(np.abs((got.astype(np.longdouble) - want) / ulp)) <= 2.0


@pytest.mark.parametrize("n,leaf,seed", [(1500, 32, 1), (1500, 20, 2), (2600, 40, 3), (2600, 48, 4)])
def test_close_singular_values(n, leaf, seed):
    """Random entries: all singular values of a leaf matrix lie within a factor of a few.  FP64
    backward errors of the LQ (p u), of the turned factor (K u) and of the Jacobi test (p u), each a few
    times over: 64 p u of the largest."""
    D = dev()
    T = D.dh2_tree_build(random_ellipsoid(n), leaf, 4.0)
    rng = np.random.default_rng(seed)
    G = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    M = D.dh2_compress(T, colmajor(G, torch.complex128), eps=1e-8, mode=D.MODE_FP64)
    invw, blk, cl = M.block_weights(), T.blocks(), T.clusters()
    checked = 0
    for side in (0, 1):
        pr = T.pairs(side)
        off, ids = T.pair_blocks(side)
        leafs = np.flatnonzero(pr["leaf"])
        for q in leafs[:: max(1, len(leafs) // 40)]:
            r0 = int(cl["start"][pr["cluster"][q]])
            m = int(cl["size"][pr["cluster"][q]])
            cols = []
            for b in ids[off[q]:off[q + 1]]:
                o = blk[b, 1 - side]
                s, w = int(cl["start"][o]), int(cl["size"][o])
                B = G[r0:r0 + m, s:s + w] if side == 0 else G[s:s + w, r0:r0 + m].conj().T
                cols.append(B * invw[b])
            A = np.concatenate(cols, axis=1)
            want = np.linalg.svd(A, compute_uv=False)
            got = M.sigma(side, int(q))
            k = min(len(got), len(want))
            tol = 64 * m * 2.0 ** -53
            assert np.all(np.abs(got[:k] - want[:k]) <= tol * want[0]), (side, int(q))
            V = M.pair_basis(side, int(q))
            r = V.shape[1]
            assert np.max(np.abs(V.conj().T @ V - np.eye(r))) <= tol
            checked += 1
    assert checked >= 20
