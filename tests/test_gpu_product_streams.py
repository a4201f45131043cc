"""Products whose nearfield runs on a second stream (n large enough for it).

Independent caller streams stay independent, and the forked product is the
product of one stream, in both precisions, for one and several vectors and the
adjoint.
"""
import ctypes
import threading
import time

import numpy as np
import pytest

from gpu_cases import colmajor, dev
from synth import helmholtz_matrix, random_ellipsoid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _matrix(fp64=False, n=4200, kappa=12.0):
    D = dev()
    pts = random_ellipsoid(n)
    T = D.dh2_tree_build(pts, 32, kappa)
    perm = T.perm()
    G = helmholtz_matrix(pts, kappa)[np.ix_(perm, perm)]
    assert (1.0 - T.stats().adm_fraction) * n * n > 2 ** 23  # the fork's threshold
    dt = torch.complex128 if fp64 else torch.complex64
    return D, D.dh2_compress(T, colmajor(G, dt), eps=1e-4, mode=D.MODE_FP64 if fp64 else D.MODE_FP32), dt, n


def test_a_held_stream_holds_no_other():
    """One thread, two streams: while the first waits for the host, a product on the second finishes.
    The host function waits 5 s at most, so the test ends in any case."""
    D, M, dt, n = _matrix()
    A, B = torch.cuda.Stream(), torch.cuda.Stream()
    x = torch.randn((2, n), dtype=dt, device="cuda")
    y = torch.zeros((3, 2, n), dtype=dt, device="cuda")
    torch.cuda.synchronize()
    for s, k in ((A, 0), (B, 1)):
        D.dh2_matvec(M, x[k], y[0, k], stream=s)
        torch.cuda.synchronize()
    release = threading.Event()
    hold = ctypes.CFUNCTYPE(None, ctypes.c_void_p)(lambda _: release.wait(5.0) and None)
    launch = ctypes.CDLL("libcuda.so.1").cuLaunchHostFunc
    assert launch(ctypes.c_void_p(A.cuda_stream), hold, None) == 0
    done = False
    try:
        for r in (1, 2):
            D.dh2_matvec(M, x[0], y[r, 0], stream=A)
            D.dh2_matvec(M, x[1], y[r, 1], stream=B)
        e = torch.cuda.Event()
        e.record(B)
        end = time.monotonic() + 3.0
        while not done and time.monotonic() < end:
            time.sleep(0.01)
            done = e.query()
    finally:
        release.set()
        torch.cuda.synchronize()
    assert done
    for r in (1, 2):
        for k in (0, 1):
            assert float((y[r, k] - y[0, k]).norm()) <= 1e-5 * float(y[0, k].norm())


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("nrhs", [1, 2, 3])
def test_forked_products_are_those_of_one_stream(fp64, nrhs):
    """dh2_matvec (forked) against dh2_matvec_noalloc (never forked), and the forked adjoint by
    <G~ x, z> = <x, G~^* z>.  Sums of at most n terms in another order: 1e-12 (FP64), 1e-5 (FP32)."""
    D, M, dt, n = _matrix(fp64)
    tol = 1e-12 if fp64 else 1e-5
    x, z = (torch.randn((nrhs, n), dtype=dt, device="cuda").t() for _ in range(2))
    y, y1, w = (torch.full((nrhs, n), float("nan"), dtype=dt, device="cuda").t() for _ in range(3))
    D.dh2_matvec(M, x, y)
    D.dh2_matvec_noalloc(M, x, y1)
    D.dh2_matvec_adjoint(M, z, w)
    torch.cuda.synchronize()
    for k in range(nrhs):
        assert float((y[:, k] - y1[:, k]).norm()) <= tol * float(y1[:, k].norm())
        p = torch.vdot(z[:, k].to(torch.complex128), y[:, k].to(torch.complex128))
        q = torch.vdot(w[:, k].to(torch.complex128), x[:, k].to(torch.complex128))
        assert abs(complex(p - q)) <= tol * float(y[:, k].norm()) * float(z[:, k].norm())
