"""Products with many right-hand sides: chunks of one width share a launch.

Counts on both sides of the compiled widths (FP32 fills a chunk of 8 from 5
vectors on, FP64 takes exact widths), with full chunks and every remainder, each
column against its lone product, forward and adjoint, with and without the
second stream.  Sums of at most n terms in another order: 1e-12 (FP64), 1e-5 (FP32).
"""
import numpy as np
import pytest

from gpu_cases import colmajor, dev
from synth import helmholtz_matrix, random_ellipsoid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n,kappa", [(900, 6.0), (4200, 12.0)])
def test_columns_of_many_vectors(fp64, n, kappa):
    D = dev()
    pts = random_ellipsoid(n)
    T = D.dh2_tree_build(pts, 32, kappa)
    G = helmholtz_matrix(pts, kappa)[np.ix_(T.perm(), T.perm())]
    dt = torch.complex128 if fp64 else torch.complex64
    M = D.dh2_compress(T, colmajor(G, dt), eps=1e-4, mode=D.MODE_FP64 if fp64 else D.MODE_FP32)
    most = 71
    x = torch.randn((most, n), dtype=dt, device="cuda")
    one = torch.empty((2, most, n), dtype=dt, device="cuda")
    for a, f in enumerate((D.dh2_matvec, D.dh2_matvec_adjoint)):
        for k in range(most):
            f(M, x[k], one[a, k])
    tol = 1e-12 if fp64 else 1e-5
    for w in (10, 11, 12, 13, 14, 15, 16, 17, 24, 37, 63, 64, 65, 70, 71):
        for a, f in enumerate((D.dh2_matvec, D.dh2_matvec_adjoint)):
            y = torch.full((w + 1, n), float("nan"), dtype=dt, device="cuda")
            f(M, x[:w].t(), y[:w].t())
            d = (y[:w] - one[a, :w]).norm(dim=1) / one[a, :w].norm(dim=1)
            assert float(d.max()) <= tol, (w, a)
            assert torch.isnan(y[w].real).all() and (y[w].imag == 0).all()  # nothing past the last column
