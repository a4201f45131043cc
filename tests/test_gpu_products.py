"""Products with several right-hand sides, nearfield copy and view.

Every chunk width of the right-hand sides (compiled widths, remainders) must
give each column the product of that column alone, the adjoint product must
satisfy <G~ x, z> = <x, G~^* z>, and both must approximate G x and G^* z within
the error bound of the compression.  The trees hold nearfield blocks of more
than 128 rows (row slabs), odd row counts (the 16-byte copies' padding) and
several pieces per block.  Sums of at most n terms in different orders differ
by n u relative to |G| |x| at most; the bounds are 1e-12 (FP64) and 1e-5 (FP32).
"""
import numpy as np
import pytest

from gpu_cases import colmajor, dev
from synth import (dlp_matrix, ellipsoid_normals, helmholtz_matrix, random_complex_vectors,
                   random_ellipsoid)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("view", [0, 1])
@pytest.mark.parametrize("n,kappa,leaf,kernel", [(3000, 3.0, 64, "slp"), (1501, 6.0, 24, "dlp"), (37, 1.0, 64, "slp")])
def test_products_by_columns(fp64, view, n, kappa, leaf, kernel):
    D = dev()
    if kernel == "dlp":
        pts = random_ellipsoid(n)
        G = dlp_matrix(pts, ellipsoid_normals(pts), kappa)
    else:
        pts = random_ellipsoid(n)
        G = helmholtz_matrix(pts, kappa)
    T = D.dh2_tree_build(pts, leaf, kappa)
    perm = T.perm()
    G = G[np.ix_(perm, perm)]
    if n == 3000:
        size, b = T.clusters()["size"], T.blocks()
        assert size[b[b[:, 2] == 0, 0]].max() > 128
    dt = torch.complex128 if fp64 else torch.complex64
    tol = 1e-12 if fp64 else 1e-5
    Gd = colmajor(G, dt)
    M = D.dh2_compress(T, Gd, eps=1e-4, mode=D.MODE_FP64 if fp64 else D.MODE_FP32, nearfield=view)
    xs, zs = random_complex_vectors(n, 9, seed=5), random_complex_vectors(n, 9, seed=6)
    gn = np.linalg.norm(G)

    def product(f, v):
        vd = torch.from_numpy(np.ascontiguousarray(v.T)).to("cuda", dt).t()
        out = torch.full((v.shape[1], n), float("nan"), dtype=dt, device="cuda").t()
        f(M, vd, out)
        torch.cuda.synchronize()
        return out.cpu().numpy().astype(np.complex128)

    for f, v, A in ((D.dh2_matvec, xs, G), (D.dh2_matvec_adjoint, zs, G.conj().T)):
        one = np.concatenate([product(f, v[:, j:j + 1]) for j in range(9)], axis=1)
        scale = gn * np.linalg.norm(v, axis=0)
        assert np.all(np.linalg.norm(one - A @ v, axis=0) <= 1e-4 * scale + tol * scale)
        for w in range(2, 10):
            got = product(f, v[:, :w])
            assert np.all(np.linalg.norm(got - one[:, :w], axis=0) <= tol * np.linalg.norm(one[:, :w], axis=0)), w
    y, t = product(D.dh2_matvec, xs), product(D.dh2_matvec_adjoint, zs)
    for j in range(9):
        a, b = np.vdot(zs[:, j], y[:, j]), np.vdot(t[:, j], xs[:, j])
        assert abs(a - b) <= 10 * tol * gn * np.linalg.norm(xs[:, j]) * np.linalg.norm(zs[:, j])


def test_products_on_several_streams_and_threads():
    """The nearfield runs on a second stream beside the transformations (n large enough): products of
    one matrix from several threads, each on a stream of its own, and the use of x and y right after
    the call on the caller's stream give the product of a lone call (bounds as above)."""
    import threading

    D = dev()
    n, kappa = 4200, 12.0
    pts = random_ellipsoid(n)
    T = D.dh2_tree_build(pts, 32, kappa)
    perm = T.perm()
    G = helmholtz_matrix(pts, kappa)[np.ix_(perm, perm)].astype(np.complex64)
    assert (1.0 - T.stats().adm_fraction) * n * n > 2 ** 23
    M = D.dh2_compress(T, colmajor(G, torch.complex64), eps=1e-4)
    xs = torch.randn((8, n), dtype=torch.complex64, device="cuda")
    want = torch.empty_like(xs)
    for i in range(8):
        D.dh2_matvec(M, xs[i], want[i])
    torch.cuda.synchronize()
    got = torch.zeros((8, 20, n), dtype=torch.complex64, device="cuda")
    torch.cuda.synchronize()

    def work(i):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for k in range(20):
                x = xs[i] * 2.0  # made and dropped on this stream
                y = torch.empty_like(x)
                D.dh2_matvec(M, x, y)
                x.zero_()
                got[i, k] = 0.5 * y

    ts = [threading.Thread(target=work, args=(i,)) for i in range(8)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    for i in range(8):
        d = (got[i] - want[i]).norm(dim=1)
        assert float(d.max()) <= 1e-5 * float(want[i].norm())
