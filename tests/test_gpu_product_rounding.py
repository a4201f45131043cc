"""Rounding of the FP32 products against the FP64 representation of the same ranks.

A nearfield row has ~1600 columns at leaf size 64.  Summed in chains of c and
then C terms its rounding errors add up to about u / sqrt(3) sqrt(c / 2 + C / 2)
of the sum for terms of random sign: 1.9e-7 for pieces (c = 15, C = 44), 5.8e-7
for one chain.  Bound: 1.5 times the former.
"""
import numpy as np
import pytest

from gpu_cases import dev
from synth import fibonacci_sphere

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_fp32_products_round_by_pieces():
    D = dev()
    n, kappa = 8192, 16.0
    pts = fibonacci_sphere(n)
    T = D.dh2_tree_build(pts, 64, kappa)
    p = torch.from_numpy(pts[T.perm()]).cuda()
    G = torch.empty((n, n), dtype=torch.complex64, device="cuda")
    for s in range(0, n, 1024):
        r = (p[None] - p[s:s + 1024, None]).norm(dim=-1)
        r[torch.arange(1024), torch.arange(s, s + 1024)] = 0.02
        G[s:s + 1024] = torch.polar(1.0 / (4 * np.pi * r), kappa * r).to(torch.complex64)
    M = D.dh2_compress(T, G.t(), eps=1e-4, mode=D.MODE_FP32)
    M64 = D.dh2_compress(T, G.to(torch.complex128).t(), eps=1e-4, mode=D.MODE_FP64,
                         rank_override=(M.ranks(0), M.ranks(1)))
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((3, n), dtype=torch.complex64, device="cuda", generator=g).t()
    y, y64 = torch.empty_like(x.t()).t(), torch.empty((3, n), dtype=torch.complex128, device="cuda").t()
    for f in (D.dh2_matvec, D.dh2_matvec_adjoint):
        f(M, x, y)
        f(M64, x.t().to(torch.complex128).t(), y64)
        assert float((y - y64).norm() / y64.norm()) <= 1.5 * 1.9e-7
