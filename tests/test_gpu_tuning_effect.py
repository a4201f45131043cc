"""The tuning table acts where it says, and the autotuner times only what acts."""
import numpy as np
import pytest

from gpu_cases import colmajor, dev
from synth import helmholtz_matrix, random_ellipsoid

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(autouse=True)
def _restore_table():
    D = dev()
    saved = D.tuning()
    yield
    D.set_tuning(saved)


def _problem(n, leaf, kappa, dtype=torch.complex64, **eta):
    D = dev()
    pts = random_ellipsoid(n)
    T = D.dh2_tree_build(pts, leaf, kappa, **eta)
    p = torch.from_numpy(pts[T.perm()]).cuda()
    G = torch.empty((n, n), dtype=dtype, device="cuda")
    for s in range(0, n, 1024):
        r = (p[None] - p[s:s + 1024, None]).norm(dim=-1)
        r[torch.arange(r.shape[0]), torch.arange(s, s + r.shape[0])] = 0.02
        G[s:s + 1024] = torch.polar(1.0 / (4 * np.pi * r), kappa * r).to(dtype)
    return D, T, G.t()


def _classes(log, knob):
    return sorted({r["cls"] for r in log if r["knob"] == knob})


@pytest.mark.parametrize("mode", ["fp32", "mixed"])
def test_classes_with_launches_of_their_own_are_tuned(mode):
    """Many leaf pairs: every class launches its own Jacobi and is tuned; few: only the class whose
    launch takes them all (and, for jacobi_tpp, classes that the level steps launch)."""
    D, T, G = _problem(12000, 64, 32.0)
    m = D.MODE_FP32 if mode == "fp32" else D.MODE_MIXED_BF16X3
    assert sum(int(T.pairs(s)["leaf"].sum()) for s in (0, 1)) > 2432
    table, log = D.autotune(T, G, eps=1e-4, mode=m, reps=1)
    assert _classes(log, "jacobi_narrow") == [0, 1, 2, 3] == _classes(log, "jacobi_tpp")
    for c in range(4):
        for knob in ("jacobi_narrow", "jacobi_tpp"):
            rec = [r for r in log if r["knob"] == knob and r["cls"] == c]
            assert table[knob][c] == min(rec, key=lambda r: r["ms"])["value"]
    D, T, G = _problem(4096, 64, 12.0)
    before = D.tuning()
    table, log = D.autotune(T, G, eps=1e-4, mode=m, reps=1)
    assert _classes(log, "jacobi_narrow") == [3] == _classes(log, "jacobi_tpp")
    assert table["jacobi_narrow"][:3] == before["jacobi_narrow"][:3]
    assert table["jacobi_tpp"][:3] == before["jacobi_tpp"][:3]


def test_segment_width_is_tuned_only_where_it_acts():
    """Wide level pairs of at most 64 rows: the FP32 mode factors them from Gram matrices, without the
    table's segments; FP64 by those segments."""
    for mode, dt, want in (("fp32", torch.complex64, False), ("fp64", torch.complex128, True)):
        D, T, G = _problem(4096, 32, 12.0, dt, eta1=20.0, eta2=5.0)
        assert max(int(T.pairs(0)["ncols"][T.pairs(0)["leaf"] == 0].max()), 0) > 1024
        _, log = D.autotune(T, G, eps=1e-3, mode=D.MODE_FP64 if mode == "fp64" else D.MODE_FP32, reps=1)
        assert bool([r for r in log if r["knob"] == "level_seg_cols"]) == want


def test_jacobi_width_acts_on_fp64_leaf_pairs():
    """Another number of threads per column pair sums the rotation products in another order: the
    singular values keep FP64 accuracy but not every bit."""
    n, kappa = 2048, 6.0
    D = dev()
    pts = random_ellipsoid(n)
    T = D.dh2_tree_build(pts, 64, kappa)
    G = colmajor(helmholtz_matrix(pts, kappa)[np.ix_(T.perm(), T.perm())], torch.complex128)
    leafs = np.flatnonzero(T.pairs(0)["leaf"])
    sig = {}
    for w in (4, 8, 16, 32):
        t = D.tuning()
        t["jacobi_tpp"] = [w] * 5
        D.set_tuning(t)
        M = D.dh2_compress(T, G, eps=1e-4, mode=D.MODE_FP64)
        sig[w] = np.concatenate([M.sigma(0, int(q)) for q in leafs])
    assert np.array_equal(sig[4], sig[32])  # the default's FP64 choice
    for w in (8, 16):
        assert not np.array_equal(sig[w], sig[4])
        assert np.max(np.abs(sig[w] - sig[4])) <= 64 * 64 * 2.0 ** -53 * sig[4].max()
    assert not np.array_equal(sig[8], sig[16])
