"""The parts of the FP64 factorisation that use less than FP64 on the way: the
reciprocal and reciprocal square root of dh2_scalar.cuh over their range against
the exact values.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

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
