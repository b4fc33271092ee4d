"""The Newton reciprocals under the FP64 collision, the MLS weights and the adjoint
(csrc/lbmib_internal.cuh), against division and square root over the ranges they see."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1903_03356_gb300", "csrc")
SOURCE = """
#include "lbmib_internal.cuh"
__global__ void k(const double* x, double* r, double* q, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        r[i] = lbmib::rcp_newton(x[i]);
        q[i] = lbmib::rsqrt_newton(x[i]);
    }
}
extern "C" int newton(const double* x, double* r, double* q, int n) {
    k<<<(n + 255) / 256, 256>>>(x, r, q, n);
    return (int)cudaDeviceSynchronize();
}
"""


def test_newton_reciprocals(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src, lib = tmp_path / "newton.cu", tmp_path / "newton.so"
    src.write_text(SOURCE)
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                           "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-shared", "-I", CSRC,
                           "-o", str(lib), str(src)])
    rng = np.random.default_rng(7)
    x = np.concatenate([
        rng.uniform(0.5, 4.0, 200000),                    # densities, relaxation rates times them
        np.exp(rng.uniform(-1.66, 1.66, 200000)),         # MLS exponentials
        np.exp(rng.uniform(np.log(1e-8), np.log(1e6), 200000)),   # squared edges, weight sums
        np.nextafter(1.0, [0.0, 2.0]), [1.0, 2.0, 0.25],
    ])
    dx = torch.from_numpy(x).cuda()
    r, q = torch.empty_like(dx), torch.empty_like(dx)
    assert ctypes.CDLL(str(lib)).newton(ctypes.c_void_p(dx.data_ptr()), ctypes.c_void_p(r.data_ptr()),
                                        ctypes.c_void_p(q.data_ptr()), len(x)) == 0
    # the last fma's rounding alone, against a correctly rounded quotient
    rcp = 1.0 / x
    assert (np.abs(r.cpu().numpy() - rcp) <= np.spacing(rcp)).all()
    # x y rounded once (half an ulp of the correction, halved), the last fma, and the two
    # roundings of the reference
    ref = 1.0 / np.sqrt(x)
    assert (np.abs(q.cpu().numpy() - ref) <= 3.0 * np.spacing(ref)).all()
