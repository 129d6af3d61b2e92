"""FP64 scalars of the Jacobi rotations (csrc/fp64_scalar.cuh) by themselves, against extended precision:
the reciprocal square root to 2 ulp, next to CUDA's rsqrt, and the tangent of the rotation to 4 ulp (a last
correction that is itself rounded, of a value whose residual is rounded against 1), over their ranges."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "fp64_scalar.cuh"
__global__ void k(const double* x, double* a, double* b, double* t, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double v = x[i] < 0 ? -x[i] : x[i];
    a[i] = mrd::rsqrt_fp64(v);
    b[i] = rsqrt(v);
    t[i] = mrd::jacobi_tangent(x[i]);
  }
}
extern "C" int run(const double* x, double* a, double* b, double* t, int n) {
  k<<<64, 256>>>(x, a, b, t, n);
  return (int)cudaDeviceSynchronize();
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("scalar")
    (d / "s.cu").write_text(SRC)
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    so = str(d / "libs.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-shared", "-Xcompiler", "-fPIC",
                    "-I", os.path.join(ROOT, "paper_1512_03318_gb300", "csrc"), str(d / "s.cu"), "-o", so], check=True)
    return ctypes.CDLL(so)


def _run(lib, x):
    x = np.ascontiguousarray(x, dtype=np.float64)
    d = torch.from_numpy(x).cuda()
    out = [torch.empty_like(d) for _ in range(3)]
    assert lib.run(*[ctypes.c_void_p(v.data_ptr()) for v in (d, *out)], ctypes.c_int(len(x))) == 0
    return [o.cpu().numpy() for o in out]


def test_reciprocal_square_root(lib):
    rng = np.random.RandomState(5)
    x = np.concatenate([2.0 ** rng.uniform(-1000, 1000, 200000), 2.0 ** np.arange(-1000, 1001),
                        np.nextafter(2.0 ** np.arange(-1000, 1001), 0.0), rng.uniform(1.0, 4.0, 200000)])
    got, cuda, _ = _run(lib, x)
    ref = 1.0 / np.sqrt(x.astype(np.longdouble))
    ulp = np.spacing(ref.astype(np.float64))
    assert np.max(np.abs(got - ref) / ulp) <= 2.0
    assert np.max(np.abs(got - cuda) / ulp) <= 3.0


def test_tangent(lib):
    rng = np.random.RandomState(7)
    mag = np.concatenate([2.0 ** rng.uniform(-80, 119, 300000), rng.uniform(0.0, 4.0, 200000), [0.0]])
    x = np.concatenate([mag, -mag])
    t = _run(lib, x)[2]
    z = np.abs(x).astype(np.longdouble)
    ref = 1.0 / (z + np.sqrt(1.0 + z * z))
    ref = np.where(np.signbit(x), -ref, ref)
    assert np.max(np.abs(t - ref) / np.spacing(np.abs(ref).astype(np.float64))) <= 4.0
