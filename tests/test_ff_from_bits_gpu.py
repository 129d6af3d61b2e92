"""Float-float numbers taken from the bits of an FP64 number (csrc/ff.cuh): over all exponents, ties and carries
they hold what the conversion in FP64 arithmetic holds. The low part is at most half an ulp of the high one,
and the sum is right to 2^-49 (28 bits rounded to 24) or half of the smallest FP32 number."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "ff.cuh"
__global__ void k(const double* x, float* hi, float* lo, float* hi2, float* lo2, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const mrd::FF a = mrd::ff_from_bits(x[i]), b = mrd::ff_from(x[i]);
    hi[i] = a.hi; lo[i] = a.lo; hi2[i] = b.hi; lo2[i] = b.lo;
  }
}
extern "C" int run(const double* x, float* a, float* b, float* c, float* d, int n) {
  k<<<64, 256>>>(x, a, b, c, d, n);
  return (int)cudaDeviceSynchronize();
}
'''


def _inputs():
    rng = np.random.RandomState(11)
    base = np.concatenate([2.0 ** rng.uniform(-160, 127.9, 200000), 2.0 ** np.arange(-160, 128)])
    m = base.view(np.int64) & ~np.int64((1 << 29) - 1)
    low = [m, m | (1 << 28), (m | (1 << 28)) + 1, (m | (1 << 28)) - 1, m | ((1 << 29) - 1), m | 1,
           m | (((1 << 23) - 1) << 29) | (1 << 28)]   # the last: the carry reaches the exponent
    x = np.concatenate([base] + [v.view(np.float64) for v in low] + [np.zeros(1)])
    x = x[x < 2.0 ** 127.99]
    return np.concatenate([x, -x])


def test_conversion_from_bits(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    (tmp_path / "s.cu").write_text(SRC)
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    so = str(tmp_path / "libff.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-shared", "-Xcompiler", "-fPIC",
                    "-I", os.path.join(ROOT, "paper_1512_03318_gb300", "csrc"), str(tmp_path / "s.cu"), "-o", so], check=True)
    x = _inputs()
    d = torch.from_numpy(x).cuda()
    out = [torch.empty(len(x), dtype=torch.float32, device="cuda") for _ in range(4)]
    assert ctypes.CDLL(so).run(*[ctypes.c_void_p(v.data_ptr()) for v in (d, *out)], ctypes.c_int(len(x))) == 0
    hi, lo, hi2, lo2 = [o.cpu().numpy() for o in out]
    tie = np.abs(lo2) * 2.0 == np.spacing(np.abs(hi2))   # half way: either neighbour is right
    assert np.array_equal(hi[~tie], hi2[~tie]) and np.array_equal(lo[~tie], lo2[~tie])
    assert np.all(np.abs(lo) <= np.spacing(np.abs(hi)) / 2)
    rest = (x - hi.astype(np.float64)) - lo.astype(np.float64)   # both differences are exact
    assert np.all(np.abs(rest) <= np.maximum(np.abs(x) * 2.0 ** -49, 2.0 ** -150))
