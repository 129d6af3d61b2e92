"""FP64 scalars of the Jacobi rotations (csrc/fp64_scalar.cuh) by themselves, against extended precision:
the reciprocal square root to 2 ulp, next to CUDA's rsqrt, and the tangent of the rotation to 4 ulp (a last
correction that is itself rounded, of a value whose residual is rounded against 1), over their ranges.

And the SVD of a charge block far below the others: its singular vectors are as orthogonal as theirs."""
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


@pytest.mark.parametrize("power", [0, -60, -245, -400])
def test_small_block_is_an_isometry(power):
    """One middle sector of the two-site tensor scaled by 2^power (a single Lanczos step leaves the tensor as it
    is): every kept singular vector, of that block too, is orthonormal to 1e-12 as elsewhere."""
    import paper_1512_03318_gb300 as P
    import synth
    from tests.test_dmrg_gpu import _isometry_error
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = P.Context(0, torch.cuda.current_stream())
    lx, ly, chi = 6, 4, 130
    n_sites = lx * ly
    caps = [[(q[0], q[1], d) for q, d in synth.bond_sectors(chi, ly, round(j / ly), synth.substream(97, 7, j), min_dim=1)]
            if 2 <= j <= n_sites - 2 else [] for j in range(n_sites + 1)]
    i = (lx // 2) * ly + ly // 2 - 1
    mpo = P.MPO(None, lx, ly, 1, 4, 1.0, 1.0, P.MRD_BASIS_MIXED)
    d = P.DMRG(ctx, mpo, lx, 0, 100000, seed=5, center=i, caps=caps)
    # tensor i + 1 is grouped by its left (the middle) sector: scale the largest group
    mode, t = d.site(i + 1)
    assert mode == 1
    left, right = d.bond(i + 1), {(int(a), int(b)): int(c) for a, b, c in d.bond(i + 2)}
    m2 = (i + 1) % ly
    cols = [sum(right.get((int(n) + s, (int(k) + s * m2) % ly), 0) for s in (0, 1)) for n, k, _ in left]
    size = [int(dim) * c for (_, _, dim), c in zip(left, cols)]
    g = int(np.argmax(size))
    x = t.copy()
    x[sum(size[:g]):sum(size[:g + 1])] *= 2.0 ** power
    host = np.ascontiguousarray(x)
    d.set_site(i + 1, host.ctypes.data)
    p = P.DMRG.params(100000, 0.0, 1, 0.0, P.MRD_PREC_FP64, 0, 1e-13, svd_mode=3)
    e, _ = d.update(i, +1, p)
    assert np.isfinite(e)
    assert _isometry_error(d.site(i)[1], d.bond(i), d.bond(i + 1), i % ly, ly) < 1e-12
    d.close()
