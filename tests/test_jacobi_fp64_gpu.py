"""FP64 Jacobi rounds (svd_mode 3) on blocks around a warp's 32 rows, one column group and several: the
canonical factor is an isometry, and the Schmidt values are those of the float-float form (svd_mode
1), whose columns are orthogonal to 5e-13."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from tests.test_dmrg_gpu import _isometry_error  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chi", [28, 64, 130, 390])
def test_update_fp64_jacobi(chi):
    import paper_1512_03318_gb300 as P
    import synth
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = P.Context(0, torch.cuda.current_stream())
    lx, ly = 6, 4
    n_sites = lx * ly
    caps = [[(q[0], q[1], d) for q, d in synth.bond_sectors(chi, ly, round(j / ly), synth.substream(97, 7, j), min_dim=1)]
            if 2 <= j <= n_sites - 2 else [] for j in range(n_sites + 1)]
    i = (lx // 2) * ly + ly // 2 - 1
    spectra = []
    for mode in (3, 1):
        mpo = P.MPO(None, lx, ly, 1, 4, 1.0, 1.0, P.MRD_BASIS_MIXED)
        d = P.DMRG(ctx, mpo, lx, 0, max(2 * chi, 2), seed=5, center=i, caps=caps)
        p = P.DMRG.params(max(2 * chi, 2), 0.0, 6, 0.0, P.MRD_PREC_FP64, 0, 1e-13, svd_mode=mode)
        e, trunc = d.update(i, +1, p)
        assert math.isfinite(e)
        assert _isometry_error(d.site(i)[1], d.bond(i), d.bond(i + 1), i % ly, ly) < 1e-12
        c = d.site(i + 1)[1]
        assert abs(np.vdot(c, c).real - 1.0) < 1e-12
        spectra.append(np.sort(np.concatenate([np.asarray(v) for v in d.schmidt()[1].values()]))[::-1])
        d.close()
    n = min(len(s) for s in spectra)
    assert n > 0 and np.max(np.abs(spectra[0][:n] - spectra[1][:n])) < 1e-11
