"""Lowest Ritz value of a Lanczos run of k steps, from the smallest k to the largest, at scales of H
where its brackets differ: the oracle's run with the same start vector has the same to rounding."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import dmrg as D  # noqa: E402
from tests import gpu_cases as G  # noqa: E402
from tests.test_lanczos_gpu import _hermitian_case, _oracle_op  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-7, -3e8])
@pytest.mark.parametrize("k", [1, 2, 3, 9, 17, 33, 60])
def test_ritz_value(k, scale):
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = P.Context(0, torch.cuda.current_stream())
    case = _hermitian_case(47, 5, 60, 64, 2, 4)
    case = dict(case, lflat=case["lflat"] * scale)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(torch.from_numpy(case["lflat"]).cuda(), torch.from_numpy(case["rflat"]).cuda())
    th = torch.from_numpy(case["tflat"].copy()).cuda()
    e, it = h.lanczos(th, max_iter=k, tol=0.0)
    e_or, v_or, it_or = D.lanczos_ground(_oracle_op(case), case["tflat"].copy(), kmax=k, tol=0.0)
    assert it == k and it_or == k
    assert abs(e - e_or) < 1e-11 * abs(e_or)
    assert abs(abs(np.vdot(th.cpu().numpy(), v_or)) - 1) < 1e-9
    h.close()
