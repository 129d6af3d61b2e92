"""Digit-split products as a program uses a handle: precisions in turn."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from tests import gpu_cases as G  # noqa: E402
from tests.test_digits_gpu import _one_block_case, _oracle, TOL  # noqa: E402
from tests.test_heff_gpu import _dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return P.Context(0, torch.cuda.current_stream())


def test_precisions_in_turn_keep_their_operands(ctx):
    """FP64 and float-float applications in turn on one handle: once each has run, a change of precision
    launches nothing besides the application (no second planning or packing of the environments), and the
    results stay the same bits."""
    import paper_1512_03318_gb300 as P
    case = _one_block_case(91, 256, 200, 4)
    ref = _oracle(case)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    out = torch.empty_like(T)
    first, launches = {}, {}
    for prec in (0, 0, 3, 3, 0, 3, 0, 0, 3):
        n = P.launch_count()
        h.apply(T, out, prec)
        h.status()
        launches.setdefault(prec, []).append(P.launch_count() - n)
        got = out.cpu().numpy()
        assert np.max(np.abs(got - ref)) <= TOL[prec] * np.max(np.abs(ref))
        assert np.array_equal(got, first.setdefault(prec, got))
    for prec in (0, 3):
        assert len(set(launches[prec][1:])) == 1, launches
    # new environments are packed once for each precision
    h.set_env(_dev(2.0 * case["lflat"]), _dev(case["rflat"]))
    for prec in (0, 3):
        h.apply(T, out, prec)
        assert np.array_equal(out.cpu().numpy(), 2.0 * first[prec])
    h.close()
