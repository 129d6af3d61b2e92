"""Tensor-core H_eff products where their tiles can go wrong: edges of the 128-row and 16-column
tiles and of the K steps, K lists long enough to fill the pipeline from several segments, rows of the
two spin parts with different K lists, and infinities or NaN there.

Errors are bounded against the same product of absolute values: four roundings of 2^-11 (TF32) or
2^-17 (the BF16 pair) per chained product, twice for a complex one, and 2^-23 for each of the at most
2000 accumulations of an element."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import blocksparse as B  # noqa: E402
from tests import gpu_cases as G  # noqa: E402
from tests.test_digits_gpu import _one_block_case, _oracle  # noqa: E402
from tests.test_heff_gpu import _dev  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {1: 8 * 2.0 ** -11 + 2000 * 2.0 ** -23, 2: 8 * 2.0 ** -17 + 2000 * 2.0 ** -23}


@pytest.fixture(scope="module")
def ctx():
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return P.Context(0, torch.cuda.current_stream())


def _scale(case):
    ab = dict(case, **{k: np.abs(case[k]).astype(complex) for k in ("lflat", "rflat", "tflat")},
              **{k: [e[:4] + (abs(e[4]),) for e in case[k]] for k in ("wi", "wj")})
    return np.max(np.abs(_oracle(ab)))


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("dl,dr,channels", [(1, 1, 2), (7, 33, 3), (8, 16, 30), (16, 17, 2), (65, 96, 12), (128, 49, 2),
                                            (129, 130, 2), (40, 90, 30)])
def test_tile_edges(ctx, prec, real, dl, dr, channels):
    import paper_1512_03318_gb300 as P
    case = _one_block_case(91 + dl, dl, dr, channels)
    if real:
        case = dict(case, **{k: case[k].real.astype(complex) for k in ("lflat", "rflat", "tflat")},
                    **{k: [e[:4] + (complex(e[4].real),) for e in case[k]] for k in ("wi", "wj")})
    ref, tol = _oracle(case), TOL[prec] * _scale(case)
    outs = []
    for per_task, tune in ((0, 0), (1, 0), (0, 1)):
        h = P.Heff(ctx, **G.heff_args(case))
        h.set_option(P.MRD_OPT_REAL, int(real))
        h.set_option(P.MRD_OPT_AUTOTUNE, tune)
        h.set_option(P.MRD_OPT_PER_TASK_LAUNCH, per_task)
        h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
        T = _dev(case["tflat"])
        for _ in range(2):
            out = torch.full_like(T, complex(7.0, -3.0))
            h.apply(T, out, prec)
        h.status()
        outs.append(out.cpu().numpy())
        h.close()
    assert np.max(np.abs(outs[0] - ref)) <= tol
    for o in outs[1:]:   # the order of every element's sum does not depend on the tiles
        assert np.array_equal(o, outs[0])


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("where", ["lflat", "rflat", "tflat"])
@pytest.mark.parametrize("prec", [1, 2])
def test_non_finite_operands(ctx, prec, where, bad):
    """Non-finite exactly where the plain block products are: a row takes nothing from the K blocks
    of its tile's other rows. The next finite environments are computed as before."""
    import paper_1512_03318_gb300 as P
    case = G.random_case(7, 6, 150, 170, 5, 3, 4, 8, 6)
    x = case[where].copy()
    x[len(x) // 3] = bad
    bad_case = dict(case, **{where: x})
    with np.errstate(all="ignore"):
        fine = np.isfinite(_oracle(bad_case))
    assert np.any(fine) and not np.all(fine)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    good, out = torch.empty_like(T), torch.empty_like(T)
    h.apply(T, good, prec)
    h.set_env(_dev(bad_case["lflat"]), _dev(bad_case["rflat"]))
    h.apply(_dev(bad_case["tflat"]), out, prec)
    got = out.cpu().numpy()
    assert np.array_equal(np.isfinite(got), fine)
    assert np.array_equal(got[fine], good.cpu().numpy()[fine])
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    h.apply(T, out, prec)
    assert torch.equal(out, good)
    h.close()
