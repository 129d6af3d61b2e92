"""Folding the environments with the MPO (LW and WR) where the fold's chunks and entry forms can go
wrong: blocks of one element (more of them in a chunk than a CTA stages), blocks around and beyond a
chunk, more entries per block than are staged, entries of value 1, -1, real and complex.

The FP64 H_eff application of a folded case against the oracle: sums of at most 300 * 130 terms in
64-bit arithmetic, relative to the largest output, as in the other FP64 cases."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import blocksparse as B  # noqa: E402
from tests import gpu_cases as G  # noqa: E402
from tests.test_heff_gpu import _dev  # noqa: E402

pytestmark = pytest.mark.gpu

VALUES = [1.0, -1.0, 0.75, -2.5, 0.5 + 0.25j, -1j]


def _case(seed, dl, dr, channels, full):
    left = B.BondSectors([((5, 0), dl)])
    right = B.BondSectors([((5, 0), dr), ((6, 0), max(1, dr // 2))])
    c = [(0, 0)] * channels
    pairs = [(w, x) for w in range(channels) for x in (range(channels) if full else {w, (w + 1) % channels})]
    ent = [(w, x, s, s, complex(VALUES[(w + 3 * x + s) % len(VALUES)])) for w, x in pairs for s in (0, 1)]
    return G.finish_case(seed, left, right, 0, 0, 1, c, c, c, ent, ent)


@pytest.mark.parametrize("dl,dr,channels,full", [(1, 1, 300, False), (3, 2, 40, True), (90, 91, 3, True),
                                                 (130, 64, 35, True), (17, 5, 7, False)])
def test_fold_edges(dl, dr, channels, full):
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = P.Context(0, torch.cuda.current_stream())
    case = _case(83 + dl, dl, dr, channels, full)
    ref = B.heff_apply(case["left"], case["right"], case["m1"], case["m2"], case["mod"], case["cl"], case["cm"],
                       case["cr"], case["wi"], case["wj"], case["lflat"], case["rflat"], case["tflat"])
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    out = torch.full_like(T, complex(7.0, -3.0))
    h.apply(T, out, 0)
    assert np.max(np.abs(out.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))
    h.close()
