"""Folding the environments over flat chunks where tiny blocks lie between large ones: more blocks in a chunk
than a CTA stages the offsets of, so that elements walk beyond them, and chunks of one block only."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import blocksparse as B  # noqa: E402
from tests import gpu_cases as G  # noqa: E402
from tests.test_heff_gpu import _dev  # noqa: E402

pytestmark = pytest.mark.gpu

VALUES = [1.0, -1.0, 0.75, 0.5 + 0.25j]


# `tiny` sectors of dimension 1 and one large one on each bond; the flat form takes means above 128
# elements per block, a CTA stages 257 offsets, a chunk here has at least 1024 elements
@pytest.mark.parametrize("tiny,large", [(300, 330), (520, 400), (40, 260)])
def test_tiny_blocks_between_large_ones(tiny, large):
    """FP64 H_eff application against the oracle: sums of at most 2 * 400 * 400 terms in 64-bit arithmetic."""
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = P.Context(0, torch.cuda.current_stream())
    left = B.BondSectors([((n, 0), 1) for n in range(tiny)] + [((tiny, 0), large)])
    right = B.BondSectors([((n, 0), 1) for n in range(tiny + 1)] + [((tiny + 1, 0), large)])
    c = [(0, 0)] * 2
    ent = [(w, x, s, s, complex(VALUES[(w + 2 * x + s) % 4])) for w in (0, 1) for x in (0, 1) for s in (0, 1)]
    case = G.finish_case(191 + tiny, left, right, 0, 0, 1, c, c, c, ent, ent)
    blocks, length = 2 * 2 * (tiny + 1), 2 * 2 * (tiny + large * large)
    assert length > 128 * blocks and max(256, min(8192, length // 608)) >= 256
    if tiny > 257:
        assert length // 608 > tiny            # a whole run of tiny blocks fits one chunk
    ref = B.heff_apply(case["left"], case["right"], case["m1"], case["m2"], case["mod"], case["cl"], case["cm"],
                       case["cr"], case["wi"], case["wj"], case["lflat"], case["rflat"], case["tflat"])
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_option(P.MRD_OPT_DIGITS, 0)
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    out = torch.full_like(T, complex(7.0, -3.0))
    h.apply(T, out, 0)
    got = out.cpu().numpy()
    # block by block: the tiny ones have their own scale
    for m in case["lay"]:
        view = lambda x: x[m["offset"]: m["offset"] + m["rowdim"] * m["coldim"]].reshape(m["rowdim"], m["coldim"])
        for _, _, da, ro in m["rows"]:
            for _, _, db, co in m["cols"]:
                g, r = view(got)[ro:ro + da, co:co + db], view(ref)[ro:ro + da, co:co + db]
                assert np.max(np.abs(g - r)) <= 1e-12 * max(np.max(np.abs(r)), 1.0)
    h.close()
