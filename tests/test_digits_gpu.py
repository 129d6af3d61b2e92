"""Digit-split tensor-core products (the FP64 and float-float forms of H_eff and of the DMRG
GEMMs) where their tiling, cutting and scaling can go wrong.

Operands are 62-bit (FP64) or 55-bit (float-float) fixed-point numbers against the largest entry
of their row or column. A real product's dropped digit pairs and operand roundings are below
8 * 2^-62 (8 * 2^-55) of the two largest entries; a complex product of K terms is off by at most
16 K times that, and the bounds below allow that worst case for each of the two chained products
(K at most 2^9 here, 2^9 * 16 * 2^-59 = 2^-46 = 1.5e-14; 2^-39 = 1.9e-12), relative to the largest
possible output, which the largest element stays within a factor of 10 of."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from oracle import blocksparse as B  # noqa: E402
from tests import gpu_cases as G  # noqa: E402
from tests.test_heff_gpu import _dev  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 3: 1e-11}


@pytest.fixture(scope="module")
def ctx():
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return P.Context(0, torch.cuda.current_stream())


def _oracle(case):
    return B.heff_apply(case["left"], case["right"], case["m1"], case["m2"], case["mod"], case["cl"], case["cm"],
                        case["cr"], case["wi"], case["wj"], case["lflat"], case["rflat"], case["tflat"])


def _one_block_case(seed, dl, dr, channels):
    """Every charge zero modulus 1 (m = 0, diagonal entries): two middle sectors whose blocks are dl
    x dr, so that the tile edges are exactly those of dl and dr."""
    left = B.BondSectors([((5, 0), dl)])
    right = B.BondSectors([((5, 0), dr), ((6, 0), max(1, dr // 2))])
    c = [(0, 0)] * channels
    u = synth.uniform_pm1(synth.substream(seed, 3), 4 * channels * channels)
    ent = [(w, x, s, s, complex(u[2 * (w * channels + x)], u[2 * (w * channels + x) + 1]))
           for w in range(channels) for x in range(channels) for s in (0, 1)]
    return G.finish_case(seed, left, right, 0, 0, 1, c, c, c, ent, ent)


# rows / columns at the edges of the 128-row and 32- / 16-column tiles and of the K steps of 16,
# and a chain long enough to be cut along K (30 channels)
@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("dl,dr,channels", [(1, 1, 2), (7, 33, 3), (8, 16, 30), (16, 17, 2), (31, 32, 2), (128, 31, 2),
                                            (129, 48, 2), (255, 7, 2), (136, 257, 2), (40, 90, 30)])
def test_tile_edges(ctx, prec, dl, dr, channels):
    import paper_1512_03318_gb300 as P
    case = _one_block_case(61 + dl, dl, dr, channels)
    ref = _oracle(case)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    outs = []
    for per_task in (0, 0, 1, 0):
        h.set_option(P.MRD_OPT_PER_TASK_LAUNCH, per_task)
        out = torch.full_like(T, complex(7.0, -3.0))
        h.apply(T, out, prec)
        h.status()
        outs.append(out.cpu().numpy())
    assert np.max(np.abs(outs[0] - ref)) <= TOL[prec] * np.max(np.abs(ref))
    for o in outs[1:]:   # exact integer sums: the same bits however the tiles are cut and launched
        assert np.array_equal(o, outs[0])
    h.close()


@pytest.mark.parametrize("prec", [0, 3])
def test_graded_and_tiny_operands(ctx, prec):
    """Columns of theta over 40 decades, an exactly zero row, and numbers far from 1: the errors stay
    below the largest output's share."""
    import paper_1512_03318_gb300 as P
    case = dict(_one_block_case(67, 90, 70, 2))
    lay = case["lay"]
    scale = 1e-120
    t = case["tflat"].copy()
    for m in lay:
        blk = t[m["offset"]: m["offset"] + m["rowdim"] * m["coldim"]].reshape(m["rowdim"], m["coldim"])
        blk *= 10.0 ** -(np.arange(m["coldim"]) % 40)[None, :]
        blk[3 % m["rowdim"], :] = 0.0
    case["tflat"] = t * scale
    ref = _oracle(case)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    out = torch.empty_like(T)
    h.apply(T, out, prec)
    got = out.cpu().numpy()
    assert np.max(np.abs(got - ref)) <= TOL[prec] * np.max(np.abs(ref))
    h.close()


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("where", ["theta", "left", "right"])
def test_non_finite_operands(ctx, bad, where):
    """An infinity or NaN has no fixed-point form: the FP64 product is then the FP64 kernel's
    (non-finite exactly where the plain product is), and the next finite product is right again."""
    import paper_1512_03318_gb300 as P
    case = dict(_one_block_case(71, 90, 70, 2))
    good = _oracle(case)
    key = {"theta": "tflat", "left": "lflat", "right": "rflat"}[where]
    x = case[key].copy()
    x[len(x) // 3] = bad
    bad_case = dict(case, **{key: x})
    with np.errstate(all="ignore"):
        ref = _oracle(bad_case)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(_dev(bad_case["lflat"]), _dev(bad_case["rflat"]))
    T = _dev(bad_case["tflat"])
    out = torch.empty_like(T)
    h.apply(T, out, 0)
    got = out.cpu().numpy()
    assert np.any(~np.isfinite(ref))
    fine = np.isfinite(ref)
    assert np.all(~np.isfinite(got[~fine]))
    assert np.max(np.abs(got[fine] - ref[fine]), initial=0.0) <= TOL[0] * np.max(np.abs(good))
    h.apply(T, out, 3)                       # float-float: non-finite there too
    assert np.all(~np.isfinite(out.cpu().numpy()[~fine]))
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    h.apply(T, out, 0)
    assert np.max(np.abs(out.cpu().numpy() - good)) <= TOL[0] * np.max(np.abs(good))
    h.close()


def test_wait_limit_reports_timeout(ctx):
    """A zero wait limit makes every wait of the FP64 product give up before any copy or MMA; the
    status reports it once and the next product is right."""
    import paper_1512_03318_gb300 as P
    case = _one_block_case(73, 129, 90, 3)
    ref = _oracle(case)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    out = torch.empty_like(T)
    h.set_option(P.MRD_OPT_WAIT_LIMIT_US, 0)
    h.apply(T, out, 0)
    with pytest.raises(P.MrdError) as ex:
        h.status()
    assert ex.value.code == -7
    h.status()
    h.set_option(P.MRD_OPT_WAIT_LIMIT_US, 1000000)
    h.apply(T, out, 0)
    h.status()
    assert np.max(np.abs(out.cpu().numpy() - ref)) <= TOL[0] * np.max(np.abs(ref))
    h.close()
