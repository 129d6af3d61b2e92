"""Digit-split products by themselves: forced for every size (MRD_OPT_DIGITS), with the arithmetic that ran
asserted (mrd_heff_form), against exact sums.

The operands are multiples of 2^-52 below 1. With one channel of value 1 and theta an identity (K ones on
each block's diagonal), step 1 copies LW, and step 2 is one product of K terms: a result is off by its own
rounding (2^-53 of it) and by the fixed point. The latter per real product: two operand roundings and seven
dropped pairs of digits, independent and of either sign, 2^-62 (62-bit form, FP64) or 2^-56.2 (55-bit form,
float-float) of the bounds 1 x 1, rms; a complex product has 2 K of them, and the bounds below allow eight
times the rms of their sum. Results of 55-bit digits, or without the last digits, miss the FP64 bound; those
of FMAs (K terms, a rounding of 2^-53 of the partial sum each) and of float-float sums miss theirs."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from oracle import blocksparse as B  # noqa: E402
from tests import gpu_cases as G  # noqa: E402
from tests.test_digits_gpu import TOL, _one_block_case, _oracle  # noqa: E402
from tests.test_heff_gpu import _dev  # noqa: E402

pytestmark = pytest.mark.gpu

DIGITS, BITS = {0: 62.0, 3: 56.2}, 52


@pytest.fixture(scope="module")
def ctx():
    import paper_1512_03318_gb300 as P
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return P.Context(0, torch.cuda.current_stream())


def _ints(x):
    """Numbers that are multiples of 2^-BITS as Python integers (real, imaginary)."""
    f = lambda v: np.array([int(e) for e in np.ldexp(v, BITS).reshape(-1)], dtype=object).reshape(v.shape)
    return f(np.real(x)), f(np.imag(x))


def _errors(got, a, b):
    """(|got - a @ b|, |a @ b|) of the real and of the imaginary parts, the differences exact."""
    (ar, ai), (br, bi) = _ints(a), _ints(b)
    out = []
    for g, e in ((got.real, ar.dot(br) - ai.dot(bi)), (got.imag, ar.dot(bi) + ai.dot(br))):
        ref = [Fraction(x, 2 ** (2 * BITS)) for x in e.reshape(-1)]
        out.append((np.array([abs(float(Fraction(float(y)) - x)) for y, x in zip(g.reshape(-1), ref)]),
                    np.array([abs(float(x)) for x in ref])))
    return out


# edges of the 128-row, 32- and 16-column tiles, of K steps of 16 and of their halves
@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("dl,dr", [(1, 1), (7, 33), (8, 16), (16, 17), (31, 32), (33, 33), (128, 31), (129, 48), (60, 136),
                                   (200, 150)])
def test_one_product_exactly(ctx, prec, dl, dr):
    import paper_1512_03318_gb300 as P
    left = B.BondSectors([((5, 0), dl)])
    right = B.BondSectors([((5, 0), dr), ((6, 0), max(1, dr // 2))])
    c = [(0, 0)]
    ent = [(0, 0, s, s, 1.0 + 0.0j) for s in (0, 1)]
    case = G.finish_case(131 + dl, left, right, 0, 0, 1, c, c, c, ent, ent)
    grid = lambda x: np.ldexp(np.rint(np.ldexp(x.real, BITS)), -BITS) + 1j * np.ldexp(np.rint(np.ldexp(x.imag, BITS)), -BITS)
    lf, rf, t = grid(case["lflat"]), grid(case["rflat"]), np.zeros_like(case["tflat"])
    for m in case["lay"]:
        blk = t[m["offset"]: m["offset"] + m["rowdim"] * m["coldim"]].reshape(m["rowdim"], m["coldim"])
        for _, _, da, ro in m["rows"]:
            for _, _, db, co in m["cols"]:
                k = min(da, db)
                blk[ro + np.arange(k), co + np.arange(k)] = 1.0
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_option(P.MRD_OPT_DIGITS, 2)
    h.set_env(_dev(lf), _dev(rf))
    T = _dev(t)
    outs = []
    for per_task in (0, 1):
        h.set_option(P.MRD_OPT_PER_TASK_LAUNCH, per_task)
        out = torch.full_like(T, complex(7.0, -3.0))
        h.apply(T, out, prec)
        h.status()
        assert h.form() == 1
        outs.append(out.cpu().numpy())
    assert np.array_equal(outs[0], outs[1])
    blocks = {row[1]: rf[row[3]:row[3] + row[4] * row[5]].reshape(row[4], row[5]) for row in case["rl"]}
    (_, _, _, off, d0, d1), = case["ll"]
    L = lf[off:off + d0 * d1].reshape(d0, d1)
    for m in case["lay"]:
        got = outs[0][m["offset"]: m["offset"] + m["rowdim"] * m["coldim"]].reshape(m["rowdim"], m["coldim"])
        for _, _, da, ro in m["rows"]:
            for _, bi, db, co in m["cols"]:
                k = min(da, db)
                for err, ref in _errors(got[ro:ro + da, co:co + db], L[:, :k], blocks[bi][:k]):
                    assert np.all(err <= 2.0 ** -53 * ref + 8.0 * np.sqrt(2.0 * k) * 2.0 ** -DIGITS[prec])
    h.close()


# the shapes of the tile-edge tests, with the arithmetic that runs asserted; 30 channels are cut along K
@pytest.mark.parametrize("prec,real", [(0, False), (3, False), (3, True)])
@pytest.mark.parametrize("dl,dr,channels", [(1, 1, 2), (7, 33, 3), (8, 16, 30), (16, 17, 2), (31, 32, 2), (128, 31, 2),
                                            (129, 48, 2), (255, 7, 2), (136, 257, 2), (40, 90, 30)])
def test_forced_digits(ctx, prec, real, dl, dr, channels):
    import paper_1512_03318_gb300 as P
    case = dict(_one_block_case(161 + dl, dl, dr, channels))
    if real:
        case.update(lflat=case["lflat"].real + 0j, rflat=case["rflat"].real + 0j, tflat=case["tflat"].real + 0j,
                    wi=[(*e[:4], complex(e[4].real)) for e in case["wi"]], wj=[(*e[:4], complex(e[4].real)) for e in case["wj"]])
    ref = _oracle(case)
    h = P.Heff(ctx, **G.heff_args(case))
    assert h.form() == -1
    if real:
        h.set_option(P.MRD_OPT_REAL, 1)
    h.set_env(_dev(case["lflat"]), _dev(case["rflat"]))
    T = _dev(case["tflat"])
    outs = {}
    for mode, per_task in ((2, 0), (2, 1), (0, 0), (2, 0)):
        h.set_option(P.MRD_OPT_DIGITS, mode)
        h.set_option(P.MRD_OPT_PER_TASK_LAUNCH, per_task)
        out = torch.full_like(T, complex(7.0, -3.0))
        h.apply(T, out, prec)
        h.status()
        assert h.form() == (1 if mode else 0)
        got = out.cpu().numpy()
        assert np.max(np.abs(got - ref)) <= TOL[prec] * np.max(np.abs(ref))
        assert np.array_equal(got, outs.setdefault(mode, got))
    with pytest.raises(P.MrdError):
        h.set_option(P.MRD_OPT_DIGITS, 3)
    h.close()


@pytest.mark.parametrize("prec,ly,chi,form", [(0, 4, 48, 1), (0, 8, 250, 1), (3, 4, 40, 0), (3, 8, 400, 0), (3, 8, 1024, 1)])
def test_default_choice(ctx, prec, ly, chi, form):
    """What the default choice takes at sizes on either side of it."""
    import paper_1512_03318_gb300 as P
    mpo = P.MPO(None, 4, ly, 1, ly, 1.0, 1.0, P.MRD_BASIS_MIXED)
    site = 2 * ly + ly // 2 - 1
    sec = lambda tag: np.array([[q[0], q[1], d] for q, d in synth.bond_sectors(chi, ly, 10, synth.substream(181, tag), min_dim=1)],
                               dtype=np.int32)
    wi, wj = mpo.site(site), mpo.site(site + 1)
    h = P.Heff(ctx, left=sec(1), right=sec(2), m1=site % ly, m2=(site + 1) % ly, modulus=mpo.modulus, cl=mpo.bond(site),
               cm=mpo.bond(site + 1), cr=mpo.bond(site + 2), wi_idx=wi[0], wi_val=wi[1], wj_idx=wj[0], wj_val=wj[1])
    z = lambda n: torch.ones(n, dtype=torch.complex128, device="cuda")
    h.set_env(z(h.lenv_len), z(h.renv_len))
    T = z(h.theta_len)
    h.apply(T, torch.empty_like(T), prec)
    h.status()
    assert h.form() == form
    h.close()
