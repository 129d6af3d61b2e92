"""What digit-split products cannot represent is computed again in FP64: infinities, NaN, and operands
graded against each other along K."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import synth  # noqa: E402
from oracle import blocksparse as B  # noqa: E402
from tests import gpu_cases as G  # noqa: E402
from tests import test_env_gpu as E  # noqa: E402
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


def _spin_channels(seed, dl, dr, channels, own):
    """Modulus 1, diagonal entries. With `own`, channel x is fed by spin s1 = x mod 2 only and
    becomes channel x of the right environment, so the two row parts of an output block
    multiply different right blocks."""
    left = B.BondSectors([((5, 0), dl), ((6, 0), dl)])
    right = B.BondSectors([((5, 0), dr), ((6, 0), dr), ((7, 0), dr)])
    c = [(0, 0)] * channels
    u = synth.uniform_pm1(synth.substream(seed, 3), 4 * channels * channels)
    wi = [(w, x, s, s, complex(u[2 * (w * channels + x)], u[2 * (w * channels + x) + 1]))
          for w in range(channels) for x in range(channels) for s in (0, 1) if not own or x % 2 == s]
    wj = [(x, x, s, s, complex(1.0, -0.5)) for x in range(channels) for s in (0, 1)] if own else wi
    return G.finish_case(seed, left, right, 0, 0, 1, c, c, c, wi, wj)


@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_right_block_stays_with_its_part(ctx, prec, bad):
    """An infinity or NaN in a right block that one spin part multiplies leaves the other part's outputs
    finite and right, and that part's own non-finite where the plain product is."""
    import paper_1512_03318_gb300 as P
    case = dict(_spin_channels(79, 120, 96, 12, True))
    good = _oracle(case)
    r = case["rflat"].copy()
    off, d0, d1 = next(row[3:] for row in case["rl"] if row[:2] == (3, 1))
    r[off + (d0 // 2) * d1 + d1 // 3] = bad          # a block of channel 3: spin part 1 only
    case["rflat"] = r
    with np.errstate(all="ignore"):
        ref = _oracle(case)
    fine = np.isfinite(ref)
    assert np.any(~fine) and np.any(fine)
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_option(P.MRD_OPT_DIGITS, 2)
    h.set_env(_dev(case["lflat"]), _dev(r))
    T = _dev(case["tflat"])
    out = torch.empty_like(T)
    h.apply(T, out, prec)
    h.status()
    assert h.form() == 1
    got = out.cpu().numpy()
    assert np.all(np.isfinite(got[fine]))
    assert np.all(~np.isfinite(got[~fine]))
    assert np.max(np.abs(got[fine] - ref[fine])) <= TOL[prec] * np.max(np.abs(good))
    h.close()


def _raw_env(d, bond, side):
    """Environment as real numbers (an infinite imaginary part must not touch the real one)."""
    import ctypes
    import paper_1512_03318_gb300 as P
    n = ctypes.c_int64()
    x = np.zeros(2 * d.env_len(bond, side))
    d.ctx.check(P.lib().mrd_dmrg_env(d.h, bond, side, ctypes.byref(n), x.ctypes.data_as(ctypes.POINTER(ctypes.c_double))))
    return x


@pytest.mark.parametrize("direction", [+1, -1])
@pytest.mark.parametrize("prec", [0, 3])
def test_env_update_non_finite(ctx, direction, prec):
    """Environment update from a site tensor with one infinite entry: non-finite exactly where the plain
    sums are, the rest right."""
    import paper_1512_03318_gb300 as P
    ly, chi = 4, 400
    mpo = P.MPO(None, 6, ly, 1, 4, 1.0, 1.0, P.MRD_BASIS_MIXED)
    d = P.DMRG(ctx, mpo, 12, 0, chi, seed=3, center=12)
    j = 10 if direction > 0 else 14
    _, t = d.site(j)
    x = t.copy()
    x[len(x) // 2] = np.inf
    host = np.ascontiguousarray(x)
    d.set_site(j, host.ctypes.data)
    d.env_update(j, direction, prec)
    with np.errstate(all="ignore"):
        pairs = E.oracle_left(d, mpo, j, d.env(j, 0)) if direction > 0 else E.oracle_right(d, mpo, j, d.env(j + 1, 1))
    flat = _raw_env(d, j + 1, 0) if direction > 0 else _raw_env(d, j, 1)
    n_bad = 0
    for (w, xi, xpi, off, d0, d1), blk in pairs:
        got = flat[2 * off:2 * (off + d0 * d1)]
        ref = np.ascontiguousarray(blk).reshape(-1).view(np.float64)
        n_bad += int(np.sum(~np.isfinite(ref)))
        assert np.array_equal(np.isfinite(got), np.isfinite(ref))
        f = np.isfinite(ref)
        assert np.max(np.abs(got[f] - ref[f]), initial=0.0) <= TOL[prec]
    assert n_bad > 0
    d.close()


@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("decades", [0, 3, 6, 10, 16, 150])
def test_graded_along_k(ctx, prec, decades):
    """Both products with their operands graded against each other along K: every term counts alike, but the
    largest row times the largest column is 10^decades of it. With n terms in all (a fold, a product over dl
    and one over channels * dr, each complex), FP64 sums are off by at most n 2^-53 of the sum of the terms'
    magnitudes, the oracle's too, and float-float ones by n 2^-46; the bounds are twice the sum of both,
    relative to the largest such sum of the output block."""
    import paper_1512_03318_gb300 as P
    dl, dr, channels = 120, 96, 4
    case = dict(_spin_channels(83, dl, dr, channels, False))
    up = 10.0 ** (decades * np.arange(dl) / (dl - 1) - decades / 2.0)
    vp = 10.0 ** (decades * np.arange(dr) / (dr - 1) - decades / 2.0)
    l, r, t = case["lflat"].copy(), case["rflat"].copy(), case["tflat"].copy()
    for row in case["ll"]:
        off, d0, d1 = row[3:]
        l[off:off + d0 * d1].reshape(d0, d1)[:] *= up[None, :]
    for row in case["rl"]:
        off, d0, d1 = row[3:]
        r[off:off + d0 * d1].reshape(d0, d1)[:] *= (1.0 / vp)[:, None]
    for m in case["lay"]:
        blk = t[m["offset"]: m["offset"] + m["rowdim"] * m["coldim"]].reshape(m["rowdim"], m["coldim"])
        for _, _, da, ro in m["rows"]:
            blk[ro:ro + da] /= up[:, None]
        for _, _, db, co in m["cols"]:
            blk[:, co:co + db] *= vp[None, :]
    case.update(lflat=l, rflat=r, tflat=t)
    ref = _oracle(case)
    mag = dict(case, lflat=np.abs(l), rflat=np.abs(r), tflat=np.abs(t),
               wi=[(*e[:4], abs(e[4])) for e in case["wi"]], wj=[(*e[:4], abs(e[4])) for e in case["wj"]])
    bound = np.abs(_oracle(mag))
    n = 4 * (dl + channels + channels * dr)
    tol = 2.0 * n * (2.0 ** -53 + (2.0 ** -53 if prec == 0 else 2.0 ** -46))
    h = P.Heff(ctx, **G.heff_args(case))
    h.set_option(P.MRD_OPT_DIGITS, 2)
    h.set_env(_dev(l), _dev(r))
    T = _dev(t)
    out = torch.empty_like(T)
    h.apply(T, out, prec)
    h.status()
    assert h.form() == 1
    got = out.cpu().numpy()
    for m in case["lay"]:
        view = lambda x: x[m["offset"]: m["offset"] + m["rowdim"] * m["coldim"]].reshape(m["rowdim"], m["coldim"])
        for _, _, da, ro in m["rows"]:
            for _, _, db, co in m["cols"]:
                e = np.abs(view(got) - view(ref))[ro:ro + da, co:co + db]
                assert np.max(e) <= tol * np.max(view(bound)[ro:ro + da, co:co + db])
    h.close()


@pytest.mark.parametrize("prec", [0, 3])
def test_environment_wait_limit(ctx, prec):
    """With no time to wait, an environment update's products give up before any copy or MMA and the call says
    so, every time; with time, the next one is right."""
    import paper_1512_03318_gb300 as P
    ly, chi, lx = 8, 800, 4
    mpo = P.MPO(None, lx, ly, 1, ly, 1.0, 1.0, P.MRD_BASIS_MIXED)
    n, j = lx * ly, 15
    caps = [[(q[0], q[1], m) for q, m in synth.bond_sectors(chi, ly, round(b / 2), synth.substream(97, 7, b), min_dim=1)]
            if 2 <= b <= n - 2 else [] for b in range(n + 1)]
    d = P.DMRG(ctx, mpo, n // 2, 0, chi, seed=3, center=16, caps=caps)
    good = d.env(j + 1, 0)
    d.set_option(P.MRD_DMRG_OPT_WAIT_LIMIT_US, 0)
    for _ in range(2):
        with pytest.raises(P.MrdError) as ex:
            d.env_update(j, +1, prec)
        assert ex.value.code == -7
    with pytest.raises(P.MrdError):
        d.set_option(P.MRD_DMRG_OPT_WAIT_LIMIT_US, -1)
    d.set_option(P.MRD_DMRG_OPT_WAIT_LIMIT_US, 1000000)
    d.env_update(j, +1, prec)
    assert np.max(np.abs(d.env(j + 1, 0) - good)) <= TOL[prec] * np.max(np.abs(good))
    d.close()
